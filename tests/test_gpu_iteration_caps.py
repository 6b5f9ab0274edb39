"""An iteration cap of INT_MAX ("no limit") is a cap like any other.

Every way a CG solve runs (one cluster launch up to 27^3, the graph loop with
the plane pass at 45^3 and with the separate passes at 75^3, the loop from the
host, a group's graph, finite strain) gives the bits it gives with the default
cap, which none of these solves reaches. (The legacy default stream cannot be
captured: the handles work in a stream of their own, so that graphs run.)
"""
import numpy as np
import pytest

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MOST = 2 ** 31 - 1
# to just below the soft yield strain, then through it
PATH = np.outer([2.2e-3, 6e-4], [0.4, -0.2, -0.2, 0.3, -0.25, 0.9])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_05970_gb300 import build
    build.build()
    fftg.load()


def _phase(N, seed=5):
    r = min(4.0, N / 4)
    return I.random_spheres(N, 0.3, seed, r_min=r / 2, r_max=r)[0]


@pytest.mark.parametrize("N,precision,cg_graph", [(3, "mixed", 1), (9, "mixed", 1), (27, "mixed", 0), (45, "mixed", 1),
                                                  (45, "mixed", 0), (75, "mixed", 1), (75, "mixed", 0),
                                                  (15, "fp64", 1), (15, "fp64", 0)])
def test_small_strain(N, precision, cg_graph):
    ph, got, s = _phase(N), [], torch.cuda.Stream()
    for caps in ({}, dict(max_cg=MOST, max_newton=MOST)):
        c = fftg.Cell(N, ph, I.TWO_PHASE, precision=precision, cg_graph=cg_graph, stream=s, **caps)
        c.step(PATH[0], 1e-6, 1e-8)
        sig, nn, nc = c.step(PATH[1], 1e-6, 1e-8)
        assert nc > 0
        got.append((sig, nn, nc) + c.tangent(1e-8))
        c.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_group():
    ph = [np.stack([_phase(N, 5 + b) for b in range(2)]) for N in (9, 45)]
    got = []
    for caps in ({}, dict(max_cg=MOST, max_newton=MOST)):
        cells = [fftg.Cell(p.shape[1], p, I.TWO_PHASE, precision="mixed", nrhs_tangent=0, **caps) for p in ph]
        g = fftg.Group(cells)
        g.step([np.tile(PATH[0], (2, 1))] * 2, 1e-6, 1e-8)
        got.append(g.step([np.tile(PATH[1], (2, 1))] * 2, 1e-6, 1e-8))
        g.close()
        for c in cells:
            c.close()
    for one, two in zip(*got):
        assert (one[2] > 0).all()
        for a, b in zip(one, two):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("precision,cg_graph", [("mixed", 1), ("mixed", 0), ("fp64", 0)])
def test_finite_strain(precision, cg_graph):
    N, got, s = 9, [], torch.cuda.Stream()
    dF = np.array([[0.02, 0.03, 0.0], [0.01, -0.02, 0.01], [0.0, 0.02, 0.01]])
    for caps in ({}, dict(max_cg=MOST, max_newton=MOST)):
        c = fftg.FsCell(N, _phase(N), I.SVK_TWO_PHASE, precision=precision, cg_graph=cg_graph, stream=s, **caps)
        P, nn, nc = c.step(dF, 1e-7, 1e-8)
        assert nc > 0
        got.append((P, nn, nc) + c.tangent(1e-8))
        c.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
