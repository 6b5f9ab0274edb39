"""The CG loop on the device (a graph's conditional WHILE node) and the loop
from the host run the same kernels in the same order: the same bits.

On a stream of their own (the legacy default stream cannot be captured), at
45^3 (plane pass) and 75^3 (separate passes) in the mixed path, where the last
block of the last kernel sets the loop's condition, for several cells that end
at different iterations, for a tangent's six right-hand sides, and at finite
strain. The launch counts tell that the two loops did run.
"""
import numpy as np
import pytest

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PATH = np.outer([2.2e-3, 6e-4], [0.4, -0.2, -0.2, 0.3, -0.25, 0.9])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_05970_gb300 import build
    build.build()
    fftg.load()


def _phase(N, seed):
    r = min(4.0, N / 4)
    return I.random_spheres(N, 0.3, seed, r_min=r / 2, r_max=r)[0]


@pytest.mark.parametrize("N,precision,cells", [(45, "mixed", 1), (45, "mixed", 5), (75, "mixed", 1), (75, "mixed", 3),
                                               (27, "fp64", 3)])
def test_small_strain(N, precision, cells):
    ph = np.stack([_phase(N, 5 + b) for b in range(cells)])
    dE = np.stack([np.outer([1.0, 1.0 + 0.4 * b], np.ones(6)) * PATH for b in range(cells)], axis=1)
    got, launches = [], []
    for graph in (1, 0):
        c = fftg.Cell(N, ph, I.TWO_PHASE, precision=precision, cg_graph=graph, stream=torch.cuda.Stream())
        out = []
        for k in range(2):
            sig, nn, nc, st = c.batch_step(dE[k], 1e-6, 1e-8)
            assert (st == 0).all()
            out += [sig, nn, nc]
        assert (nc > 0).all() and (cells < 3 or len(set(nc)) > 1)
        out += list(c.tangent(1e-8))
        got.append(out)
        launches.append(c.launch_count())
        c.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert launches[0] != launches[1]


@pytest.mark.parametrize("N,precision", [(9, "mixed"), (45, "mixed"), (75, "mixed"), (15, "fp64")])
def test_finite_strain(N, precision):
    dF = np.array([[0.02, 0.03, 0.0], [0.01, -0.02, 0.01], [0.0, 0.02, 0.01]])
    got, launches = [], []
    for graph in (1, 0):
        c = fftg.FsCell(N, _phase(N, 5), I.SVK_TWO_PHASE, precision=precision, cg_graph=graph,
                        stream=torch.cuda.Stream())
        P, nn, nc = c.step(dF, 1e-7, 1e-8)
        got.append([P, nn, nc] + (list(c.tangent(1e-8)) if N <= 45 else []))
        launches.append(c.launches())
        c.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert launches[0] != launches[1]
