"""The mixed CG on displacement coefficients against the FP64 path, on every
kind of grid it has: one and two stages per pass, even and odd column counts
and ragged last tiles, the cluster solve (up to 27^3, at each cluster size),
the plane pass (45^3) and the separate passes above.

The FP64 path (CG on real fields, FP64 transforms) agrees with the oracle in
the parity tests; the tolerances are those of the mixed path there.
"""
import numpy as np
import pytest

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

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


@pytest.mark.parametrize("N", [3, 5, 9, 15, 25, 27, 45, 75, 81, 125, 135, 225])
def test_increment_and_tangent(N):
    ph = _phase(N)
    out = {}
    for precision in ("fp64", "mixed"):
        c = fftg.Cell(N, ph, I.TWO_PHASE, precision=precision, nrhs_tangent=6 if N <= 81 else 0)
        sig = [c.step(dE, 1e-6, 1e-8)[0] for dE in PATH]
        assert c.stats()["cg_iters"] > 0
        out[precision] = (np.stack(sig), c.tangent(1e-8)[0] if N <= 81 else None)
        c.close()
        torch.cuda.empty_cache()
    (s64, t64), (s, t) = out["fp64"], out["mixed"]
    assert np.abs(s - s64).max() <= 1e-6 * np.abs(s64).max()
    if t is not None:
        assert np.abs(t - t64).max() <= 1e-5 * np.abs(t64).max()


@pytest.mark.parametrize("N", [3, 9, 27, 45, 81, 125])
def test_finite_strain_increment_and_tangent(N):
    ph = _phase(N)
    dF = np.array([[0.02, 0.03, 0.0], [0.01, -0.02, 0.01], [0.0, 0.02, 0.01]])
    out = {}
    for precision in ("fp64", "mixed"):
        c = fftg.FsCell(N, ph, I.SVK_TWO_PHASE, precision=precision)
        P = c.step(dF, 1e-7, 1e-8)[0]
        out[precision] = (P, c.tangent(1e-8)[0] if N <= 45 else None)
        c.close()
    (P64, t64), (P, t) = out["fp64"], out["mixed"]
    assert np.abs(P - P64).max() <= 1e-6 * np.abs(P64).max()
    if t is not None:
        assert np.abs(t - t64).max() <= 1e-5 * np.abs(t64).max()


@pytest.mark.parametrize("N", [3, 9, 15, 27])
@pytest.mark.parametrize("cells", [2, 17, 40])
def test_cluster_sizes_give_the_same_bits(N, cells):
    """One cell alone runs in a cluster of 16 blocks; 17 and 40 cells in
    smaller ones. A cell's result does not depend on it."""
    ph = np.stack([_phase(N, 5 + b) for b in range(cells)])
    c = fftg.Cell(N, ph, I.TWO_PHASE, precision="mixed", nrhs_tangent=0)
    got = [c.batch_step(np.tile(dE, (cells, 1)), 1e-6, 1e-8) for dE in PATH]
    c.close()
    for b in {0, 1, cells - 1}:
        one = fftg.Cell(N, ph[b], I.TWO_PHASE, precision="mixed", nrhs_tangent=0)
        for dE, (sig, nn, nc, st) in zip(PATH, got):
            s, n, k = one.step(dE, 1e-6, 1e-8)
            assert st[b] == 0 and np.array_equal(s, sig[b]) and (n, k) == (nn[b], nc[b])
        one.close()
