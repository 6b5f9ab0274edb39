"""||d eps||^2 of the mixed Newton test is summed in FP64.

The solution's values are FP32 numbers, so their squares span 1e-76 to 1e76:
in double-float (the range of FP32) those of strains below 1e-19 are zero, and
a Newton iteration that changed the strain counts as converged without one.
Moduli times 2^60 and strains times 2^-60 are the same problem, by exact
scalings in every step but for what is subnormal in FP32 (below 1e-16 of the
largest values): the norms relative to the strain agree to 1e-9.
"""
import numpy as np
import pytest

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_05970_gb300 import build
    build.build()
    fftg.load()


@pytest.mark.parametrize("N", [15, 45, 75])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_small_strains(N, precision):
    ph = I.random_spheres(N, 0.3, 5, r_min=1.5, r_max=3.0)[0]
    dE = np.array([4e-4, -2e-4, -2e-4, 3e-4, -2.5e-4, 9e-4])
    got = []
    for scale in (1.0, 2.0 ** 60):
        mats = [(2.0 * scale, 1.0 * scale, 1e300, 0.0), (7.0 * scale, 5.0 * scale, 1e300, 0.0)]
        c = fftg.Cell(N, ph, mats, precision=precision, nrhs_tangent=0)
        sig, nn, nc = c.step(dE / scale, 1e-9, 1e-6)
        got.append((sig, nn, c.stats()["newton_norm"]))
        c.close()
    (s0, n0, r0), (s1, n1, r1) = got
    assert r0[0] > 1e-3 and n0 > 1 and n1 == n0
    assert abs(r1[0] - r0[0]) <= 1e-9 * r0[0]
    assert np.abs(s1 - s0).max() <= 1e-9 * np.abs(s0).max()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_small_gradients(precision):
    """Finite strain near the identity (off-diagonal gradients, which F = I + H
    holds exactly): quadratic terms are below 1e-10 of the linear ones at both
    scales, and FP32 rounding through the inner solve stays below 1e-5."""
    N = 15
    ph = I.random_spheres(N, 0.3, 5, r_min=1.5, r_max=3.0)[0]
    dF = np.array([[0.0, 0.03, 0.02], [0.01, 0.0, 0.01], [0.0, 0.02, 0.0]])
    norms = []
    for e in (30, 70):
        s = 2.0 ** e
        c = fftg.FsCell(N, ph, [(1.0 * s, 2.0 * s), (5.0 * s, 8.0 * s)], precision=precision)
        c.step(dF / s, 1e-9, 1e-6)
        norms.append(c.stats()["newton_norm"][0])
        c.close()
    assert norms[0] > 1e-3
    assert abs(norms[1] - norms[0]) <= 1e-5 * norms[0]
