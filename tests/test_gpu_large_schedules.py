"""P3 in both of its forms on the grids where the fused one is the default
(75^3 and up): schedule variant 3 is the other form there. It sums in another
order, so that its bits differ, and its G tau agrees to FP32 rounding."""
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
    yield
    for N in (75, 81, 125, 135, 225):
        for k in fftg.SCHED_KINDS:
            fftg.schedule_set(N, k, 0)


@pytest.mark.parametrize("N", [75, 81, 125, 225])
def test_both_forms_of_p3(N):
    tau = torch.tensor(np.random.default_rng(N).standard_normal(6 * N ** 3).astype(np.float32), device="cuda")
    cell = fftg.Cell(N, np.zeros((N, N, N), dtype=np.uint8), I.TWO_PHASE, precision="mixed", nrhs_tangent=0)
    out = {}
    for v in (0, 3):
        fftg.schedule_set(N, "p3", v)
        out[v] = cell.project(tau).cpu().numpy().astype(np.float64)
    fftg.schedule_set(N, "p3", 0)
    cell.close()
    assert np.isfinite(out[3]).all() and not np.array_equal(out[3], out[0])
    assert np.linalg.norm(out[3] - out[0]) <= 1e-6 * np.linalg.norm(out[0])


@pytest.mark.parametrize("N", [75, 125, 135])
def test_schedules_of_the_solver_passes(N):
    """Up to 45^3 a solve runs none of the tuned row and column passes; from
    75^3 every schedule of them reaches the FP64 path's stress to 1e-6 (the
    mixed path's tolerance)."""
    ph = I.random_spheres(N, 0.3, 5, r_min=2.0, r_max=4.0)[0]
    path = np.outer([2.2e-3, 6e-4], [0.4, -0.2, -0.2, 0.3, -0.25, 0.9])  # to just below the soft yield, through it

    def stress(precision):
        c = fftg.Cell(N, ph, I.TWO_PHASE, precision=precision, nrhs_tangent=0)
        for dE in path:
            sig, nn, nc = c.step(dE, 1e-6, 1e-8)
        c.close()
        torch.cuda.empty_cache()
        assert nc > 0
        return sig

    ref = stress("fp64")
    for kind in ("p1", "p2", "p4"):
        for v in range(fftg.SCHED_VARIANTS):
            fftg.schedule_set(N, kind, v)
            sig = stress("mixed")
            assert np.abs(sig - ref).max() <= 1e-6 * np.abs(ref).max(), (kind, v)
        fftg.schedule_set(N, kind, 0)
