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
    for N in (75, 81, 125, 225):
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
