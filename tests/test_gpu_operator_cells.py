"""Operators on a chosen cell of a batch give the bits of that cell alone.

The caller's fields are one cell's whatever cell is chosen, used in place or
through the handle's buffers (unaligned, overlapping)."""
import ctypes as C

import numpy as np
import pytest

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DE = np.array([0.002, -0.001, 0.0, 0.0005, 0.0, 0.0035])
OFFSETS = [(0, 0), (0, 48), (48, 0), (2, 0), (0, 2), (2, 3)]  # as in the one-cell tests, in bytes


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_05970_gb300 import build
    build.build()
    fftg.load()


def _call(fn, x, like, i, o):
    buf = torch.zeros(max(x.numel() * x.element_size(), like.numel() * like.element_size()) + 64, dtype=torch.uint8,
                      device="cuda")
    n = x.numel() * x.element_size()
    buf[i:i + n] = x.view(torch.uint8)
    assert fn(C.c_void_p(buf.data_ptr() + i), C.c_void_p(buf.data_ptr() + o)) == 0
    return buf[o:o + n].clone().view(x.dtype)


@pytest.mark.parametrize("N", [9, 45])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_chosen_cell(N, precision):
    cells = 3
    ph = np.stack([I.random_spheres(N, 0.3, 5 + b, r_min=1.0, r_max=2.0)[0] for b in range(cells)])
    batch = fftg.Cell(N, ph, I.TWO_PHASE, precision=precision, nrhs_tangent=0)
    batch.batch_step(np.outer([0.5, 0.8, 1.0], DE), 1e-6, 1e-8)
    lib, d = fftg.load(), (0.3 * DE).ctypes.data_as(C.POINTER(C.c_double))
    code = fftg.FFTG_FP64 if precision == "fp64" else fftg.FFTG_MIXED
    g = torch.Generator(device="cuda").manual_seed(N)
    eps = 5e-4 * torch.randn(6 * N ** 3, dtype=torch.float64, device="cuda", generator=g)
    p = torch.randn(6 * N ** 3, dtype=torch.float64 if precision == "fp64" else torch.float32, device="cuda",
                    generator=g)
    for b in (2, 1, 0):
        batch.select(b)
        one = fftg.Cell(N, ph[b], I.TWO_PHASE, precision=precision, nrhs_tangent=0)
        one.set_state(batch.get_state())
        for i, o in OFFSETS:
            got = [(_call(lambda a, q: lib.fftg_op_constitutive(c.h, d, a, q), eps, eps, i, o),
                    c.field(fftg.FFTG_FIELD_TANGENT),
                    _call(lambda a, q: lib.fftg_op_matvec(c.h, code, a, q, None), p, p, i, o)) for c in (batch, one)]
            assert torch.equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1]), (b, i, o)
            assert torch.equal(got[0][2], got[1][2]), (b, i, o)
        one.close()
    batch.close()


@pytest.mark.parametrize("N", [5, 15, 25, 75, 135, 225])
def test_finite_strain_grids(N):
    """The finite-strain CG on coefficients against the FP64 path on the grids
    that the coefficient tests leave out, 225 among them with its 25 x 9 split
    of x1 beside the 15 x 15 plan of x2; to 1e-6, as there."""
    r = min(4.0, N / 4)
    ph = I.random_spheres(N, 0.3, 5, r_min=r / 2, r_max=r)[0]
    dF = np.array([[0.02, 0.03, 0.0], [0.01, -0.02, 0.01], [0.0, 0.02, 0.01]])
    out = {}
    for precision in ("fp64", "mixed"):
        c = fftg.FsCell(N, ph, I.SVK_TWO_PHASE, precision=precision)
        out[precision] = c.step(dF, 1e-7, 1e-8)[0]
        c.close()
        torch.cuda.empty_cache()
    assert np.abs(out["mixed"] - out["fp64"]).max() <= 1e-6 * np.abs(out["fp64"]).max()
