"""The operators on a caller's fields: any overlap and any byte alignment.

project, matvec and constitutive read and write device pointers in place
(one voxel a lane, since the components of an odd grid start on any element).
Fields that are the same, that overlap partly, or that are not aligned to
their elements give the bits of separate, aligned ones.
"""
import ctypes as C

import numpy as np
import pytest

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DE = np.array([0.002, -0.001, 0.0, 0.0005, 0.0, 0.0035])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_05970_gb300 import build
    build.build()
    fftg.load()


def _ptr(buf, byte):
    return C.c_void_p(buf.data_ptr() + byte)


def _place(x, buf, byte):
    buf[byte:byte + x.numel() * x.element_size()] = x.view(torch.uint8)


def _take(buf, byte, like):
    n = like.numel() * like.element_size()
    return buf[byte:byte + n].clone().view(like.dtype)


# (offset of the input, offset of the output) in bytes: the same field,
# overlapping by all but some elements either way, unaligned in either or both
OFFSETS = [(0, 0), (0, 48), (48, 0), (2, 0), (0, 2), (2, 3)]


@pytest.mark.parametrize("N", [3, 9, 15, 45])
@pytest.mark.parametrize("precision", ["fp32", "dd", "fp64"])
@pytest.mark.parametrize("fs", [False, True])
def test_project_and_matvec_fields(N, precision, fs):
    fp64 = precision == "fp64"
    nc = 9 if fs else 6
    ph, _, _ = I.random_spheres(N, 0.3, 5, r_min=1.0, r_max=2.0)
    make = fftg.FsCell if fs else fftg.Cell
    cell = make(N, ph, I.SVK_TWO_PHASE if fs else I.TWO_PHASE, precision="fp64" if fp64 else "mixed")
    if not fs:
        cell.constitutive(DE)
    lib, pre = fftg.load(), "fftg_fs_op_" if fs else "fftg_op_"
    code = fftg.FFTG_DD if precision == "dd" else fftg.FFTG_FP64 if fp64 else fftg.FFTG_MIXED
    g = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn(nc * N ** 3, device="cuda", generator=g,
                    dtype=torch.float32 if precision == "fp32" else torch.float64)
    calls = [lambda a, b: getattr(lib, pre + "project")(cell.h, code, a, b)]
    if precision != "dd":
        calls.append(lambda a, b: getattr(lib, pre + "matvec")(cell.h, code, a, b, None))
    for call in calls:
        ref = torch.empty_like(x)
        assert call(C.c_void_p(x.data_ptr()), C.c_void_p(ref.data_ptr())) == 0
        assert torch.isfinite(ref).all() and ref.abs().max() > 0
        for i, o in OFFSETS:
            buf = torch.zeros(x.numel() * x.element_size() + 64, dtype=torch.uint8, device="cuda")
            _place(x, buf, i)
            assert call(_ptr(buf, i), _ptr(buf, o)) == 0
            assert torch.equal(_take(buf, o, x), ref), (i, o)
    cell.close()


@pytest.mark.parametrize("fs", [False, True])
def test_page_locked_host_fields(fs):
    N, nc = 15, 9 if fs else 6
    ph, _, _ = I.random_spheres(N, 0.3, 5, r_min=1.0, r_max=2.0)
    cell = (fftg.FsCell if fs else fftg.Cell)(N, ph, I.SVK_TWO_PHASE if fs else I.TWO_PHASE, precision="mixed")
    if not fs:
        cell.constitutive(DE)
    lib, pre = fftg.load(), "fftg_fs_op_" if fs else "fftg_op_"
    x = torch.randn(nc * N ** 3, generator=torch.Generator().manual_seed(N)).pin_memory()
    xd = x.cuda()
    for call in (lambda a, b: getattr(lib, pre + "project")(cell.h, fftg.FFTG_MIXED, a, b),
                 lambda a, b: getattr(lib, pre + "matvec")(cell.h, fftg.FFTG_MIXED, a, b, None)):
        ref, out = torch.empty_like(xd), torch.zeros_like(x).pin_memory()
        assert call(_ptr(xd, 0), _ptr(ref, 0)) == 0
        assert call(_ptr(x, 0), _ptr(out, 0)) == 0
        torch.cuda.synchronize()
        assert torch.equal(out, ref.cpu())
    cell.close()


@pytest.mark.parametrize("N", [3, 15, 45])
def test_constitutive_fields(N):
    ph, _, _ = I.random_spheres(N, 0.3, 5, r_min=1.0, r_max=2.0)
    cell = fftg.Cell(N, ph, I.TWO_PHASE, precision="mixed", nrhs_tangent=0)
    g = torch.Generator(device="cuda").manual_seed(N)
    eps = 5e-4 * torch.randn(6 * N ** 3, dtype=torch.float64, device="cuda", generator=g)
    ref = cell.constitutive(DE, eps)
    ref7 = cell.field(fftg.FFTG_FIELD_TANGENT)
    d = DE.ctypes.data_as(C.POINTER(C.c_double))
    for i, o in OFFSETS:
        buf = torch.zeros(eps.numel() * 8 + 64, dtype=torch.uint8, device="cuda")
        _place(eps, buf, i)
        assert fftg.load().fftg_op_constitutive(cell.h, d, _ptr(buf, i), _ptr(buf, o)) == 0
        assert torch.equal(_take(buf, o, eps), ref), (i, o)
        assert np.array_equal(cell.field(fftg.FFTG_FIELD_TANGENT), ref7)
    cell.close()
