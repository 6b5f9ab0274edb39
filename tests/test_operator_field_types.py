"""A tensor of a type that the operators do not have never reaches a kernel.

The C calls take any type but float64 as float32, so a field of 16-bit numbers
holds half of the bytes that they read and write. It is refused on the host,
before the library is called, as is an output of such a type. Runs without a
GPU: the tensors are the host's and the library records its calls.
"""
import types

import pytest

from paper_1601_05970_gb300 import fftg

torch = pytest.importorskip("torch")


class _Lib:
    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        def call(*a):
            self.calls.append(name)
            return 0
        return call


def _handle(cls, V):
    c = types.SimpleNamespace(h=None, V=V, _lib=_Lib())
    return c, {n: (lambda *a, n=n, **k: getattr(cls, n)(c, *a, **k)) for n in ("project", "matvec")}


class _Field(torch.Tensor):
    """A host tensor that says it is the device's."""
    @property
    def is_cuda(self):
        return True


def _field(n, dtype):
    return torch.zeros(n, dtype=dtype).as_subclass(_Field)


@pytest.mark.parametrize("cls,ncomp", [(fftg.Cell, 6), (fftg.FsCell, 9)])
@pytest.mark.parametrize("name", ["project", "matvec"])
@pytest.mark.parametrize("dtype,out,fits", [(torch.float16, None, False), (torch.bfloat16, None, False),
                                            (torch.float16, torch.float32, False),
                                            (torch.float32, torch.float16, False),
                                            (torch.float64, torch.float32, False),
                                            (torch.float32, None, True), (torch.float64, None, True),
                                            (torch.float32, torch.float64, True)])
def test_types(cls, ncomp, name, dtype, out, fits):
    c, ops = _handle(cls, 27)
    n = ncomp * 27
    args = [_field(n, dtype)] + ([_field(n, out)] if out else [])
    if fits:
        ops[name](*args)
        assert len(c._lib.calls) == 1
    else:
        with pytest.raises(fftg.FftgError):
            ops[name](*args)
        assert c._lib.calls == []
