"""Operators return after enqueueing: a call's host arguments are its own.

Several calls are queued behind work that keeps the stream busy, so that the
host is far ahead of it, each with other arguments; every one gives the bits
it gives when the stream is waited for after each call.
"""
import ctypes as C

import numpy as np
import pytest

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 15
PATH = np.outer([2.2e-3, 6e-4], [0.4, -0.2, -0.2, 0.3, -0.25, 0.9])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_05970_gb300 import build
    build.build()
    fftg.load()


def _phase(seed=5):
    return I.random_spheres(N, 0.3, seed, r_min=1.0, r_max=2.0)[0]


def _busy():
    """Some tens of milliseconds of work in the current stream."""
    a = torch.randn(8192, 8192, device="cuda")
    for _ in range(4):
        a = a @ a
    return a


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_small_strain(precision):
    cells = 3
    ph = np.stack([_phase(5 + b) for b in range(cells)])
    c = fftg.Cell(N, ph, I.TWO_PHASE, precision=precision, nrhs_tangent=0)
    for dE in PATH:
        assert (c.batch_step(np.tile(dE, (cells, 1)), 1e-6, 1e-8)[3] == 0).all()
    dt = torch.float64 if precision == "fp64" else torch.float32
    code = fftg.FFTG_FP64 if precision == "fp64" else fftg.FFTG_MIXED
    g = torch.Generator(device="cuda").manual_seed(N)
    p = torch.randn(6 * N ** 3, dtype=dt, device="cuda", generator=g)
    more = [k * 3e-4 * np.array([0.4, -0.2, -0.2, 0.3, -0.25, 0.9]) for k in range(1, 4)]

    def run(wait):
        out = []
        for k, dE in enumerate(more):
            for b in range(cells):
                c.select(b)
                out.append(c.constitutive(dE))
                q = torch.empty_like(p)
                assert fftg.load().fftg_op_matvec(c.h, code, C.c_void_p(p.data_ptr()), C.c_void_p(q.data_ptr()),
                                                  None) == 0
                out.append(q)
                if wait:
                    torch.cuda.synchronize()
        stress = c.field(fftg.FFTG_FIELD_STRESS)
        sig = c.batch_step(np.tile(PATH[1], (cells, 1)), 1e-6, 1e-8)[0]
        return [t.cpu().numpy() for t in out] + [stress, sig]

    states = []
    for b in range(cells):
        c.select(b)
        states.append(c.get_state())
    ref = run(True)
    for b in range(cells):
        c.select(b)
        c.set_state(states[b])
    torch.cuda.synchronize()
    keep = _busy()
    got = run(False)
    assert not np.array_equal(ref[0], ref[-4 - 2 * (cells - 1)])  # the strains differ
    for i, (a, b) in enumerate(zip(ref, got)):
        assert np.array_equal(a, b), i
    del keep
    c.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_finite_strain(precision):
    c = fftg.FsCell(N, _phase(), I.SVK_TWO_PHASE, precision=precision)
    dF = np.array([[0.02, 0.03, 0.0], [0.01, -0.02, 0.01], [0.0, 0.02, 0.01]])
    c.step(dF, 1e-7, 1e-8)
    dt = torch.float64 if precision == "fp64" else torch.float32
    code = fftg.FFTG_FP64 if precision == "fp64" else fftg.FFTG_MIXED
    g = torch.Generator(device="cuda").manual_seed(N)
    p = torch.randn(9 * N ** 3, dtype=dt, device="cuda", generator=g)
    state = c.get_state()

    def run(wait):
        q = torch.empty_like(p)
        assert fftg.load().fftg_fs_op_matvec(c.h, code, C.c_void_p(p.data_ptr()), C.c_void_p(q.data_ptr()), None) == 0
        if wait:
            torch.cuda.synchronize()
        P = c.step(dF, 1e-7, 1e-8)[0]
        return q.cpu().numpy(), P

    ref = run(True)
    c.set_state(state)
    torch.cuda.synchronize()
    keep = _busy()
    for a, b in zip(ref, run(False)):
        assert np.array_equal(a, b)
    del keep
    c.close()
