"""Operators in a caller's stream capture.

They only enqueue (no host output, no synchronisation), so a captured call can
be replayed: on the fields' contents at that time, with the strain of the call
that was captured, in place and through the handle's buffers."""
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


@pytest.mark.parametrize("offset", [0, 2])
def test_replay(offset):
    N, s = 15, torch.cuda.Stream()
    ph = I.random_spheres(N, 0.3, 5, r_min=1.0, r_max=2.0)[0]
    cell = fftg.Cell(N, ph, I.TWO_PHASE, precision="mixed", nrhs_tangent=0, stream=s)
    lib, n = fftg.load(), 6 * N ** 3
    bufs = {k: torch.zeros(n * b + 64, dtype=torch.uint8, device="cuda")
            for k, b in (("eps", 8), ("sig", 8), ("p", 4), ("q", 4), ("g", 4))}
    at = {k: C.c_void_p(b.data_ptr() + offset) for k, b in bufs.items()}
    rng = torch.Generator(device="cuda").manual_seed(3)

    def fill():
        for k, dt in (("eps", torch.float64), ("p", torch.float32)):
            x = 5e-4 * torch.randn(n, dtype=dt, device="cuda", generator=rng)
            bufs[k][offset:offset + n * x.element_size()] = x.view(torch.uint8)

    def calls(dE):
        d = np.ascontiguousarray(dE).ctypes.data_as(C.POINTER(C.c_double))
        assert lib.fftg_op_constitutive(cell.h, d, at["eps"], at["sig"]) == 0
        assert lib.fftg_op_matvec(cell.h, fftg.FFTG_MIXED, at["p"], at["q"], None) == 0
        assert lib.fftg_op_project(cell.h, fftg.FFTG_MIXED, at["p"], at["g"]) == 0

    fill()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        calls(DE)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        calls(DE)
    for _ in range(2):
        fill()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            calls(2 * DE)  # another call's strain is not the graph's
            graph.replay()
        torch.cuda.synchronize()
        got = {k: bufs[k].clone() for k in ("sig", "q", "g")}
        with torch.cuda.stream(s):
            calls(DE)
        torch.cuda.synchronize()
        for k, b in got.items():
            assert torch.equal(b, bufs[k]) and b.any(), k
    cell.close()
