"""Launches that the handles count for solves whose loop runs on the device.

With the number of CG iterations fixed, ten more of them per solve are ten
times the kernels of an iteration, which the loop from the host counts one by
one (less the kernel that sets the device loop's condition, where there is one
of its own).
"""
import numpy as np
import pytest

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DE = np.array([0.003, -0.001, -0.001, 0.001, -0.0005, 0.002])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_05970_gb300 import build
    build.build()
    fftg.load()


def _launches(N, precision, fixed_cg, cg_graph):
    s = torch.cuda.Stream()  # the legacy default stream cannot be captured
    ph = I.random_spheres(N, 0.3, 5, r_min=2.0, r_max=4.0)[0]
    c = fftg.Cell(N, ph, I.TWO_PHASE, precision=precision, nrhs_tangent=0, fixed_cg=fixed_cg, fixed_newton=2,
                  cg_graph=cg_graph, stream=s)
    c.step(DE, 1e-5, 1e-8)
    assert c.stats()["cg_per_newton"] == [fixed_cg, fixed_cg]
    n = c.launch_count()
    c.close()
    return n


@pytest.mark.parametrize("N,precision,kernels,loop_kernels", [(45, "fp64", 6, 1), (75, "mixed", 6, 0),
                                                              (45, "mixed", 4, 0)])
def test_kernels_of_an_iteration(N, precision, kernels, loop_kernels):
    graph = [_launches(N, precision, k, 1) for k in (10, 20)]
    assert graph[1] - graph[0] == 2 * 10 * (kernels + loop_kernels)
    # from the host: chunks of 2, 4, 8 and 16 iterations
    host = [_launches(N, precision, k, 0) for k in (14, 30)]
    assert host[1] - host[0] == 2 * 16 * kernels
