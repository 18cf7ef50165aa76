"""The FP64 V-cycle on grids whose first coarse level has few enough nodes for
the coarse levels' one launch but not the shared memory (37 x 95 x 18 and 68 x 54 x
17: the launch begins one level further down), against the V-cycle's
definition."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import test_gpu_edges as E  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n,nu,post", [((73, 189, 35), 2, 2), ((135, 107, 33), 1, 2)])
def test_vcycle(n, nu, post):
    E.test_vcycle_sizes(n, nu, post)
