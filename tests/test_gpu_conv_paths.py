"""The convolution's operand paths at the widths and sizes where the choice
between them changes: windows by TMA from 32 channels in and out (fewer voxels
than a tile, a remainder past one and several, rows before the first and past
the last), by threads below, and 32 -> 64 either side of where planes are
marched."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import test_gpu_edges as E  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("d,cin,cout", [((3, 3, 3), 32, 32), ((5, 3, 3), 64, 64), ((17, 9, 3), 128, 64),
                                        ((40, 7, 11), 32, 32), ((40, 7, 11), 32, 16), ((126, 30, 21), 64, 128),
                                        ((70, 60, 33), 32, 64), ((61, 62, 33), 32, 64)])
def test_layer(d, cin, cout):
    """Forward, input gradient, weight and bias gradients against the oracle
    with the bounds of the other layer tests."""
    E.test_layer_sizes(d, cin, cout)
