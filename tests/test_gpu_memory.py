"""What the room that short im2col maps need costs: only the buffers that such a
map reads have it."""
import pytest

from paper_2504_13850_gb300 import api, build
from paper_2504_13850_gb300 import workloads as W

pytestmark = pytest.mark.gpu
KB = 1024


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


def server(hw, affines=0, dtype="bf16", omega=3):
    b = W._Builder()
    t = b.add("conv", 0, cin=64, cout=128, k=3, stride=1, bias=0)
    t = b.add("avgpool", t)
    for _ in range(affines):
        t = b.add("affine", t, c=128)
    b.add("linear", t, cin=128, cout=10, bias=1)
    s = api.Server(b.ops, 1, omega, 2, 1, (hw, hw, 64), 10, dtype, 0.01, 0.9)
    out = s.activation_bytes(), s.device_bytes()
    s.close()
    return out


@pytest.mark.parametrize("hw,slot", [(16, 16 * 16 * 64 * 2),        # rows of 16 pixels: tiled boxes
                                     (7, 21 * 7 * 7 * 64 * 2)])     # im2col: the images that fill 128 KB
def test_slab(hw, slot):
    assert hw == 16 or slot - 7 * 7 * 64 * 2 < 128 * KB <= slot
    assert server(hw)[0] == 3 * ((slot + 255) // 256 * 256 + 2 * 4)


def test_small_tensors_take_what_they_hold():
    """Eight more affines of [1, 1, 1, 128]: two tensors of 256 bytes each, and parameters, momentum, gradient,
    shadow and partial sums of a few KB together."""
    assert server(7, 8)[1] - server(7, 0)[1] < 8 * 16 * KB
