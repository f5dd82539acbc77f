"""Convolutions on the tensor cores whose pixel count is no multiple of a tile
or whose image rows do not fill one (im2col tensor maps): odd and non-square
maps, strides 1 and 2, batches of one and odd ones, and a max-pool epilogue
whose last tile is partial.  Against the exact oracle under the gates of the
bf16 path (harness.gate_failures)."""
import pytest

from harness import check_teacher_forced, teacher_forced
from paper_2504_13850_gb300 import api, build
from paper_2504_13850_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


def strided_ops(k):
    """stride-2 and stride-1 convolutions of the uploaded batch and of a hidden map."""
    b = W._Builder()
    t = b.add("conv", 0, cin=64, cout=128, k=k, stride=2, bias=1)
    t = b.add("relu", t)
    t = b.add("conv", t, cin=128, cout=128, k=3, stride=1, bias=1)
    t = b.add("relu", t)
    t = b.add("conv", t, cin=128, cout=256, k=k, stride=2, bias=0)
    t = b.add("affine", t, c=256)
    t = b.add("avgpool", t)
    b.add("linear", t, cin=256, cout=10, bias=1)
    return b.ops


@pytest.mark.parametrize("k,batch,h,w", [(3, 1, 7, 7), (3, 5, 14, 14), (1, 3, 14, 14), (3, 3, 9, 12), (1, 2, 12, 9),
                                         (3, 11, 28, 28), (3, 37, 8, 8), (3, 2, 20, 11), (3, 4, 2, 3)])
def test_strided_and_ragged(k, batch, h, w):
    cfg = W.shrink(W.CONFIGS["resnet"], ops=strided_ops(k), batch=batch, in_hwc=(h, w, 64), K=2, omega=2, depth=1,
                   classes=10)
    _, _, recs = teacher_forced(cfg, [("enq", 0), ("enq", 1), ("step",), ("step",)])
    check_teacher_forced(recs)


@pytest.mark.parametrize("batch,hw", [(37, 8), (3, 16), (5, 8), (3, 4), (3, 14)])
def test_pooled_forward(batch, hw):
    b = W._Builder()
    t = b.add("conv", 0, cin=64, cout=128, k=3, stride=1, bias=1)
    t = b.add("relu", t)
    t = b.add("conv", t, cin=128, cout=128, k=3, stride=1, bias=1)
    t = b.add("relu", t)
    t = b.add("maxpool2", t)
    t = b.add("avgpool", t)
    b.add("linear", t, cin=128, cout=10, bias=1)
    cfg = W.shrink(W.CONFIGS["resnet"], ops=b.ops, batch=batch, in_hwc=(hw, hw, 64), K=2, omega=2, depth=1, classes=10)
    _, _, recs = teacher_forced(cfg, [("enq", 0), ("enq", 1), ("step",), ("step",)])
    check_teacher_forced(recs)
