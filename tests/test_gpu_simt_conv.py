"""The CUDA-core convolution and linear kernels at the edges of their tiles:
channel counts that are no multiple of four or of a tile (scalar loads, ragged
columns), narrow outputs (a 3-channel first layer's weight gradient), maps and
batches that leave partial row tiles, strides, and every tile shape.  fp32
whole traces at 1e-4 (the bound of the fp32 path), bf16 steps under the gates
of harness.gate_failures."""
import pytest

from harness import check_teacher_forced, teacher_forced
from paper_2504_13850_gb300 import api, build
from paper_2504_13850_gb300 import workloads as W
from test_gpu_train import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


def conv_ops(cin, mid, out, k, stride):
    b = W._Builder()
    t = b.add("conv", 0, cin=cin, cout=mid, k=k, stride=stride, bias=1)
    t = b.add("relu", t)
    t = b.add("conv", t, cin=mid, cout=out, k=3, stride=1, bias=1)
    t = b.add("relu", t)
    t = b.add("conv", t, cin=out, cout=out, k=1, stride=2, bias=0)
    t = b.add("avgpool", t)
    b.add("linear", t, cin=out, cout=10, bias=1)
    return b.ops


EV = [("enq", 0), ("enq", 1), ("step",), ("step",)]
SHAPES = [(3, 7, 10, 3, 1, 3, 9, 7), (5, 130, 66, 3, 2, 2, 11, 8), (32, 64, 128, 3, 1, 16, 16, 16),
          (4, 32, 36, 1, 2, 1, 5, 5), (8, 128, 4, 3, 1, 40, 24, 24)]


@pytest.mark.parametrize("cin,mid,out,k,stride,batch,h,w", SHAPES)
def test_fp32(cin, mid, out, k, stride, batch, h, w):
    cfg = W.shrink(W.CONFIGS["tiny"], ops=conv_ops(cin, mid, out, k, stride), batch=batch, in_hwc=(h, w, cin), K=2,
                   omega=2, depth=1, lr=1e-3)
    compare(cfg, EV, loss_tol=1e-4, param_tol=1e-4, upd_tol=1e-4)


@pytest.mark.parametrize("cin,mid,out,k,stride,batch,h,w", [SHAPES[0], SHAPES[1], (3, 128, 128, 3, 1, 8, 32, 32)])
def test_bf16(cin, mid, out, k, stride, batch, h, w):
    cfg = W.shrink(W.CONFIGS["resnet"], ops=conv_ops(cin, mid, out, k, stride), batch=batch, in_hwc=(h, w, cin), K=2,
                   omega=2, depth=1, classes=10)
    _, _, recs = teacher_forced(cfg, EV)
    check_teacher_forced(recs)
