"""The classifier head (logits, softmax cross-entropy, dz, input and weight
gradient) at the edges of its split: fewer classes than the cluster has CTAs,
class counts that leave a ragged last CTA, contraction lengths that are no
multiple of four (scalar loads), one row, a ragged last group of rows, more
groups than fit at once, a head on the uploaded batch itself (no input
gradient) and behind a ReLU (its mask).  fp32 whole traces at 1e-4 (the bound
of the fp32 path), bf16 steps under the gates of harness.gate_failures.

The fp32 traces run at the workload's learning rate of 0.01: each step rounds
the stored parameters to fp32 (about 3.4e-8 of their size, rms), which after
two steps is 5e-8 |theta|; the update of the smallest network here is 4e-4
|theta| at a rate of 0.001, so the rounding alone would be 1.2e-4 of it, and
1.2e-5 at 0.01."""
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


def head_ops(cin, mid, classes, relu, bias=1):
    b = W._Builder()
    t = 0
    if mid:
        t = b.add("conv", t, cin=cin, cout=mid, k=1, stride=1, bias=1)
        if relu:
            t = b.add("relu", t)
    t = b.add("flatten", t)
    b.add("linear", t, cin=(mid or cin) * 6, cout=classes, bias=bias)
    return b.ops


EV = [("enq", 0), ("enq", 1), ("step",), ("step",)]


@pytest.mark.parametrize("cin,mid,classes,batch,relu,bias", [
    (32, 48, 1, 5, 1, 1), (32, 0, 3, 1, 0, 1), (5, 7, 9, 17, 1, 0), (3, 0, 37, 130, 0, 0), (16, 64, 129, 16, 0, 1),
    (8, 100, 1000, 3, 1, 1), (64, 256, 1024, 40, 1, 1)])
def test_fp32(cin, mid, classes, batch, relu, bias):
    cfg = W.shrink(W.CONFIGS["tiny"], ops=head_ops(cin, mid, classes, relu, bias), batch=batch, in_hwc=(2, 3, cin),
                   K=2, omega=2, depth=1, lr=1e-2, classes=classes)
    compare(cfg, EV, loss_tol=1e-4, param_tol=1e-4, upd_tol=1e-4)


@pytest.mark.parametrize("cin,mid,classes,batch", [(64, 64, 200, 64), (64, 24, 10, 33), (64, 3, 5, 2)])
def test_bf16(cin, mid, classes, batch):
    cfg = W.shrink(W.CONFIGS["resnet"], ops=head_ops(cin, mid, classes, 1), batch=batch, in_hwc=(2, 3, cin), K=2,
                   omega=2, depth=1, classes=classes)
    _, _, recs = teacher_forced(cfg, EV)
    check_teacher_forced(recs)
