"""Affines and pools on the vectorised bf16 kernels: channel counts whose
vectors do not divide a block (the grid is then a multiple of them), affines
added to a plain residual and to another affine, on either side of the add,
with and without a ReLU; global average pools of one pixel and of many, with
few channels and more than one block's.  bf16 steps under the gates of
harness.gate_failures."""
import pytest

from harness import check_teacher_forced, teacher_forced
from paper_2504_13850_gb300 import api, build
from paper_2504_13850_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


def block_ops(cin, c, two, swapped, relu):
    b = W._Builder()
    x = b.add("conv", 0, cin=cin, cout=c, k=1, stride=1, bias=1)
    x = b.add("relu", x)
    t = b.add("conv", x, cin=c, cout=c, k=1, stride=1, bias=0)
    t = b.add("affine", t, c=c)
    r = x
    if two:
        r = b.add("conv", x, cin=c, cout=c, k=1, stride=1, bias=0)
        r = b.add("affine", r, c=c)
    y = b.add("add", r, in1=t) if swapped else b.add("add", t, in1=r)
    if relu:
        y = b.add("relu", y)
    y = b.add("avgpool", y)
    b.add("linear", y, cin=c, cout=10, bias=1)
    return b.ops


@pytest.mark.parametrize("c,two,swapped,relu,batch,h,w", [
    (8, 0, 0, 1, 20, 1, 1), (40, 1, 0, 1, 16, 5, 3), (264, 0, 1, 0, 16, 3, 3), (264, 1, 1, 1, 33, 2, 5),
    (120, 0, 0, 0, 64, 16, 16), (648, 1, 0, 0, 17, 4, 4)])
def test_block(c, two, swapped, relu, batch, h, w):
    cfg = W.shrink(W.CONFIGS["resnet"], ops=block_ops(16, c, two, swapped, relu), batch=batch, in_hwc=(h, w, 16), K=2,
                   omega=4, depth=2, classes=10, lr=1e-3)
    ev = [("enq", k) for _ in range(2) for k in range(2)] + [("step",)] * 4
    _, _, recs = teacher_forced(cfg, ev)
    assert len(recs) == 4
    check_teacher_forced(recs)


def test_more_channels_than_a_grid_dimension():
    """One more block of 256 channels than a grid has rows: the scalar pool takes them."""
    import numpy as np
    c = 65535 * 256 + 8
    b = W._Builder()
    t = b.add("avgpool", 0)
    t = b.add("linear", t, cin=c, cout=8, bias=0)
    b.add("linear", t, cin=8, cout=3, bias=0)
    s = api.Server(b.ops, 1, 1, 1, 1, (1, 1, c), 3, "bf16", 0.0, 0.0)
    theta = np.zeros(s.n_params, np.float32)
    theta[c - 1] = 1.0                  # the first layer's first output is the last channel
    theta[8 * c] = 1.0                  # and the first logit is that
    s.set_params(theta)
    x = np.zeros((1, 1, 1, c), np.uint16)
    x[..., -1] = 0x4000                 # 2.0
    assert s.enqueue_activations(0, x, np.zeros(1, np.int32))[0] == api.OK
    s.server_step()
    loss = s.read_losses(0, 1)[0]
    s.close()
    assert abs(loss - np.log(np.exp(2.0) + 2.0) + 2.0) < 1e-5
