"""Depthwise convolutions on the eight-channel bf16 kernels where they can go
wrong: even and odd maps at both strides, maps of one pixel and narrower than
the window, blocks of 64 channels that are full, partial and several, weight
gradients of several chunks with a ragged last one, first layers (no input
gradient) and accumulated input gradients.  Against the exact oracle under the
gates of the bf16 path; and taps outside the map stay out of the sums whatever
the weights hold."""
import math

import pytest
import torch

from harness import check_teacher_forced, teacher_forced
from paper_2504_13850_gb300 import api, build
from paper_2504_13850_gb300 import workloads as W
from test_gpu_attention_precision import DeviceArray

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


def ops_of(c, k, stride, bias, twice):
    b = W._Builder()
    t = b.add("conv", 0, cin=16, cout=c, k=1, stride=1, bias=1)
    u = b.add("dwconv", t, c=c, k=k, stride=stride, bias=bias)
    if twice:      # two readers: the second input gradient is accumulated onto the first
        u = b.add("add", u, in1=b.add("dwconv", t, c=c, k=8 - k, stride=stride, bias=0))
    u = b.add("avgpool", u)
    b.add("linear", u, cin=c, cout=10, bias=1)
    return b.ops


@pytest.mark.parametrize("c,k,stride,bias,twice,batch,h,w", [
    (64, 3, 2, 1, 0, 9, 8, 8), (72, 5, 2, 0, 1, 9, 6, 10), (120, 5, 1, 1, 0, 5, 9, 4), (8, 3, 1, 1, 0, 33, 1, 1),
    (136, 5, 2, 1, 1, 17, 1, 3), (16, 3, 1, 0, 1, 130, 11, 13), (64, 5, 1, 1, 0, 64, 16, 16), (24, 3, 2, 0, 0, 1, 2, 2)])
def test_shapes(c, k, stride, bias, twice, batch, h, w):
    cfg = W.shrink(W.CONFIGS["mobilenet"], ops=ops_of(c, k, stride, bias, twice), classes=10, batch=batch,
                   in_hwc=(h, w, 16), K=2, omega=4, depth=2, lr=1e-3)
    _, _, recs = teacher_forced(cfg, [("enq", k) for _ in range(2) for k in range(2)] + [("step",)] * 4)
    assert len(recs) == 4
    check_teacher_forced(recs)


def test_first_layer():
    b = W._Builder()
    t = b.add("dwconv", 0, c=72, k=5, stride=1, bias=1)
    t = b.add("avgpool", t)
    b.add("linear", t, cin=72, cout=10, bias=1)
    cfg = W.shrink(W.CONFIGS["mobilenet"], ops=b.ops, classes=10, batch=40, in_hwc=(10, 7, 72), K=2, omega=4, depth=2,
                   lr=1e-3)
    _, _, recs = teacher_forced(cfg, [("enq", k) for _ in range(2) for k in range(2)] + [("step",)] * 4)
    check_teacher_forced(recs)


@pytest.mark.parametrize("k,stride", [(3, 1), (5, 1), (3, 2), (5, 2)])
def test_taps_outside_the_map_take_no_part(k, stride):
    """The window's first tap is infinite.  Outputs whose first tap falls outside the map keep the values that
    they have with a finite one."""
    c, h, batch = 16, 6, 4
    ops = [dict(kind="affine", in0=0, c=c), dict(kind="dwconv", in0=1, c=c, k=k, stride=stride, bias=0),
           dict(kind="avgpool", in0=2), dict(kind="linear", in0=3, cin=c, cout=10, bias=0)]
    g = torch.Generator(device="cuda").manual_seed(k)
    x = torch.randn(batch, h, h, c, device="cuda", generator=g).bfloat16()
    w = torch.randn(c, k, k, device="cuda", generator=g) * 0.3
    labels = torch.zeros(batch, dtype=torch.int32, device="cuda")
    ho = (h - 1) // stride + 1

    def outputs(first_tap):
        w[:, 0, 0] = first_tap
        theta = torch.cat([t.flatten() for t in (torch.ones(c, device="cuda"), torch.zeros(c, device="cuda"), w,
                                                 torch.zeros(10, c, device="cuda"))])
        s = api.Server(ops, 1, 1, 1, batch, (h, h, c), 10, "bf16", 0.0, 0.0)
        s.set_params(theta.cpu().numpy())
        torch.cuda.synchronize()
        assert s.enqueue_activations(0, x, labels)[0] == api.OK
        s.server_step()
        s.synchronize()
        y = torch.as_tensor(DeviceArray(s.tensor(2)[0], (batch, ho, ho, c), "<i2"), device="cuda").view(torch.bfloat16)
        y = y.float().clone()
        s.close()
        return y

    finite, inf = outputs(0.25), outputs(math.inf)
    outside = (torch.arange(ho, device="cuda") * stride - k // 2) < 0
    edge = outside[:, None] | outside[None, :]
    assert torch.equal(inf[:, edge], finite[:, edge])
    assert not torch.isfinite(inf[:, ~edge]).any()
