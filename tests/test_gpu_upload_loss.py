"""Uploads of batches that are in device memory (one kernel) against the same
batches from host memory (stream copies): byte counts with a tail, sources off
the 16-byte boundary (which keep the copies), with and without lengths, and
parameters equal bit for bit.  Losses read from the host mirror against those
read step by step, over more steps than the mirror holds."""
import numpy as np
import pytest
import torch

from paper_2504_13850_gb300 import api, build
from paper_2504_13850_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


def ops_of(h, w, c):
    b = W._Builder()
    t = b.add("flatten", 0)
    b.add("linear", t, cin=h * w * c, cout=7, bias=1)
    return b.ops


def to_device(a, off):
    """`a` in device memory, its first byte `off` elements past an aligned address."""
    t = torch.from_numpy(np.ascontiguousarray(a)).flatten()
    buf = torch.empty(t.numel() + off, dtype=t.dtype, device="cuda")
    buf[off:].copy_(t)
    return buf[off:]


@pytest.mark.parametrize("name,h,w,c,batch,off", [("tiny", 5, 7, 3, 3, 0), ("tiny", 5, 7, 3, 3, 1),
                                                  ("tiny", 16, 16, 32, 64, 0), ("resnet", 3, 5, 1, 1, 0),
                                                  ("resnet", 3, 5, 7, 33, 0), ("resnet", 8, 8, 64, 1000, 0),
                                                  ("resnet", 8, 8, 64, 9, 4)])
def test_device_and_host_uploads_agree(name, h, w, c, batch, off):
    cfg = W.shrink(W.CONFIGS[name], ops=ops_of(h, w, c), batch=batch, in_hwc=(h, w, c), K=2, omega=2, depth=1,
                   classes=7)
    theta, losses = [], []
    for device in (False, True):
        s = api.Server.from_config(cfg)
        s.set_params(W.init_params(cfg))
        for k in (0, 1):
            x, bits, y, _ = W.device_batch(cfg, k, 0)
            up = np.ascontiguousarray(bits if cfg["dtype"] == W.BF16 else x)
            if device:
                if up.dtype == np.uint16:
                    up = up.view(np.int16)
                up, y = to_device(up, off), to_device(y, 0)
                torch.cuda.synchronize()
            assert s.enqueue_activations(k, up, y)[0] == api.OK
        for _ in range(2):
            s.server_step()
        losses.append(s.read_losses(0, 2))
        theta.append(s.get_params())
        s.close()
    assert np.array_equal(theta[0], theta[1])
    assert np.array_equal(losses[0], losses[1])


def test_lengths_upload():
    cfg = W.shrink(W.CONFIGS["transformer"], ops=W.transformer_ops(d=64, heads=1, ffn=64, blocks=1, classes=2), batch=5,
                   in_hwc=(50, 1, 64), K=1, omega=1, depth=1)
    theta = []
    for device in (False, True):
        s = api.Server.from_config(cfg)
        s.set_params(W.init_params(cfg))
        _, bits, y, ln = W.device_batch(cfg, 0, 0)
        args = [np.ascontiguousarray(bits), y, ln]
        if device:
            args = [to_device(a.view(np.int16) if a.dtype == np.uint16 else a, 0) for a in args]
            torch.cuda.synchronize()
        assert s.enqueue_activations(0, *args)[0] == api.OK
        s.server_step()
        theta.append(s.get_params())
        s.close()
    assert np.array_equal(theta[0], theta[1])


def test_losses_beyond_the_mirror():
    n = 1100
    cfg = W.shrink(W.CONFIGS["tiny"], ops=ops_of(2, 2, 4), batch=4, in_hwc=(2, 2, 4), K=1, omega=1, depth=1, classes=7,
                   lr=1e-3)
    s = api.Server.from_config(cfg)
    s.set_params(W.init_params(cfg))
    x, _, y, _ = W.device_batch(cfg, 0, 0)
    one = []
    for i in range(n):
        assert s.enqueue_activations(0, x, y)[0] == api.OK
        s.server_step()
        one.append(s.read_losses(i, 1)[0])
    assert len(set(one)) > n // 2          # the losses do move
    assert np.array_equal(s.read_losses(0, n), np.array(one, np.float32))
    assert np.array_equal(s.read_losses(n - 1024, 1024), np.array(one[-1024:], np.float32))
    s.close()
