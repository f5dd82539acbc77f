"""Which uploads the copy kernel takes, and what becomes of the others: the host
rule over device, extent and alignment (CPU), and buffers that end before the
batch does, which get an error and leave the server usable (GPU)."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2504_13850_gb300 import api, build
from paper_2504_13850_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB = 1 << 20


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_rule(tmp_path):
    so = str(tmp_path / "upload_shim.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "native", "upload_shim.cpp"), "-o", so], check=True)
    f = C.CDLL(so).shim_may_read
    f.argtypes = [C.c_int, C.c_int] + [C.c_uint64] * 5 + [C.c_int, C.c_int]

    def rule(device=1, device_id=0, base=2 * MB, length=MB, p=2 * MB, nbytes=1000, align=16, server=0, current=0):
        return bool(f(device, device_id, base, length, p, nbytes, align, server, current))

    assert rule() and rule(nbytes=MB) and rule(p=3 * MB - 1008, nbytes=1008) and rule(p=3 * MB, nbytes=0)
    assert not rule(device=0)                                   # host or managed memory
    assert not rule(device_id=1)                                # another GPU's memory
    assert not rule(device_id=1, current=1)                     # and the calling thread's device is that GPU
    assert not rule(current=1) and rule(device_id=1, server=1, current=1)
    assert not rule(nbytes=MB + 1) and not rule(p=3 * MB - 992, nbytes=1000)   # ends too early
    assert not rule(length=0) and not rule(length=0, base=0)                   # extent unknown
    assert not rule(p=2 * MB - 16) and not rule(p=3 * MB + 16, nbytes=16)      # not inside
    assert not rule(nbytes=2 ** 64 - 16)                                       # no wrap-around
    assert not rule(p=2 * MB + 8) and rule(p=2 * MB + 8, align=4)


def runtime():
    import torch
    return C.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")


@pytest.mark.gpu
@pytest.mark.parametrize("short", ["acts", "labels"])
def test_buffer_that_ends_early_is_refused(short):
    """The buffer is the end of an allocation of 4 MB less 128 KB, of whose last 128 KB nothing is asked for but
    everything is mapped (allocations come in 2 MB pages)."""
    import torch
    build.build()
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    b = W._Builder()
    t = b.add("flatten", 0)
    b.add("linear", t, cin=8 * 8 * 16, cout=7, bias=1)
    batch, size = 32, 4 * MB - 128 * 1024
    s = api.Server(b.ops, 1, 2, 2, batch, (8, 8, 16), 7, "bf16", 0.01, 0.9)
    s.set_params(np.zeros(s.n_params, np.float32))
    rt, ptr = runtime(), C.c_void_p()
    assert rt.cudaMalloc(C.byref(ptr), C.c_size_t(size)) == 0
    try:
        acts = torch.zeros(batch * 8 * 8 * 16, dtype=torch.bfloat16, device="cuda")
        labels = torch.zeros(batch, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        tail = C.c_void_p(ptr.value + size - 64)         # 64 bytes: half of the labels, a sliver of the batch
        on = C.c_int(-1)
        args = [C.c_void_p(acts.data_ptr()), C.c_void_p(labels.data_ptr())]
        args[0 if short == "acts" else 1] = tail
        rc = api.lib().fo_enqueue_activations(s.h, 0, *args, None, C.byref(on))
        assert rc == api.ERR_CUDA
        assert s.enqueue_activations(0, acts, labels)[0] == api.OK          # the server goes on
        assert s.server_step()[0] == api.OK
        assert np.isfinite(s.read_losses(0, 1)).all()
    finally:
        s.close()
        rt.cudaFree(ptr)
