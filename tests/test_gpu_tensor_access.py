"""Outputs read through fo_server_tensor: an affine whose only reader is a
residual add is formed inside the add's pass, and its own output is there all
the same, as bf16(x * scale + shift) of the step's batch."""
import pytest
import torch

from paper_2504_13850_gb300 import api, build
from test_gpu_affine_pool import block_ops
from test_gpu_attention_precision import DeviceArray

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


@pytest.mark.parametrize("c,two,swapped,relu,h,w", [(64, 0, 0, 1, 5, 3), (40, 1, 0, 1, 2, 3), (264, 0, 1, 0, 3, 3),
                                                    (128, 1, 1, 0, 8, 8)])
def test_affine_in_front_of_an_add(c, two, swapped, relu, h, w):
    ops = block_ops(16, c, two, swapped, relu)
    batch = 12
    g = torch.Generator(device="cuda").manual_seed(c)
    s = api.Server(ops, 1, 1, 1, batch, (h, w, 16), 10, "bf16", 0.0, 0.0)
    theta = torch.randn(s.n_params, device="cuda", generator=g) * 0.3
    s.set_params(theta.cpu().numpy())
    sizes = {"conv": lambda o: o["cout"] * o["k"] ** 2 * o["cin"] + (o["cout"] if o["bias"] else 0),
             "affine": lambda o: 2 * o["c"]}

    def out(i):
        ptr, dims, _ = s.tensor(i + 1)
        return torch.as_tensor(DeviceArray(ptr, dims, "<i2"), device="cuda").view(torch.bfloat16).clone()

    for step in range(2):       # the second batch's outputs replace the first's
        x = torch.randn(batch, h, w, 16, device="cuda", generator=g).bfloat16()
        labels = torch.zeros(batch, device="cuda", dtype=torch.int32)
        torch.cuda.synchronize()
        assert s.enqueue_activations(0, x, labels)[0] == api.OK
        s.server_step()
        s.synchronize()
        at = seen = 0
        for i, op in enumerate(ops):
            if op["kind"] == "affine":
                sc, sh = theta[at:at + c].double(), theta[at + c:at + 2 * c].double()
                want = (out(op["in0"] - 1).double() * sc + sh).float()
                # one rounding to fp32 (here or in the fused multiply-add), one to bf16
                assert ((out(i).float() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-30).all()
                seen += 1
            at += sizes.get(op["kind"], lambda o: 0)(op)
        assert seen == 1 + two
        add = next(i for i, op in enumerate(ops) if op["kind"] == "add")
        y = out(ops[add]["in0"] - 1).float() + out(ops[add]["in1"] - 1).float()
        stored = add + (1 if relu else 0)      # with a ReLU behind it, the add's pass stores that
        assert torch.equal(out(stored), (y.relu() if relu else y).bfloat16())
    s.close()
