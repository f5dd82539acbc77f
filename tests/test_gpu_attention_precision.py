"""Attention on heads narrower than 64 keeps its probabilities and score
gradients in fp32: the bf16 outputs and gradients are the exact values rounded
once, but for the few that the fp32 arithmetic carries over a rounding boundary.

The network makes every operand known exactly: a one-hot upload selects columns
of the projection's weight (q, k and v, bf16 values), and the weight gradient
that comes back is then d(q|k|v) row by row; the classifier's weight is a
power-of-two pattern in one class, so that dO is exact once its single factor
per sequence is rounded.

Bound on the share of outputs that differ from the rounded exact value: with an
fp32 error of at most 2^-20 of the result (a few roundings of the exponent's
argument and of the sums) and bf16 spacings of at least 2^-8 of it, one in 2^11
lies close enough to a boundary; twice that is allowed, 2^-10.  Sixteen bits of
P or dS give two to three times the bound."""
import math

import pytest
import torch

from paper_2504_13850_gb300 import api, build

pytestmark = pytest.mark.gpu
CLASSES = 10


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


class DeviceArray:
    def __init__(self, ptr, shape, typestr):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": typestr, "data": (ptr, False), "version": 3}


def attention_step(width, heads, L, B, seed):
    """Runs one step; returns ({name: bf16 values of the step}, {name: exact}) of O, dQ, dK, dV, [B, heads, L, width]."""
    C, D = width * heads, (B * L + 63) // 64 * 64
    ops = [dict(kind="linear", in0=0, cin=D, cout=3 * C, bias=0), dict(kind="attention", in0=1, c=C, heads=heads),
           dict(kind="flatten", in0=2), dict(kind="linear", in0=3, cin=L * C, cout=CLASSES, bias=0)]
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randn(3 * C, D, generator=g, device="cuda").bfloat16().float()
    qkv = w[:, :B * L].t().reshape(B, L, 3, heads, width).permute(2, 0, 3, 1, 4).contiguous()
    sign = torch.randint(0, 2, (L * C,), generator=g, device="cuda") * 2 - 1
    head = torch.zeros(CLASSES, L * C, device="cuda")
    head[0] = sign * 2.0 ** -torch.randint(6, 10, (L * C,), generator=g, device="cuda")
    lens = torch.randint(max(1, L // 4), L + 1, (B,), generator=g, device="cuda", dtype=torch.int32)
    labels = torch.randint(0, CLASSES, (B,), generator=g, device="cuda", dtype=torch.int32)
    x = torch.zeros(B * L, D, device="cuda", dtype=torch.bfloat16)
    x[torch.arange(B * L), torch.arange(B * L)] = 1
    x = x.reshape(B, L, 1, D)
    s = api.Server(ops, 1, 1, 1, B, (L, 1, D), CLASSES, "bf16", 0.0, 0.0, seq=True)
    s.set_params(torch.cat([w.flatten(), head.flatten()]).cpu().numpy())
    torch.cuda.synchronize()
    assert s.enqueue_activations(0, x, labels, lens)[0] == api.OK
    s.server_step()
    s.synchronize()
    s.check_error()
    at = lambda i, shape, t: torch.as_tensor(DeviceArray(s.tensor(i)[0], shape, t), device="cuda").clone()
    o = at(2, (B, L, C), "<i2").view(torch.bfloat16).double().reshape(B, L, heads, width).permute(0, 2, 1, 3)
    logits = at(4, (B, CLASSES), "<f4").double()
    dw = torch.from_numpy(s.get_momentum()[:3 * C * D]).cuda().double().reshape(3 * C, D)[:, :B * L].t()
    dq, dk, dv = dw.reshape(B, L, 3, heads, width).permute(2, 0, 3, 1, 4)
    s.close()
    q, k, v = qkv.double()
    dead = torch.arange(L, device="cuda") >= lens.view(B, 1, 1)
    score = (q @ k.transpose(-1, -2) / math.sqrt(width)).masked_fill(dead.view(B, 1, 1, L), -math.inf)
    p = score.softmax(-1)
    dz = (logits.softmax(-1) - torch.nn.functional.one_hot(labels.long(), CLASSES)) / B
    do = (dz[:, :1].float().bfloat16().double() * head[0].double()).reshape(B, L, heads, width).permute(0, 2, 1, 3)
    ds = p * (do @ v.transpose(-1, -2) - (do * o).sum(-1, keepdim=True)) / math.sqrt(width)
    exact = {"O": p @ v, "dQ": ds @ k, "dK": ds.transpose(-1, -2) @ q, "dV": p.transpose(-1, -2) @ do}
    return {"O": o, "dQ": dq, "dK": dk, "dV": dv}, exact


@pytest.mark.parametrize("width,heads,L,B", [(16, 8, 77, 3), (32, 4, 77, 3), (32, 2, 128, 4), (48, 2, 127, 3),
                                             (16, 2, 9, 24), (24, 4, 100, 3)])
def test_fp32_probabilities(width, heads, L, B):
    off = {}
    for seed in range(4):
        got, exact = attention_step(width, heads, L, B, seed)
        for n in got:
            off.setdefault(n, []).append((got[n] != exact[n].float().bfloat16().double()).double().mean().item())
    assert all(sum(v) / len(v) <= 2.0 ** -10 for v in off.values()), off


@pytest.mark.parametrize("width,heads,L", [(16, 2, 9), (32, 4, 77), (48, 2, 127), (24, 4, 100)])
@pytest.mark.parametrize("value", [math.inf, math.nan])
def test_masked_keys_and_other_sequences_stay_out(width, heads, L, value):
    """Keys past a sequence's length that hold infinities or NaN, and a whole
    sequence of them, change nothing of the other sequences.  The packed q|k|v
    passes a unit affine, whose shift gradient is the column sum of d(q|k|v)."""
    B, C = 4, width * heads
    ops = [dict(kind="affine", in0=0, c=3 * C), dict(kind="attention", in0=1, c=C, heads=heads),
           dict(kind="flatten", in0=2), dict(kind="linear", in0=3, cin=L * C, cout=CLASSES, bias=0)]
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn(B, L, 1, 3 * C, generator=g, device="cuda").bfloat16()
    head = torch.randn(CLASSES, L * C, generator=g, device="cuda") * math.sqrt(2.0 / (L * C))
    lens = torch.randint(max(1, L // 4), L, (B,), generator=g, device="cuda", dtype=torch.int32)   # one masked key at least
    labels = torch.arange(B, device="cuda", dtype=torch.int32)
    theta = torch.cat([torch.ones(3 * C, device="cuda"), torch.zeros(3 * C, device="cuda"), head.flatten()]).cpu().numpy()

    def step(batch):
        s = api.Server(ops, 1, 1, 1, B, (L, 1, 3 * C), CLASSES, "bf16", 0.0, 0.0, seq=True)
        s.set_params(theta)
        torch.cuda.synchronize()
        assert s.enqueue_activations(0, batch, labels, lens)[0] == api.OK
        s.server_step()
        s.synchronize()
        s.check_error()
        o = torch.as_tensor(DeviceArray(s.tensor(2)[0], (B, L, C), "<i2"), device="cuda").view(torch.bfloat16).clone()
        v = s.get_momentum()
        s.close()
        return o, v[3 * C:6 * C]

    o0, shift0 = step(x)
    y = x.clone()
    for b in range(B):
        y[b, lens[b]:, :, C:] = value       # keys and values only: every query still counts
    o1, shift1 = step(y)
    assert torch.equal(o1, o0) and (shift1 == shift0).all()
    y[1] = value
    o2, _ = step(y)
    keep = [0, 2, 3]
    assert torch.equal(o2[keep], o0[keep])
