"""Layernorms whose width leaves lanes of a vector idle, needs three or four
vectors a lane, or exceeds the vectorised kernels: forward, input gradient and
parameter gradients in an encoder block with a ragged row count, and directly
on the uploaded batch (no input gradient).  bf16 steps under the gates of
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


@pytest.mark.parametrize("d", [32, 288, 544, 768, 1024, 1056])
def test_block(d):
    cfg = W.shrink(W.CONFIGS["transformer"], ops=W.transformer_ops(d=d, heads=d // 32, ffn=128, blocks=1, classes=5),
                   batch=16, in_hwc=(37, 1, d), K=2, omega=4, depth=2, lr=1e-3, classes=5)
    ev = [("enq", k) for _ in range(2) for k in range(2)] + [("step",)] * 4
    _, _, recs = teacher_forced(cfg, ev)
    assert len(recs) == 4
    check_teacher_forced(recs)
