"""Encoder blocks whose heads are 16, 32 and 48 wide (the tensor-core kernels,
whose 64-column tiles then reach into the neighbouring head or past the last)
and 24 wide (the CUDA-core kernels), at lengths on both sides of a 64-key
sub-tile and of the 128-token tile, with one head and several.  bf16 steps
under the gates of harness.gate_failures."""
import pytest

from harness import check_teacher_forced, teacher_forced
from paper_2504_13850_gb300 import api, build
from paper_2504_13850_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


@pytest.mark.parametrize("width,heads,length", [(32, 8, 77), (32, 1, 128), (32, 3, 64), (16, 8, 65), (16, 2, 9),
                                                (48, 4, 127), (48, 2, 33), (24, 4, 40)])
def test_block(width, heads, length):
    d = width * heads
    cfg = W.shrink(W.CONFIGS["transformer"],
                   ops=W.transformer_ops(d=d, heads=heads, ffn=2 * d, blocks=1, classes=5), batch=16,
                   in_hwc=(length, 1, d), K=2, omega=4, depth=2, lr=1e-3, classes=5)
    ev = [("enq", k) for _ in range(2) for k in range(2)] + [("step",)] * 4
    _, _, recs = teacher_forced(cfg, ev)
    assert len(recs) == 4
    check_teacher_forced(recs)
