"""Column sums whose row chunks hold more than one block of 128 rows (many rows
and column blocks), with rows and columns that leave the last chunk and the last
column block ragged: against fp64, and the same from the entry point with the
fixed scratch where it takes the size."""
import numpy as np
import pytest
import torch

from paper_2504_13850_gb300 import api, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


@pytest.mark.parametrize("rows,cols", [(155_649, 8), (38_913, 1000), (65_500, 1000), (100_000, 1496), (257, 24_000)])
def test_large_bf16(rows, cols):
    g = torch.Generator(device="cuda").manual_seed(rows + cols)
    x = torch.randn(rows, cols, device="cuda", generator=g).to(torch.bfloat16)
    out = torch.empty(cols, device="cuda")
    assert api.column_sums(x, out) == api.OK
    torch.cuda.synchronize()
    ref, mag = x.double().sum(0).cpu().numpy(), x.double().abs().sum(0).cpu().numpy()
    # a thread adds at most rows / 8 / chunks terms, then 8 lanes and the chunks: far fewer than 2^11
    # roundings of 2^-24 each in a row
    assert np.all(np.abs(out.cpu().numpy() - ref) <= 2.0 ** -13 * mag + 1e-30)
    if (rows + 127) // 128 * cols <= 262144:
        got = torch.empty(cols, device="cuda")
        assert api.column_sums_noalloc(x, got) == api.OK
        torch.cuda.synchronize()
        assert torch.equal(got, out)
