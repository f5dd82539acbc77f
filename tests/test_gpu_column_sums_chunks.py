"""Column sums whose row chunks hold more than 128 rows (many rows and column
blocks), with rows and columns that leave the last chunk, the last group of rows
in flight and the last column block ragged.  Small whole numbers, none of them
zero: every partial sum is exact in fp32, so a row that is dropped or read twice
shows.  Normal data against fp64, and the entry point with the fixed scratch
where it takes the size."""
import pytest
import torch

from paper_2504_13850_gb300 import api, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    api.lib()


def sums(x, entry=api.column_sums):
    out = torch.empty(x.shape[1], device="cuda")
    assert entry(x, out) == api.OK
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("rows,cols", [(155_649, 8), (38_913, 1000), (65_500, 1000), (100_000, 1496), (257, 24_000),
                                       (129, 16), (8_191, 2040), (1_000_003, 64)])
def test_large_bf16(rows, cols):
    g = torch.Generator(device="cuda").manual_seed(rows + cols)
    x = torch.randint(1, 4, (rows, cols), device="cuda", generator=g)
    x *= 2 * torch.randint(0, 2, x.shape, device="cuda", generator=g) - 1      # -3 .. 3, never 0
    got = sums(x.to(torch.bfloat16))
    assert torch.equal(got.double(), x.sum(0).double())      # below 2^24 in every partial sum
    x = torch.randn(rows, cols, device="cuda", generator=g).to(torch.bfloat16)
    out = sums(x)
    # of the kind of tests/test_gpu_column_sums.py: 1e-5 of the column's magnitude
    assert ((out.double() - x.double().sum(0)).abs() <= 1e-5 * x.double().abs().sum(0) + 1e-30).all()
    if (rows + 127) // 128 * cols <= 262144:
        assert torch.equal(sums(x, api.column_sums_noalloc), out)
