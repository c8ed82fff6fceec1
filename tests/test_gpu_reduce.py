"""Row sums (cr_reduce_rows): every split of a row over blocks, piece remainders and both types."""
import pytest
import torch

from paper_2607_11340_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("rows", [1, 6, 40, 200])
@pytest.mark.parametrize("B", [1, 31, 511, 513, 4095, 4096, 8191, 16385, 40000, 65537, 262145])
def test_row_sums(rows, B, dtype):
    g = torch.Generator(device="cuda").manual_seed(B * 1000 + rows)
    x = torch.randn(rows, B, dtype=dtype, device="cuda", generator=g)
    out = api.reduce_rows(x)
    ref = x.double().sum(1)
    # each side adds B FP64 values: at most B 2^-53 sum |x| off the exact sum
    assert torch.all((out - ref).abs() <= 2 * B * 2.0 ** -53 * x.double().abs().sum(1))
    assert torch.equal(out, api.reduce_rows(x))  # a fixed order
