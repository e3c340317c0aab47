"""The rotated column-wise quantizer's warp tiles (128 rows x 16 columns): more
tiles than warps, a last CTA with idle warps, strided rows, every mode, against
the row-wise rotated quantizer on an explicit transpose (same definition, other
kernel)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("R,C,pad", [(128, 16, 0), (256, 48, 16), (1024, 1040, 0), (128, 38928, 0), (4096, 2064, 32)])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("with_signs", [False, True])
def test_equals_row_wise_on_the_transpose(R, C, pad, mode, with_signs):
    from paper_2605_31035_gb300 import ops
    g = torch.Generator(device=DEV).manual_seed(R + C)
    x = torch.zeros(R, C + pad, dtype=torch.bfloat16, device=DEV)[:, :C]
    x.copy_(torch.randn(R, C, generator=g, device=DEV) * 3)
    signs = torch.randint(0, 256, (16,), generator=g, dtype=torch.uint8, device=DEV) if with_signs else None
    a = ops.mixfp4_quantize_colwise_rht(x, signs, mode)
    b = ops.mixfp4_quantize_rht(x.t().contiguous(), signs, mode)
    assert torch.equal(a.tensor_scale, b.tensor_scale)
    assert torch.equal(a.codes, b.codes) and torch.equal(a.scales, b.scales)
