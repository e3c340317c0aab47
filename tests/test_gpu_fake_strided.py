"""Quantize-dequantize with the block position from the flat index (dense
tensors) and from a row and column (strided x or out): equal outputs for every
combination, every block size, at row lengths that are not a power of two."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("block", [8, 16, 32, 64])
@pytest.mark.parametrize("cand", [1, 2, 8, 3, 15])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_strides_do_not_change_the_result(block, cand, dtype):
    from paper_2605_31035_gb300 import ops
    rows, K = 37, 320
    g = torch.Generator(device="cpu").manual_seed(cand * 100 + block)
    dense = torch.randn(rows, K, generator=g).to(torch.bfloat16).to(DEV)
    dense[3] = 0
    dense[5, :64] *= 2.0 ** -30
    wide = torch.full((rows, K + 48), 7.0, dtype=torch.bfloat16, device=DEV)
    wide[:, :K] = dense
    ref, ch, s = ops.mixfp4_fake_quantize(dense, cand, block, dtype)
    for x in (dense, wide[:, :K]):
        buf = torch.full((rows, K + 32), -5.0, dtype=dtype, device=DEV)
        for out in (None, buf[:, :K]):
            o, c, t = ops.mixfp4_fake_quantize(x, cand, block, dtype, out=out)
            assert torch.equal(o, ref) and torch.equal(c.view(-1), ch.view(-1)) and torch.equal(s, t)
        assert torch.all(buf[:, K:] == -5.0)
