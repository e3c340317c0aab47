"""The maximum pass of the two-pass quantizers: wherever the largest element
lies, the tensor scale is the same, bit for bit, on sizes with one and several
trips of the pass's grid, ragged ends and padded rows, and with the tensor
written by the kernel just before on the same stream."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def quantizers():
    from paper_2605_31035_gb300 import ops
    return {"rows": ops.mixfp4_quantize, "2d": ops.mixfp4_quantize_2d, "colwise": ops.mixfp4_quantize_colwise,
            "sr": lambda x: ops.mixfp4_quantize_sr(x, 5),
            "rht": lambda x: ops.mixfp4_quantize_rht(x),
            "colwise_rht": lambda x: ops.mixfp4_quantize_colwise_rht(x)}


@pytest.mark.parametrize("kind", ["rows", "2d", "colwise", "sr", "rht", "colwise_rht"])
@pytest.mark.parametrize("rows,K,pad", [(128, 4096, 0), (256, 2176, 64), (2176, 4096, 0), (1920, 4224, 32)])
def test_scale_whatever_the_place_of_the_maximum(kind, rows, K, pad):
    fn = quantizers()[kind]
    x = torch.zeros(rows, K + pad, dtype=torch.bfloat16, device=DEV)
    if pad:
        x[:, K:] = 1.0e4                        # outside the tensor
    view = x[:, :K]
    n, seen = rows * K, set()
    # Rotated: one element alone in its 128 spreads to |y| = v c everywhere in
    # its chunk, so the maximum is the same wherever it lies.
    for pos in (0, 1, 15, K - 1, K, n // 2, n - K, n - 17, n - 1, 7 * n // 16, 456 * 256 * 16 % n, 5 * n // 8 + 3):
        r, c = divmod(pos, K)
        view[r, c] = -24.0                      # written by the kernel before the call
        seen.add(fn(view).tensor_scale.item())
        view[r, c] = 0.0
    assert len(seen) == 1 and 0.0 < seen.pop() < 1.0
