"""linear(): one library call for quantization and GEMM, equal to the two
calls it stands for, and the same refusals."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


# One row, the last few-row count and the first beyond it, ragged tiles, a row
# stride above K, every mode.
@pytest.mark.parametrize("M,N,K,mode,pad", [(1, 512, 256, 0, 0), (64, 700, 512, 0, 0), (65, 512, 2304, 1, 16),
                                            (300, 77, 2560, 2, 0), (257, 1030, 2816, 3, 64), (2, 3, 256, 0, 0)])
def test_linear_equals_quantize_then_gemm(M, N, K, mode, pad):
    from paper_2605_31035_gb300 import ops, synth
    x = torch.zeros(M, K + pad, dtype=torch.bfloat16, device=DEV)[:, :K]
    x.copy_(synth.activations(M, K, 8600 + M, 8601))
    w = ops.mixfp4_quantize(synth.weights(N, K, 8602, 0.02, 0.5).to(DEV), mode)
    q = ops.mixfp4_quantize(x, mode)
    y = ops.linear(x, w, mode)
    A, B = ops.mixfp4_dequantize(q).double(), ops.mixfp4_dequantize(w).double()
    D = A.abs() @ B.abs().T
    # Against the float64 product of the same operands: the bound of every GEMM path.
    assert torch.all((y.double() - A @ B.T).abs() <= 1e-5 * D)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    y2 = ops.linear(x, w, mode, stream=s)
    s.synchronize()
    assert torch.all((y2.double() - A @ B.T).abs() <= 1e-5 * D)


def test_linear_empty_and_refusals():
    from paper_2605_31035_gb300 import ops
    w = ops.empty_qtensor(8, 256, DEV)
    assert ops.linear(torch.zeros(0, 256, dtype=torch.bfloat16, device=DEV), w).shape == (0, 8)
    x = torch.zeros(4, 256, dtype=torch.bfloat16, device=DEV)
    with pytest.raises(ValueError, match="share K"):
        ops.linear(x, ops.empty_qtensor(8, 512, DEV))
    with pytest.raises(ops.MixFP4Error, match="mixfp4_quantize"):    # mode out of range
        ops.linear(x, w, 4)
    with pytest.raises(ops.MixFP4Error, match="mixfp4_gemm"):        # K % 256
        ops.linear(torch.zeros(4, 272, dtype=torch.bfloat16, device=DEV), ops.empty_qtensor(8, 272, DEV))
    with pytest.raises(ops.MixFP4Error, match="misaligned"):         # x not 32-byte aligned
        ops.linear(torch.zeros(4, 272, dtype=torch.bfloat16, device=DEV)[:, 8:264], w)
