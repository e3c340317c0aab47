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


# Many rows and one column of weight tiles (N <= 256): the activations stay codes,
# which the GEMM decodes once, instead of 2 bytes an element.  Both sides of each
# bound: half a wave of 256-row tiles (one tile more than half of the pairs), 2^25
# elements, 256 columns; ragged rows, a row stride above K, every mode.
@pytest.mark.parametrize("tiles,extra,N,K,mode,pad,codes", [
    (0, 1, 256, 4096, 0, 0, True), (0, 0, 256, 4096, 0, 0, False), (0, 1, 257, 4096, 0, 0, False),
    (10, -3, 1, 2816, 1, 16, True), (0, 1, 64, 3328, 2, 0, False), (0, 7, 100, 4352, 3, 64, True)])
def test_linear_one_column_of_tiles(tiles, extra, N, K, mode, pad, codes):
    from paper_2605_31035_gb300 import ops, synth
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    M = (pairs // 2 + tiles) * 256 + extra
    assert codes == (N <= 256 and 2 * ((M + 255) // 256) > pairs and M * K >= 1 << 25)
    x = torch.zeros(M, K + pad, dtype=torch.bfloat16, device=DEV)[:, :K]
    x.copy_(synth.activations(M, K, 8610, 8611))
    w = ops.mixfp4_quantize(synth.weights(N, K, 8612, 0.02, 0.5).to(DEV), mode)
    q = ops.mixfp4_quantize(x, mode)
    ws = torch.zeros(ops.linear_workspace_bytes(M, N, K), dtype=torch.uint8, device=DEV)
    y = ops.linear(x, w, mode, workspace=ws)
    A, B = ops.mixfp4_dequantize(q).double(), ops.mixfp4_dequantize(w).double()
    assert torch.all((y.double() - A @ B.T).abs() <= 1e-5 * (A.abs() @ B.abs().T))
    header = 2048 * 4 + 256    # the maxima and s32 come first
    assert torch.equal(ws[header:header + M * (K // 2)].view(M, K // 2), q.codes) == codes


# The activations' maximum is reduced from one word per CTA of the first pass (456
# on 152 SMs, 1216 beyond 2^23 blocks): the largest value in the blocks of the
# first, the last and middle CTAs, at the tensor's ends and in later rounds.
@pytest.mark.parametrize("M,N,K", [(2048, 600, 4096), (33000, 300, 4096)])
def test_linear_finds_the_maximum_anywhere(M, N, K):
    from paper_2605_31035_gb300 import ops, synth
    g = torch.Generator(device=DEV).manual_seed(5)
    x = (torch.randn(M, K, generator=g, device=DEV) * 0.01).to(torch.bfloat16)
    w = ops.mixfp4_quantize(synth.weights(N, K, 8620, 0.02, 0.5).to(DEV))
    B = ops.mixfp4_dequantize(w).double()
    nblocks = M * K // 16
    ctas = torch.cuda.get_device_properties(0).multi_processor_count * (8 if nblocks > 1 << 23 else 3)
    for cta in (0, 1, 255, 256, 300, ctas - 1):
        for rnd in (0, 2):
            block = nblocks - 1 - (rnd * ctas * 256 + cta * 256 + 37)    # the pass reads from the end
            if block < 0:
                continue
            r, c = divmod(block * 16 + 11, K)
            old = x[r, c].clone()
            x[r, c] = -100.0
            rows = torch.tensor([r, (r + M // 2) % M], device=DEV)
            q = ops.mixfp4_quantize(x)
            A = ops.mixfp4_dequantize(ops.QTensor(q.codes[rows], q.scales[rows], q.tensor_scale)).double()
            y = ops.linear(x, w)[rows].double()
            assert torch.all((y - A @ B.T).abs() <= 1e-5 * (A.abs() @ B.abs().T)), (cta, rnd)
            x[r, c] = old
