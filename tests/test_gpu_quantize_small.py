"""Small tensors quantized in one launch (a cluster holding the whole tensor)
against the given-scale kernel on the same values: every edge of the sizes it
takes, strided rows, all modes, tensor scales outside the plain range."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


# One block; fewer blocks than a cluster has threads; the last size of one to
# four blocks a thread and the first beyond (4096 threads; 64 x 4096 is 16384
# blocks, the largest taken).
@pytest.mark.parametrize("rows,K", [(1, 16), (7, 48), (1, 65536), (1, 65552), (16, 8192), (47, 4096), (64, 4096),
                                    (65, 4096)])
@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("pad,factor", [(0, 1.0), (32, 1.0), (0, 2.0 ** -60), (16, 2.0 ** 100)])
def test_one_launch_equals_given_scale(rows, K, mode, pad, factor):
    from paper_2605_31035_gb300 import ops
    g = torch.Generator(device="cpu").manual_seed(rows * 131 + K + mode)
    x = torch.zeros(rows, K + pad, dtype=torch.bfloat16, device=DEV)[:, :K]
    x.copy_(torch.randn(rows, K, generator=g) * factor)
    q = ops.mixfp4_quantize(x, mode)
    s32 = (x.abs().max().float().cpu() / torch.tensor(2688.0)).to(DEV)
    assert torch.equal(q.tensor_scale, s32.reshape(1))
    ref = ops.mixfp4_quantize(x, mode, tensor_scale=s32)
    assert torch.equal(q.codes, ref.codes) and torch.equal(q.scales, ref.scales)


def test_zero_tensor():
    from paper_2605_31035_gb300 import ops
    q = ops.mixfp4_quantize(torch.zeros(3, 64, dtype=torch.bfloat16, device=DEV))
    assert q.tensor_scale.item() == 0.0 and torch.all(q.scales == 0x80) and torch.all(q.codes == 0)


# linear() on few rows quantizes straight into the GEMM's operand up to 16384
# blocks of 16 (32 or 64) rows and through codes beyond: the same values.
@pytest.mark.parametrize("M,K", [(1, 4096), (16, 4096), (17, 8192), (33, 4096), (64, 4096), (33, 8192), (5, 28672)])
def test_linear_few_rows_equals_quantize_then_gemm(M, K):
    from paper_2605_31035_gb300 import ops, synth
    x = synth.activations(M, K, 8800 + M, 8801).to(DEV)
    w = ops.mixfp4_quantize(synth.weights(300, K, 8802, 0.02, 0.5).to(DEV))
    # Same operand values, same kernel, same order of sums: equal bits.
    assert torch.equal(ops.linear(x, w), ops.mixfp4_gemm(ops.mixfp4_quantize(x), w))
