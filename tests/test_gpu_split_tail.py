"""GEMMs whose last tiles are split along K and added into zeroed rows: C dense,
in a wider buffer with 16-byte aligned rows, and in one without, filled with
NaN before; nothing around C changes."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


# 80 to 154 tiles of 256 x 256: one or two whole waves of 76 pairs and a few tiles
# over; an odd number of columns; one row past a tile.
@pytest.mark.parametrize("M,N,K", [(2560, 2000, 2304), (2305, 2047, 2304), (2817, 3581, 2560)])
@pytest.mark.parametrize("extra,off", [(0, 0), (28, 8), (7, 3)])
def test_split_tail_within_bound(M, N, K, extra, off):
    from paper_2605_31035_gb300 import ops, synth
    a = ops.mixfp4_quantize(synth.activations(M, K, 9100, 9101).to(DEV))
    b = ops.mixfp4_quantize(synth.weights(N, K, 9102, 0.02, 0.5).to(DEV))
    A, B = ops.mixfp4_dequantize(a).double(), ops.mixfp4_dequantize(b).double()
    ref, D = A @ B.T, A.abs() @ B.abs().T
    an, bn = ops.mixfp4_split_native(a), ops.mixfp4_split_native(b)
    for fn in (lambda C: ops.mixfp4_gemm_native(an, bn, out=C), lambda C: ops.mixfp4_gemm(a, b, out=C)):
        big = torch.full((M, N + extra), -3.0, device=DEV)
        C = big[:, off:off + N]
        C.fill_(float("nan"))
        fn(C)
        assert torch.all((C.double() - ref).abs() <= 1e-5 * D)
        assert torch.all(big[:, :off] == -3.0) and torch.all(big[:, off + N:] == -3.0)
