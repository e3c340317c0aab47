"""The GEMM with A decoded to f16 beforehand (mixfp4_gemm_ws): every edge of
its tiles and of its K split against the float64 product of the dequantized
operands, within the 1e-5 |A| |B| bound of every GEMM path, and equal
dispatch results without a workspace."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def operands(M, N, K, seed):
    from paper_2605_31035_gb300 import ops, synth
    x = synth.activations(M, K, seed, seed + 1).to(DEV)
    w = synth.weights(N, K, seed + 2, 0.02, 0.5).to(DEV)
    return ops.mixfp4_quantize(x), ops.mixfp4_quantize(w)


def reference(a, b):
    from paper_2605_31035_gb300 import ops
    A, B = ops.mixfp4_dequantize(a).double(), ops.mixfp4_dequantize(b).double()
    # The fp32 dequantization rounds v s8 s32 once per element: 2^-24 relative
    # on each factor, 1.2e-7 of |A| |B| in all, inside the 1e-5 bound.
    return A @ B.T, A.abs() @ B.abs().T


def call(a, b, C, ws):
    from paper_2605_31035_gb300 import ops
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    p = ops._ptr
    st = ops.lib().mixfp4_gemm_ws(p(a.codes), p(a.scales), p(a.tensor_scale), p(b.codes), p(b.scales),
                                  p(b.tensor_scale), a.rows, b.rows, a.K, p(C), C.stride(0), p(ws),
                                  0 if ws is None else ws.numel(), p(status),
                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    torch.cuda.synchronize()
    assert status.item() == 0


# Sizes at which the decode pass is taken: one row and one column past a tile,
# the narrowest tiles, several waves, K split over all pairs (few tiles, long
# K), K over several accumulation chunks, N not a multiple of 4 (C row stride
# without 16-byte alignment).
@pytest.mark.parametrize("M,N,K", [(65, 96, 2304), (256, 97, 2560), (257, 300, 2304), (129, 33, 4352),
                                   (100, 512, 14336), (300, 1000, 8192), (777, 3000, 2816), (513, 4101, 2560),
                                   (2050, 4100, 2304), (700, 301, 8448)])
def test_decoded_a_within_bound(M, N, K):
    from paper_2605_31035_gb300 import ops
    a, b = operands(M, N, K, 8100 + M)
    need = ops.gemm_workspace_bytes(M, N, K)
    assert need >= 2 * M * K
    C = torch.full((M, N), float("nan"), device=DEV)
    call(a, b, C, torch.empty(need, dtype=torch.uint8, device=DEV))
    ref, D = reference(a, b)
    assert torch.all((C.double() - ref).abs() <= 1e-5 * D)
    C2 = torch.full((M, N), float("nan"), device=DEV)
    call(a, b, C2, None)                       # no workspace: A decoded in the main loop
    assert torch.all((C2.double() - ref).abs() <= 1e-5 * D)


def test_strided_and_unaligned_output():
    """C inside a wider buffer, whose base and row stride are 4-byte aligned
    only: the columns around it stay untouched."""
    from paper_2605_31035_gb300 import ops
    M, N, K = 300, 500, 2560
    a, b = operands(M, N, K, 8500)
    ws = torch.empty(ops.gemm_workspace_bytes(M, N, K), dtype=torch.uint8, device=DEV)
    ref, D = reference(a, b)
    for width, off in ((512, 8), (507, 3)):
        big = torch.full((M, width), -3.0, device=DEV)
        call(a, b, big[:, off:off + N], ws)
        assert torch.all((big[:, off:off + N].double() - ref).abs() <= 1e-5 * D)
        assert torch.all(big[:, :off] == -3.0) and torch.all(big[:, off + N:] == -3.0)


# The few-row path (M <= 64): the last row counts of its three operand widths
# and the first beyond, one weight row, one before and after a 128-row tile, one
# and several units of K, K in one and in many parts, every block type mix.
@pytest.mark.parametrize("M,N,K,mode", [(1, 1, 256, 0), (16, 129, 512, 0), (17, 127, 768, 2), (32, 4096, 1280, 0),
                                        (33, 300, 4352, 0), (64, 700, 14336, 0), (5, 20000, 1024, 1),
                                        (64, 513, 256, 3), (2, 300, 8192, 2), (48, 28672, 512, 0)])
def test_few_rows_within_bound(M, N, K, mode):
    from paper_2605_31035_gb300 import ops, synth
    a = ops.mixfp4_quantize(synth.activations(M, K, 8700 + M, 8701).to(DEV), mode)
    b = ops.mixfp4_quantize(synth.weights(N, K, 8702 + M, 0.02, 0.5).to(DEV), mode)
    ws = torch.empty(ops.gemm_workspace_bytes(M, N, K), dtype=torch.uint8, device=DEV)
    ref, D = reference(a, b)
    for width, off in ((N, 0), (N + 5, 3)):    # dense, then inside a wider buffer off 16-byte alignment
        big = torch.full((M, width), -3.0, device=DEV)
        call(a, b, big[:, off:off + N], ws)
        assert torch.all((big[:, off:off + N].double() - ref).abs() <= 1e-5 * D)
        assert torch.all(big[:, :off] == -3.0) and torch.all(big[:, off + N:] == -3.0)


# Epilogue warps share the rows in turns of eight and take them in pairs: row
# counts that leave one, two or all of a quarter's warps a partial turn, an odd
# last row, with several tiles a CTA (K whole) and with K in parts.
@pytest.mark.parametrize("M", [7, 15, 31, 39, 41, 57, 63])
@pytest.mark.parametrize("N,K", [(41000, 256), (1100, 2816)])
def test_few_rows_epilogue_turns(M, N, K):
    from paper_2605_31035_gb300 import ops
    a, b = operands(M, N, K, 8800 + M)
    ws = torch.empty(max(ops.gemm_workspace_bytes(M, N, K), 1), dtype=torch.uint8, device=DEV)
    C = torch.full((M + 1, N), -3.0, device=DEV)
    call(a, b, C[:M], ws)
    ref, D = reference(a, b)
    assert torch.all((C[:M].double() - ref).abs() <= 1e-5 * D)
    assert torch.all(C[M] == -3.0)


def test_few_rows_extreme_scales():
    """Blocks whose scale is 0, the smallest subnormal and 448, in both types,
    against every payload and sign."""
    from paper_2605_31035_gb300 import ops
    g = torch.Generator(device="cpu").manual_seed(5)
    def tensor(rows, K):
        codes = torch.randint(0, 256, (rows, K // 2), generator=g, dtype=torch.uint8)
        pick = torch.tensor([0x00, 0x80, 0x01, 0x81, 0x07, 0x87, 0x7E, 0xFE, 0x38, 0xB8], dtype=torch.uint8)
        scales = pick[torch.randint(0, len(pick), (rows, K // 16), generator=g)]
        return ops.QTensor(codes.to(DEV), scales.to(DEV), torch.tensor([0.5], device=DEV))
    a, b = tensor(20, 1024), tensor(200, 1024)
    ws = torch.empty(ops.gemm_workspace_bytes(20, 200, 1024), dtype=torch.uint8, device=DEV)
    C = torch.full((20, 200), float("nan"), device=DEV)
    call(a, b, C, ws)
    ref, D = reference(a, b)
    assert torch.all((C.double() - ref).abs() <= 1e-5 * D)


def test_small_products_take_no_workspace():
    from paper_2605_31035_gb300 import ops
    need = ops.gemm_workspace_bytes
    assert need(8000, 300, 8192) == 0         # one tile column: nothing to save
    assert need(0, 4096, 4096) == 0 and need(100, 0, 4096) == 0
