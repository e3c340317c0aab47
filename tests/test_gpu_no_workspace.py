"""The few-row GEMMs that need no workspace: mixfp4_gemm's kernel for M <= 64
(f16 decode) and mixfp4_gemm_native_fewrows' own.  They are the C entry points
of those names and what runs where no scratch memory is to be had; with one,
other kernels run (test_gpu_gemm_ws.py).  Each against the float64 product of
the dequantized operands, within the 1e-5 |A| |B| bound of every GEMM path."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def run(entry, a, b, C):
    from paper_2605_31035_gb300 import ops
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    # An empty workspace declines the forms that need one.
    getattr(ops, entry)(a, b, out=C, status_word=status, workspace=torch.empty(0, dtype=torch.uint8, device=DEV))
    torch.cuda.synchronize()
    assert status.item() == 0


def reference(a, b):
    from paper_2605_31035_gb300 import ops
    A, B = ops.mixfp4_dequantize(a).double(), ops.mixfp4_dequantize(b).double()
    return A @ B.T, 1e-5 * (A.abs() @ B.abs().T)


ENTRIES = ["mixfp4_gemm", "mixfp4_gemm_native_fewrows"]


# The last and first row counts of each activation tile height; one weight row,
# around a weight tile of 128, several tiles a CTA; one K slice, several, beyond
# an accumulation chunk (4096), all CTAs sharing one tile; every mode.
@pytest.mark.parametrize("entry", ENTRIES)
@pytest.mark.parametrize("M,N,K,mode", [(1, 1, 256, 0), (1, 5000, 4352, 0), (16, 127, 512, 0), (16, 513, 8448, 1),
                                        (17, 128, 768, 2), (17, 1000, 256, 0), (32, 129, 2560, 3), (33, 700, 4096, 0),
                                        (64, 513, 256, 0), (64, 41000, 512, 0), (64, 3, 14336, 2), (48, 28672, 1024, 0)])
def test_within_bound(entry, M, N, K, mode):
    from paper_2605_31035_gb300 import ops, synth
    a = ops.mixfp4_quantize(synth.activations(M, K, 9200 + M, 9201).to(DEV), mode)
    b = ops.mixfp4_quantize(synth.weights(N, K, 9202 + M, 0.02, 0.5).to(DEV), mode)
    ref, bound = reference(a, b)
    for width, off in ((N, 0), (N + 5, 3)):    # dense, then inside a wider buffer off 16-byte alignment
        big = torch.full((M + 1, width), -3.0, device=DEV)
        run(entry, a, b, big[:M, off:off + N])
        assert torch.all((big[:M, off:off + N].double() - ref).abs() <= bound)
        assert torch.all(big[:M, :off] == -3.0) and torch.all(big[:M, off + N:] == -3.0) and torch.all(big[M] == -3.0)


@pytest.mark.parametrize("entry", ENTRIES)
def test_extreme_scales(entry):
    """Block scales 0, smallest subnormal, 1 and 448, both types, against every payload and sign."""
    from paper_2605_31035_gb300 import ops
    g = torch.Generator(device="cpu").manual_seed(6)

    def tensor(rows, K):
        codes = torch.randint(0, 256, (rows, K // 2), generator=g, dtype=torch.uint8)
        pick = torch.tensor([0x00, 0x80, 0x01, 0x81, 0x07, 0x87, 0x7E, 0xFE, 0x38, 0xB8], dtype=torch.uint8)
        scales = pick[torch.randint(0, len(pick), (rows, K // 16), generator=g)]
        return ops.QTensor(codes.to(DEV), scales.to(DEV), torch.tensor([0.5], device=DEV))
    a, b = tensor(33, 1024), tensor(200, 1024)
    C = torch.full((33, 200), float("nan"), device=DEV)
    run(entry, a, b, C)
    ref, bound = reference(a, b)
    assert torch.all((C.double() - ref).abs() <= bound)


@pytest.mark.parametrize("entry", ENTRIES)
def test_called_again_and_captured(entry):
    """C is zeroed by each call, in a graph too."""
    from paper_2605_31035_gb300 import ops, synth
    a = ops.mixfp4_quantize(synth.activations(16, 2816, 9210, 9211).to(DEV))
    b = ops.mixfp4_quantize(synth.weights(1100, 2816, 9212, 0.02, 0.5).to(DEV))
    ref, bound = reference(a, b)
    C = torch.full((16, 1100), 7.0, device=DEV)
    ws = torch.empty(0, dtype=torch.uint8, device=DEV)
    g = torch.cuda.CUDAGraph()
    getattr(ops, entry)(a, b, out=C, workspace=ws)
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        getattr(ops, entry)(a, b, out=C, workspace=ws)
    for _ in range(3):
        C.fill_(7.0)
        g.replay()
        assert torch.all((C.double() - ref).abs() <= bound)
