"""A GEMM on one stream while another, the current one, still has work pending:
the call's scratch is not taken from memory which that work uses."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


# Few rows (operand and parts as scratch), A decoded beforehand, the native few-row entry, the layer.
@pytest.mark.parametrize("call,M", [("gemm", 16), ("gemm", 300), ("fewrows", 16), ("linear", 16), ("linear", 300)])
def test_scratch_while_the_current_stream_is_busy(call, M):
    from paper_2605_31035_gb300 import ops, synth
    N, K = 1000, 2560
    x = synth.activations(M, K, 9100, 9101).to(DEV)
    w = ops.mixfp4_quantize(synth.weights(N, K, 9102, 0.02, 0.5).to(DEV))
    a = ops.mixfp4_quantize(x)
    run = {"gemm": lambda s: ops.mixfp4_gemm(a, w, out=C, stream=s),
           "fewrows": lambda s: ops.mixfp4_gemm_native_fewrows(a, w, out=C, stream=s),
           "linear": lambda s: ops.linear(x, w, stream=s)}[call]
    C = torch.empty(M, N, device=DEV)
    ref = run(None).clone()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    # A block of every size the call may ask for, read by work that is still
    # pending when its tensor has been freed.
    sizes = sorted({max(ops.gemm_workspace_bytes(M, N, K), 1), 2 * M * K + 16384, 1 << 21, 1 << 22})
    blocks = [torch.ones(n, dtype=torch.uint8, device=DEV) for n in sizes]
    torch.cuda._sleep(50_000_000)  # some 25 ms
    sums = [b.sum(dtype=torch.int64) for b in blocks]
    del blocks
    y = run(side)
    side.synchronize()
    assert torch.equal(y, ref)
    assert [int(s) for s in sums] == sizes


# The caller's workspace: as large as asked for, one byte short (a few rows and
# many then run the forms that need none) and empty; nothing is allocated.
@pytest.mark.parametrize("M", [16, 300])
def test_callers_workspace(M):
    from paper_2605_31035_gb300 import ops, synth
    N, K = 1000, 2560
    x = synth.activations(M, K, 9110, 9111).to(DEV)
    w = ops.mixfp4_quantize(synth.weights(N, K, 9112, 0.02, 0.5).to(DEV))
    a = ops.mixfp4_quantize(x)
    A, B = ops.mixfp4_dequantize(a).double(), ops.mixfp4_dequantize(w).double()
    ref, bound = A @ B.T, 1e-5 * (A.abs() @ B.abs().T)
    C = torch.empty(M, N, device=DEV)
    entries = [ops.mixfp4_gemm] + ([ops.mixfp4_gemm_native_fewrows] if M <= 64 else [])
    for gemm in entries:
        for n in (ops.gemm_workspace_bytes(M, N, K), ops.gemm_workspace_bytes(M, N, K) - 1, 0):
            ws = torch.empty(n, dtype=torch.uint8, device=DEV)
            C.fill_(float("nan"))
            torch.cuda.synchronize()
            before = torch.cuda.memory_stats()["allocation.all.allocated"]
            gemm(a, w, out=C, workspace=ws)
            assert torch.cuda.memory_stats()["allocation.all.allocated"] == before
            assert torch.all((C.double() - ref).abs() <= bound), (gemm, n)
    for n in (ops.linear_workspace_bytes(M, N, K), 0):
        y = ops.linear(x, w, workspace=torch.empty(n, dtype=torch.uint8, device=DEV))
        assert torch.all((y.double() - ref).abs() <= bound), n
    with pytest.raises(ops.MixFP4Error, match="misaligned"):
        n = ops.gemm_workspace_bytes(M, N, K)
        ops.mixfp4_gemm(a, w, workspace=torch.empty(n + 256, dtype=torch.uint8, device=DEV)[16:16 + n])
