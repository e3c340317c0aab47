"""A call's own memory belongs to the stream the call runs on: checked on CPU with
the allocator, the streams and the library replaced by recorders."""
import contextlib

import pytest
import torch


class Stream:
    """What a caller may pass as `stream`: anything with a raw stream handle."""

    def __init__(self, handle, device=None):
        self.cuda_stream = handle


@pytest.fixture
def calls(monkeypatch):
    """(ops, log): log lists (what, shape or pointer, raw stream it happened on)."""
    from paper_2605_31035_gb300 import ops
    log, current = [], [1]

    @contextlib.contextmanager
    def on(stream):
        current.append(stream.cuda_stream)
        yield
        current.pop()

    class Lib:
        def __getattr__(self, name):
            def call(*args):
                if name.endswith("_workspace"):
                    args[-1]._obj.value = 4096
                    return 0
                log.append((name, args[-1]))
                return 0
            return call

    empty, copy_ = torch.empty, torch.Tensor.copy_

    def recorded_empty(*shape, dtype=None, device=None):
        shape = shape[0] if len(shape) == 1 else shape
        log.append(("empty", tuple(shape) if isinstance(shape, (tuple, list, torch.Size)) else (shape,), current[-1]))
        return empty(shape, dtype=dtype, device=device)

    def recorded_copy(self, src):
        log.append(("copy", None, current[-1]))
        return copy_(self, src)
    monkeypatch.setattr(torch, "empty", recorded_empty)
    monkeypatch.setattr(torch.Tensor, "copy_", recorded_copy)
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda self, s: log.append(("record", self.shape, s.cuda_stream)))
    monkeypatch.setattr(torch.cuda, "stream", on)
    monkeypatch.setattr(torch.cuda, "ExternalStream", Stream)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: Stream(current[-1]))
    monkeypatch.setattr(ops, "_stream", lambda stream=None: current[-1] if stream is None else stream.cuda_stream)
    monkeypatch.setattr(ops, "lib", lambda lib=Lib(): lib)
    monkeypatch.setattr(ops, "_check_x", lambda t: None)
    monkeypatch.setattr(ops, "_check_dev", lambda t, device, what: None)
    return ops, log


def qt(ops, rows, K):
    return ops.QTensor(torch.zeros(rows, K // 2, dtype=torch.uint8), torch.zeros(rows, K // 16, dtype=torch.uint8),
                       torch.ones(1))


CALLS = {
    "gemm": lambda o, s: o.mixfp4_gemm(qt(o, 80, 256), qt(o, 16, 256), stream=s),
    "gemm_out": lambda o, s: o.mixfp4_gemm(qt(o, 80, 256), qt(o, 16, 256), out=torch.zeros(80, 16), stream=s),
    "fewrows_out": lambda o, s: o.mixfp4_gemm_native_fewrows(qt(o, 8, 256), qt(o, 16, 256), out=torch.zeros(8, 16),
                                                             stream=s),
    "linear": lambda o, s: o.linear(torch.zeros(8, 256, dtype=torch.bfloat16), qt(o, 16, 256), stream=s),
    "quantize": lambda o, s: o.mixfp4_quantize(torch.zeros(8, 256, dtype=torch.bfloat16), stream=s),
    "quantize_given": lambda o, s: o.mixfp4_quantize(torch.zeros(8, 256, dtype=torch.bfloat16),
                                                     tensor_scale=torch.ones(1), stream=s),
    "fake": lambda o, s: o.mixfp4_fake_quantize(torch.zeros(8, 256, dtype=torch.bfloat16), 3,
                                                tensor_scale=torch.ones(1), stream=s),
    "dequantize": lambda o, s: o.mixfp4_dequantize(qt(o, 8, 256), stream=s),
    "transpose_2d": lambda o, s: o.mixfp4_transpose_2d(qt(o, 16, 256), stream=s),
    "split_native": lambda o, s: o.mixfp4_split_native(qt(o, 16, 256), stream=s),
}


@pytest.mark.parametrize("name", CALLS)
def test_allocations_and_copies_on_the_calls_stream(calls, name):
    """Another stream than the current one: a block that the allocator hands out
    on the current stream may still be in use there."""
    ops, log = calls
    CALLS[name](ops, Stream(7))
    made = [e for e in log if e[0] in ("empty", "copy")]
    assert made and all(e[2] == 7 for e in made), log
    # Results are recorded on the current stream, where the caller uses and drops them; scratch is not.
    results = {"gemm": [(80, 16)], "linear": [(8, 16)], "dequantize": [(8, 256)],
               "quantize": [(8, 128), (8, 16), (1,)]}
    if name in results:
        assert [tuple(e[1]) for e in log if e[0] == "record"] == results[name]


@pytest.mark.parametrize("name", CALLS)
def test_current_stream_needs_no_recording(calls, name):
    ops, log = calls
    for stream in (None, Stream(1)):
        CALLS[name](ops, stream)
    assert all(e[2] == 1 for e in log if e[0] in ("empty", "copy"))
    assert not [e for e in log if e[0] == "record"]


WITH_WORKSPACE = {
    "gemm": lambda o, w: o.mixfp4_gemm(qt(o, 80, 256), qt(o, 16, 256), out=torch.zeros(80, 16), workspace=w),
    "fewrows": lambda o, w: o.mixfp4_gemm_native_fewrows(qt(o, 8, 256), qt(o, 16, 256), out=torch.zeros(8, 16),
                                                         workspace=w),
}


@pytest.mark.parametrize("nbytes", [0, 4095, 4096, 10000])
@pytest.mark.parametrize("name", WITH_WORKSPACE)
def test_a_given_workspace_leaves_nothing_to_allocate(calls, name, nbytes):
    """Output and workspace the caller's: no allocation, whether the workspace is large enough or not."""
    ops, log = calls
    WITH_WORKSPACE[name](ops, torch.zeros(nbytes, dtype=torch.uint8))
    assert not [e for e in log if e[0] == "empty"]
    # The library gets the workspace, or (native few rows) the form that needs none runs.
    native_form = name == "fewrows" and nbytes < 4096
    assert log[-1][0] == ("mixfp4_gemm_native_fewrows" if native_form else "mixfp4_gemm_ws")


def test_linear_with_a_workspace_allocates_its_result_only(calls):
    ops, log = calls
    x, w = torch.zeros(8, 256, dtype=torch.bfloat16), qt(ops, 16, 256)
    ops.linear(x, w, workspace=torch.zeros(4096, dtype=torch.uint8))
    assert [e[1] for e in log if e[0] == "empty"] == [(8, 16)]
    with pytest.raises(ValueError, match="workspace"):
        ops.linear(x, w, workspace=torch.zeros(64, 128, dtype=torch.uint8).t())


def test_linear_without_room_for_scratch_makes_its_result_once(calls, monkeypatch):
    """Where the device has no room left for scratch, a second result would not
    fit either: the two calls write the one already made."""
    ops, log = calls
    monkeypatch.setattr(ops, "_scratch", lambda *args: None)
    y = ops.linear(torch.zeros(80, 256, dtype=torch.bfloat16), qt(ops, 24, 256))
    assert [e[1] for e in log if e[0] == "empty"].count((80, 24)) == 1 and y.shape == (80, 24)
    assert [e[0] for e in log if e[0].startswith("mixfp4")] == ["mixfp4_quantize", "mixfp4_gemm_ws"]
