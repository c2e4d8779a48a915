"""Calls run on the calling thread's current stream, whichever that is at the call."""
import threading

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def test_current_stream_of_each_call_and_thread():
    import paper_2403_18647_gb300 as sd
    assert sd._stream() == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert sd._stream() == side.cuda_stream
    seen = []

    def other():
        with torch.cuda.stream(side):
            seen.append(sd._stream())
        seen.append(sd._stream())

    t = threading.Thread(target=other)
    t.start()
    t.join()
    assert seen == [side.cuda_stream, torch.cuda.default_stream().cuda_stream]
    # a call on the side stream is ordered with that stream's work
    shape = synth.ModelShape("s", 1, 128, 1, 128, 256, 256, 0)
    ctx = sd.Context(shape, None, max_position=64)
    x, w = synth.normal_f32(1, 1, (6, 256), device="cuda"), synth.normal_bf16(1, 2, (512, 256), 0.02, device="cuda")
    a, b = torch.empty(6, 512, device="cuda"), torch.empty(6, 512, device="cuda")
    ctx.op_gemm(x, w, a)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        ctx.op_gemm(x, w, b)
        c = b.clone()
    side.synchronize()
    assert torch.equal(a, c)
