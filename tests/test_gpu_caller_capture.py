"""The entry points without a context recorded into a caller's own CUDA graph, behind a copy, a kernel or nothing, and replayed."""
import numpy as np
import pytest

import paper_1705_04862_b200.binding as pb

pytestmark = pytest.mark.gpu


def _calls(torch, gen):
    raw = [torch.randint(0, 256, (3, 210, 160, 3), dtype=torch.uint8, generator=gen).cuda() for _ in range(2)]
    state = torch.randint(0, 256, (3, 84, 84, 4), dtype=torch.uint8, generator=gen).cuda()
    plane = torch.randint(0, 256, (3, 84, 84), dtype=torch.uint8, generator=gen).cuda()
    grad = torch.randn(100000, generator=gen).cuda()
    theta = torch.randn(100000, generator=gen).cuda()

    def preprocess(src, out, stream):
        return pb.preprocess(raw[0], raw[1], src, out, 3, stream=stream)

    def push(src, out, stream):
        return pb.stack_push(src, plane, None, out, 3, stream=stream)

    def optimizer(src, out, stream):
        return pb.clip_rmsprop_noalloc(out[0], out[1], src, 100000, 0.02, 0.99, 0.1, 40.0, stream=stream)

    return {"preprocess": (preprocess, state, lambda: torch.zeros_like(state)), "stack": (push, state, lambda: torch.zeros_like(state)),
            "optimizer": (optimizer, grad, lambda: torch.stack([theta, torch.ones_like(theta)]))}


@pytest.mark.parametrize("before", ["nothing", "copy", "kernel"])
@pytest.mark.parametrize("name", ["preprocess", "stack", "optimizer"])
def test_recorded_by_the_caller(name, before):
    import torch
    call, src, fresh = _calls(torch, torch.Generator().manual_seed(5))[name]
    want = fresh()
    staged = torch.zeros_like(src) if before != "nothing" else src
    out = fresh()
    torch.cuda.synchronize()
    assert call(src, want, torch.cuda.current_stream().cuda_stream) == pb.OK
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        if before == "copy":
            staged.copy_(src)
        elif before == "kernel":
            torch.bitwise_xor(src, 0, out=staged) if src.dtype == torch.uint8 else torch.mul(src, 1.0, out=staged)
        status = call(staged, out, torch.cuda.current_stream().cuda_stream)
    assert status == pb.OK
    for _ in range(2):
        out.copy_(fresh())
        if before != "nothing":
            staged.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want.cpu().numpy())
