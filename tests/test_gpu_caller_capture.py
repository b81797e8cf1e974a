"""Calls captured into a caller's CUDA graph on the context's stream: the first call
after mem_create or mem_set_tiling may be the captured one (nothing is left to
allocate), the replay follows new contents of the same buffers, and its results are
the direct calls' bit for bit."""
import ctypes

import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [("fp16x3", 64, None), ("fp16x3", 256, None), ("fp16x3", 256, ("resident", 256, 4, 2)),
         ("bf16x3", 128, None), ("bf16x3", 256, ("resident", 256, 4, 3)), ("fp32_direct", 48, None),
         ("fp64_direct", 80, None)]


@pytest.mark.parametrize("form,N,tiling", CASES, ids=lambda v: str(v[0]) if isinstance(v, tuple) else str(v))
def test_captured_calls(form, N, tiling):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = S.random_problem(N, 700, 53, lam=1.0)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        ctx = ms.Context(ds, precision=form)
        ms.mem_use_graphs(ctx.handle, False)
        if tiling is not None:
            ctx.set_tiling(*tiling)
        img = torch.from_numpy(ds.truth).cuda()
        y = torch.full((ds.Z, 2), 0.25, device="cuda")
        grad = torch.empty_like(img)
        lib = ms.load()
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731

        def calls():
            assert lib.mem_objective_grad(ctx.handle, ptr(img), ptr(grad), 0, None) == 0
            return [grad, ctx.forward(img), ctx.adjoint(y)]

        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            got = calls()
        for k in range(3):
            img.mul_(1.0 + 0.125 * k)
            y.mul_(-1.5)
            graph.replay()
            kept = [t.clone() for t in got]
            want = [t.clone() for t in calls()]
            side.synchronize()
            for a, b in zip(kept, want):
                assert torch.equal(a, b)
        ctx.sync()
        del graph
        ctx.close()
