"""Evaluations in a row without a wait between them, on images whose contents change
and on alternating or repeated buffers (launched, captured, replayed), against the
same evaluations synchronised one by one: bit for bit."""
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [("fp16x3", 64, 1, False), ("fp16x3", 64, 3, False), ("fp16x3", 128, 3, True), ("fp16x3", 256, 1, False),
         ("bf16x3", 64, 1, False), ("bf16x3", 128, 2, True), ("bf16x3", 256, 1, False), ("fp32_direct", 32, 2, False),
         ("fp64_direct", 64, 1, False)]


@pytest.mark.parametrize("buffers", [1, 2, 3])
@pytest.mark.parametrize("form,N,C,shared", CASES)
def test_calls_in_a_row(form, N, C, shared, buffers):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = S.random_problem(N, 0, 61, C=C, z_list=[700 + 100 * c for c in range(C)], shared_image=shared, lam=1.0)
    base = torch.from_numpy(ds.truth).cuda()
    rounds = 24

    def image(k):
        return base * (1.0 + 0.01 * k)

    def evaluate(ctx, wait):
        imgs = [torch.empty_like(base) for _ in range(buffers)]
        grads = [torch.empty_like(base) for _ in range(buffers)]
        kept = []
        for k in range(rounds):
            b = k % buffers
            imgs[b].copy_(image(k))
            if wait:
                torch.cuda.synchronize()
            scalars = ms.mem_objective_grad(ctx.handle, imgs[b], grads[b], k % 2 if buffers == 1 and k > 12 else 0,
                                            want_scalars=wait or k % 5 == 4)
            vis = ctx.forward(imgs[b])
            back = ctx.adjoint(vis)
            if wait:
                torch.cuda.synchronize()
            kept.append((scalars, grads[b].clone(), vis, back))
        ctx.sync()
        return kept

    ctx = ms.Context(ds, precision=form)
    want = evaluate(ctx, True)
    for _ in range(2):
        for (sa, *ta), (sb, *tb) in zip(evaluate(ctx, False), want):
            assert sa is None or sa == sb
            assert all(torch.equal(a, b) for a, b in zip(ta, tb))
    ctx.close()
