"""The folded (FP16X3) adjoint at its edges against the oracle: one
visibility, stages of 16 and 32 visibilities with remainders, an accumulation
drained in the middle of a unit (more than 8,192 visibilities per unit), every
block shape (N = 64, 128, 256 and several blocks), cube, shared image and an
empty channel.  The bound is the form's gradient bound."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [
    # N, visibilities per channel, shared image, adjoint stages
    (64, [1], False, 2), (64, [31, 0, 33], False, 3), (64, [4900], True, 2), (128, [32, 65], True, 3),
    (128, [5000], False, 2), (256, [17], False, 3), (256, [16, 0, 47], False, 2), (256, [1, 300], True, 3),
    (512, [33], False, 2), (512, [15], False, 3), (768, [70], False, 2),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}-{sum(c[1])}-{'shared' if c[2] else 'cube'}-{c[3]}")
def test_adjoint_at_stage_edges(oracle_mod, case):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    N, z, shared, stages = case
    ds = S.random_problem(N, 0, 700 + N + sum(z), C=len(z), shared_image=shared, z_list=z, lam=1.0)
    y = S.random_complex(ds.Z, 5)
    ctx = ms.Context(ds, precision="fp16x3")
    kern, cols, fs, _ = ctx.tiling()
    ctx.set_tiling(kern, cols, fs, stages)
    G = ctx.adjoint(torch.from_numpy(np.stack([y.real, y.imag], 1).astype(np.float32)).cuda()).cpu().numpy()
    P = oracle_mod.Problem.from_dataset(ds)
    ref = np.zeros((P.n_images, N, N))
    for c in range(P.C):
        s = P.sl(c)
        if s.stop > s.start:
            ref[0 if shared else c] += P.pb[c] * oracle_mod.adjoint(
                N, P.dx, P.dy, P.u[s], P.v[s], y[s].astype(np.complex64).astype(np.complex128))
    assert np.linalg.norm(G - ref) <= 1e-4 * np.linalg.norm(ref)
    ctx.close()


@pytest.mark.parametrize("N,stages", [(64, 2), (128, 3), (256, 2), (256, 3)])
def test_drain_inside_a_unit(N, stages):
    """More than 8,192 visibilities per unit: the second drain adds to the
    first.  A short list of visibilities repeated makes an exact reference:
    the adjoint of the repeated data is the multiple of the short one's.  Both
    accumulate at most 8,192 visibilities with at most 2.5e-5 of truncation."""
    import dataclasses

    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    torch_sms = torch.cuda.get_device_properties(0).multi_processor_count
    base = S.random_problem(N, 12000, 33, lam=1.0)
    reps = -(-torch_sms * 9000 // base.Z)
    big = dataclasses.replace(base, u=np.tile(base.u, reps), v=np.tile(base.v, reps), vo=np.tile(base.vo, reps),
                              sigma=np.tile(base.sigma, reps), offsets=np.array([0, base.Z * reps], dtype=np.int64))
    y = S.random_complex(base.Z, 6)
    yt = torch.from_numpy(np.stack([y.real, y.imag], 1).astype(np.float32)).cuda()
    out = []
    for ds, yy in ((base, yt), (big, yt.repeat(reps, 1))):
        ctx = ms.Context(ds, precision="fp16x3")
        kern, cols, fs, _ = ctx.tiling()
        ctx.set_tiling(kern, cols, fs, stages)
        out.append(ctx.adjoint(yy).double())
        ctx.close()
    assert torch.linalg.norm(out[1] - reps * out[0]) <= 1e-4 * torch.linalg.norm(reps * out[0])
