"""The folded FP64 kernels at their edges against the oracle: image sides that
are not multiples of the row and column blocks, fewer visibilities than a tile,
remainders, work split into one and several shares, cube, shared image and an
empty channel.  V and the gradient are FP32 results (half a unit in the last
place is 6e-8); phi is summed in FP64."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [
    # N, visibilities per channel, shared image
    (16, [1], False), (16, [129], False), (32, [3, 0, 260], False), (48, [127], False), (48, [128, 1], True),
    (80, [700], False), (112, [33, 95], False), (160, [513], False), (160, [20, 0, 7], True), (272, [65], False),
    (64, [40000], False),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}-{sum(c[1])}-{'shared' if c[2] else 'cube'}")
def test_f64_edges(oracle_mod, case):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    N, z, shared = case
    ds = S.random_problem(N, 0, 300 + N + sum(z), C=len(z), shared_image=shared, z_list=z, lam=1.0)
    P = oracle_mod.Problem.from_dataset(ds)
    ctx = ms.Context(ds, precision="fp64_direct")
    image = np.random.default_rng(N).uniform(1.0, 40.0, ctx.image_shape()).astype(np.float32) * np.float32(ds.G)
    x = torch.from_numpy(image).cuda()
    V = ctx.forward(x).double().cpu().numpy()
    ref_i = image.reshape(P.n_images, N, N).astype(np.float64)
    want = np.concatenate(oracle_mod.model_vis(P, ref_i))
    got = V[:, 0] + 1j * V[:, 1]
    assert np.linalg.norm(got - want) <= 2e-7 * np.linalg.norm(want)
    phi, chi2, _, grad = ctx.objective_grad(x)
    ref = oracle_mod.objective_grad(P, ref_i)
    assert abs(chi2 - ref[1]) <= 1e-11 * abs(ref[1])
    assert abs(phi - ref[0]) <= 1e-11 * max(abs(ref[0]), abs(ref[1]))
    g = grad.double().cpu().numpy().reshape(P.n_images, N, N)
    assert np.linalg.norm(g - ref[3]) <= 2e-7 * np.linalg.norm(ref[3])
    ctx.close()
