"""The objective's scalar reduction on both sides of the line between one block
and several per image (4,096 partials, four per tile of 128 visibilities), for
one image, a cube and a shared image, and a solve of more images than the
controller's block has threads (257: one thread takes two)."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [
    # visibilities per channel, shared image
    ([131072], False), ([131073], False), ([140000, 0, 5], False), ([70000, 70000], True), ([100], True),
    ([1, 2, 3, 4, 5], False),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{sum(c[0])}-{'shared' if c[1] else 'cube'}")
def test_objective_scalars(oracle_mod, case):
    """FP64 sums of FP64 terms: 1e-11 leaves room for the order of the sums."""
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    z, shared = case
    ds = S.random_problem(16, 0, 40 + len(z), C=len(z), shared_image=shared, z_list=z, lam=1.0)
    P = oracle_mod.Problem.from_dataset(ds)
    ctx = ms.Context(ds, precision="fp64_direct")
    image = np.random.default_rng(2).uniform(1.0, 40.0, ctx.image_shape()).astype(np.float32) * np.float32(ds.G)
    want = oracle_mod.objective(P, image.reshape(P.n_images, 16, 16).astype(np.float64))
    for _ in range(2):  # the completion counter is ready for a second pass
        got = ctx.objective_grad(torch.from_numpy(image).cuda())[:3]
        for a, b in zip(got, want):
            assert abs(a - b) <= 1e-11 * max(abs(b), abs(want[1]))
    ctx.close()


def test_solve_of_many_images():
    """Images of a cube are independent: image c of 257 ends where it ends alone.
    The FP64 sums of the two runs are cut differently (shares of the adjoint),
    so the images agree to FP32 rounding of the result and of the gradient."""
    import dataclasses

    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    C, N = 257, 16
    ds = S.random_problem(N, 0, 77, C=C, z_list=[20 + c % 7 for c in range(C)], lam=1.0)
    ctx = ms.Context(ds, precision="fp64_direct")
    image = torch.full(ctx.image_shape(), float(ds.G), dtype=torch.float32, device="cuda")
    x, _, _ = ctx.solve(image.clone(), 2)
    ctx.close()
    for c in (0, 1, 255, 256):
        a, b = int(ds.offsets[c]), int(ds.offsets[c + 1])
        one = dataclasses.replace(ds, u=ds.u[a:b], v=ds.v[a:b], vo=ds.vo[a:b], sigma=ds.sigma[a:b], pb=ds.pb[c:c + 1],
                                  offsets=np.array([0, b - a], dtype=np.int64))
        ctx = ms.Context(one, precision="fp64_direct")
        y, _, _ = ctx.solve(torch.full(ctx.image_shape(), float(ds.G), dtype=torch.float32, device="cuda"), 2)
        ctx.close()
        got = x.reshape(C, N, N)[c].double()
        assert torch.linalg.norm(got - y.double().reshape(N, N)) <= 1e-6 * torch.linalg.norm(got)
