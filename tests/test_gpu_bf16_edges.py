"""The BF16X3 operator pair at the edges of its tiles (64 visibilities in the
forward, 32 in the adjoint) against the oracle: one visibility, ragged last
tiles, several channels with an empty one, every resident and streaming tiling.
A two-part BF16 value is within 2^-16 of itself, in the table and in the operand,
so a sum of N^2 products is within 2 x 2^-16 of the sum of their magnitudes."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [
    # N, visibilities per channel, shared image, tiling (None: default)
    (64, [1], False, None), (64, [63, 0, 65], True, None), (64, [128], False, ("resident", 64, 4, 2)),
    (128, [64, 1], False, None), (128, [20001], False, None), (128, [193], False, ("resident", 128, 5, 3)),
    (128, [300], False, ("resident", 128, 4, 2)), (128, [130], False, ("stream", 64, 3, 2)),
    (256, [65, 0, 127], False, ("resident", 256, 4, 3)), (256, [20001], False, ("resident", 256, 6, 2)),
    (256, [1, 200], True, None), (256, [129], False, ("stream", 128, 4, 2)), (512, [127], False, None),
    (512, [65], False, ("stream", 32, 3, 3)), (768, [70], False, None),
    (64, [700001], False, None),  # over 4,096 visibilities a block: the adjoint's accumulator is drained within a unit
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}-{sum(c[1])}-{c[3][0] + str(c[3][2]) if c[3] else 'default'}")
def test_pair_at_tile_edges(oracle_mod, case):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    N, z, shared, tiling = case
    ds = S.random_problem(N, 0, 400 + N + sum(z), C=len(z), z_list=z, shared_image=shared, lam=1.0)
    P = oracle_mod.Problem.from_dataset(ds)
    ctx = ms.Context(ds, precision="bf16x3")
    if tiling is not None:
        ctx.set_tiling(*tiling)
    image = np.maximum(ds.truth, ds.G).astype(np.float32).reshape(P.n_images, N, N)
    V = ctx.forward(torch.from_numpy(image).cuda().reshape(ctx.image_shape())).double().cpu().numpy()
    ref = oracle_mod.model_vis(P, image.astype(np.float64))
    y = S.random_complex(ds.Z, 5).astype(np.complex64)
    G = ctx.adjoint(torch.from_numpy(np.stack([y.real, y.imag], 1)).cuda()).double().cpu().numpy()
    back, size = np.zeros((P.n_images, N, N)), np.zeros((P.n_images, N, N))
    for c in range(P.C):
        s = P.sl(c)
        if s.stop == s.start:
            continue
        i = 0 if shared else c
        got = V[s, 0] + 1j * V[s, 1]
        assert np.max(np.abs(got - ref[c])) <= 2.0 ** -15 * np.sum(np.abs(P.pb[c] * image[i]))
        back[i] += P.pb[c] * oracle_mod.adjoint(N, P.dx, P.dy, P.u[s], P.v[s], y[s].astype(np.complex128))
        size[i] += np.abs(P.pb[c]) * np.sum(np.abs(y[s].real) + np.abs(y[s].imag))
    assert np.all(np.abs(G.reshape(back.shape) - back) <= 2.0 ** -15 * size + 1e-30)
    ctx.close()
