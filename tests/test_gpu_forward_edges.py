"""The folded (FP16X3) forward at the edges of its tiles (128 visibilities, column
blocks and row segments of the folded image) against the oracle: ragged last
tiles, several channels with an empty one, every operand residency, column
blocks that are not a power of two, and a size with three row segments.  The
bound is the form's visibility bound."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [
    # N, visibilities per channel, tiling (None: default)
    (64, [1], None), (64, [127, 0, 129], None), (128, [128, 255], None), (128, [20001], None),
    (64, [300], ("stream", 32, 3, 3)), (128, [300], ("stream", 128, 4, 3)),
    (256, [1, 127], None), (256, [257], ("stream", 32, 4, 3)), (256, [385, 0, 64], ("resident", 256, 5, 2)),
    (256, [20001], ("resident", 256, 4, 3)), (512, [129], None), (512, [130], ("stream", 64, 3, 3)),
    (768, [131], None), (768, [100], ("stream", 96, 4, 3)), (768, [64], ("stream", 192, 3, 3)),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}-{sum(c[1])}-{c[2][0] + str(c[2][1]) if c[2] else 'default'}")
def test_forward_at_tile_edges(oracle_mod, case):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    N, z, tiling = case
    ds = S.random_problem(N, 0, 900 + N + sum(z), C=len(z), z_list=z, lam=1.0)
    ctx = ms.Context(ds, precision="fp16x3")
    if tiling is not None:
        ctx.set_tiling(*tiling)
    V = ctx.forward(torch.from_numpy(ds.truth).cuda()).cpu().numpy().astype(np.float64)
    ref = np.concatenate(oracle_mod.model_vis(oracle_mod.Problem.from_dataset(ds), ds.truth.astype(np.float64)))
    assert np.max(np.abs(V[:, 0] + 1j * V[:, 1] - ref)) <= 1e-5 * np.max(np.abs(ref))
    ctx.close()
