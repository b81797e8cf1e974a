"""FP16X3 on images in small units (fluxes in W/m^2/Hz: 1 mJy is 1e-29): the operand
scale follows the data down to 2^-113, so that visibilities and residual maps keep
the form's bounds relative to the oracle on the same numbers."""
import dataclasses

import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,tiling", [(64, None), (128, ("stream", 64, 4, 3)), (256, None),
                                      (256, ("resident", 256, 4, 2))],
                         ids=["64", "128-stream", "256", "256-resident"])
@pytest.mark.parametrize("unit", [1.0, 1e-30, 1e-32, 1e-33])
def test_images_in_small_units(oracle_mod, N, tiling, unit):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = S.random_problem(N, 500, 17, lam=1.0)
    img = (ds.truth / ds.truth.max() * np.float32(unit)).astype(np.float32)
    ds = dataclasses.replace(ds, truth=img, vo=ds.vo * unit, G=float(img.min()) * 0.5)
    P = oracle_mod.Problem.from_dataset(ds)
    ref = np.concatenate(oracle_mod.model_vis(P, img.astype(np.float64)))
    ctx = ms.Context(ds, precision="fp16x3")
    if tiling is not None:
        ctx.set_tiling(*tiling)
    V = ctx.forward(torch.from_numpy(img).cuda()).cpu().numpy().astype(np.float64)
    assert np.max(np.abs(V[:, 0] + 1j * V[:, 1] - ref)) <= 1e-5 * np.max(np.abs(ref))
    got = ctx.residual_image(img).cpu().numpy().astype(np.float64)
    want = oracle_mod.dirty_image(P, vis=P.vo - ref)
    assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)
    ctx.close()
