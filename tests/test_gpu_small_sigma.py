"""FP16X3 with the resident operand (the default for N <= 128) finishes each
visibility in FP64: weights above FP32's range and squares of residuals below it.
A data set in units of 2^-80 (8e-25; sigma 4e-26, weights 6e50) against the oracle,
and a short solve against the same data in units of one, which differ by powers
of two only."""
import dataclasses

import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -80


def _in_units(ds, unit):
    return dataclasses.replace(ds, truth=(ds.truth * np.float32(unit)).astype(np.float32), vo=ds.vo * unit,
                               sigma=ds.sigma * unit, G=ds.G * unit, lam=ds.lam / unit)


@pytest.mark.parametrize("N,tiling", [(64, None), (128, None), (256, ("resident", 256, 4, 2))],
                         ids=["64", "128", "256-resident"])
def test_objective_with_weights_beyond_fp32(oracle_mod, N, tiling):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = _in_units(S.random_problem(N, 700, 23, lam=1.0), UNIT)
    P = oracle_mod.Problem.from_dataset(ds)
    phi, chi2, ent, grad = oracle_mod.objective_grad(P, ds.truth.astype(np.float64))
    ctx = ms.Context(ds, precision="fp16x3")
    if tiling is not None:
        ctx.set_tiling(*tiling)
    got = ctx.objective_grad(torch.from_numpy(ds.truth).cuda())
    ctx.close()
    # the form's objective, entropy and gradient bounds
    assert abs(got[1] - chi2) <= 3e-6 * chi2
    assert abs(got[0] - phi) <= 3e-6 * abs(phi)
    assert abs(got[2] - ent) <= 1e-12 * abs(ent)
    g = got[3].cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - grad) <= 1e-4 * np.linalg.norm(grad)


@pytest.mark.parametrize("N", [64, 128])
def test_solve_in_small_units(N):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    base = S.random_problem(N, 700, 29, lam=1.0)
    out = []
    for unit in (1.0, UNIT):
        ds = _in_units(base, unit)
        ctx = ms.Context(ds, precision="fp16x3")
        img, rep, _ = ctx.solve(torch.full(ctx.image_shape(), ds.G, dtype=torch.float32, device="cuda"), 4)
        ctx.close()
        out.append((img.cpu().numpy().astype(np.float64) / unit, rep.phi))
    # the same sums scaled: what rounding remains is FP32's subnormal low words
    assert abs(out[0][1] - out[1][1]) <= 1e-9 * abs(out[0][1])
    assert np.linalg.norm(out[0][0] - out[1][0]) <= 1e-6 * np.linalg.norm(out[0][0])
