"""The gridded forward of samples a tiny fraction of a cell beside a grid point where
the transform is zero: the interpolated value is that fraction times the
neighbour's, to FP32 accuracy of itself."""
import dataclasses

import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,pad", [(64, 2), (64, 3), (256, 2)])
def test_small_fractions_beside_a_zero(oracle_mod, N, pad):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    base = S.random_problem(N, 400, 19)
    M = pad * N
    f = np.array([2.0 ** -20, 2.0 ** -31, 2.0 ** -34, 2.0 ** -36, 3 * 2.0 ** -42])
    zero = np.zeros_like(f)
    # two opposite pixels: no flux, so the transform is zero at the origin
    img = np.zeros((1, N, N), np.float32)
    img[0, N // 2 + 3, N // 2 - 9] = 1.0
    img[0, N // 2 - 5, N // 2 + 7] = -1.0
    pb = np.ones((1, N, N), np.float32)
    for gu, gv in ((f, zero), (zero, f)):
        ds = dataclasses.replace(base, u=gu / (M * base.dx), v=gv / (M * base.dy), vo=base.vo[:f.size],
                                 sigma=base.sigma[:f.size], pb=pb, offsets=np.array([0, f.size], dtype=np.int64))
        ctx = ms.Context(ds, precision="fp32_direct")
        got = ctx.forward_gridded(torch.from_numpy(img).cuda(), pad).double().cpu().numpy()
        ctx.close()
        ref = oracle_mod.forward_gridded(N, ds.dx, ds.dy, ds.u, ds.v, img[0].astype(np.float64), pad)
        assert np.all(np.abs(got[:, 0] + 1j * got[:, 1] - ref) <= 2e-5 * np.abs(ref))
