"""The gridded forward where its grid coordinates can go wrong, against the
oracle's statement of the same steps: samples on grid points, just beside them,
at the wrap of the grid (frequency just below zero, half a turn and beyond), and
the largest transform (8,192 points).  FP32 transform: 2e-5 of max |V|; a grid
coordinate within 2^-33 of a cell moves a value by as much of its neighbour's."""
import dataclasses

import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,pad", [(64, 1), (64, 3), (64, 5), (256, 2)])
def test_coordinates_at_cell_edges(oracle_mod, N, pad):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    base = S.random_problem(N, 400, 19)
    M = pad * N
    near = np.array([0.0, 1e-7, -1e-7, 0.5, 1.0, -1.0, -0.5, M / 2, M / 2 - 1e-7, -M / 2, M / 2 - 1, 1 - M / 2, 0.25, -3.0,
                     M + 1.5, -M - 0.5, 7.0 + 1e-7, 7.0 - 1e-7, M / 2 - 0.5, 0.5 - M / 2])
    gu, gv = (g.ravel() for g in np.meshgrid(near, near))
    ds = dataclasses.replace(base, u=gu / (M * base.dx), v=gv / (M * base.dy))
    ctx = ms.Context(ds, precision="fp32_direct")
    got = ctx.forward_gridded(torch.from_numpy(ds.truth).cuda(), pad).double().cpu().numpy()
    ref = oracle_mod.forward_gridded(N, ds.dx, ds.dy, ds.u, ds.v, ds.pb[0].astype(np.float64) * ds.truth[0], pad)
    assert np.max(np.abs(got[:, 0] + 1j * got[:, 1] - ref)) <= 2e-5 * np.max(np.abs(ref))
    ctx.close()


def test_largest_transform(oracle_mod):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = S.random_problem(1024, 200, 23)
    ctx = ms.Context(ds, precision="fp16x3")
    got = ctx.forward_gridded(torch.from_numpy(ds.truth).cuda(), 8).double().cpu().numpy()
    ref = oracle_mod.forward_gridded(1024, ds.dx, ds.dy, ds.u, ds.v, ds.pb[0].astype(np.float64) * ds.truth[0], 8)
    assert np.max(np.abs(got[:, 0] + 1j * got[:, 1] - ref)) <= 2e-5 * np.max(np.abs(ref))
    ctx.close()
