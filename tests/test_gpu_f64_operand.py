"""The FP64 form's operand preparation on both sides of its block size (512 x 512) and
at sizes with a ragged last block: objective, entropy and gradient against the
oracle, one image, a cube and a shared image."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,shared", [(16, 1, False), (48, 3, False), (176, 2, True), (512, 1, False), (528, 1, False)])
def test_objective(oracle_mod, N, C, shared):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = S.random_problem(N, 0, 73, C=C, z_list=[9 + c for c in range(C)], shared_image=shared, lam=1.0)
    P = oracle_mod.Problem.from_dataset(ds)
    phi, chi2, ent, grad = oracle_mod.objective_grad(P, ds.truth.astype(np.float64))
    ctx = ms.Context(ds, precision="fp64_direct")
    got = ctx.objective_grad(torch.from_numpy(ds.truth).cuda())
    ctx.close()
    for a, b in zip(got[:3], (phi, chi2, ent)):
        assert abs(a - b) <= 1e-11 * abs(b)
    assert np.linalg.norm(got[3].cpu().numpy() - grad) <= 2e-7 * np.linalg.norm(grad)
