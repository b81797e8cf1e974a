"""The BF16X3 gradient reduction on both sides of its rule (one or four groups of
threads per element, by the units of an output block and the pixels): the gradient and
the adjoint against the oracle at the form's bound."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [
    # N, visibilities per channel: units per block on a 152-SM GPU
    (64, [3000]), (64, [1000] * 4), (64, [500] * 20), (128, [3000]), (128, [1200] * 4), (128, [700] * 9),
    (256, [300]), (256, [3000]), (256, [1300] * 3), (256, [900] * 4), (512, [700]), (512, [3000]), (768, [200]),
]


@pytest.mark.parametrize("N,z", CASES, ids=lambda v: str(v) if isinstance(v, int) else f"{len(v)}x{v[0]}")
def test_gradient(oracle_mod, N, z):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = S.random_problem(N, 0, 79 + N, C=len(z), z_list=z, lam=1.0)
    P = oracle_mod.Problem.from_dataset(ds)
    ctx = ms.Context(ds, precision="bf16x3")
    img = torch.from_numpy(ds.truth).cuda()
    phi, chi2, ent, grad = oracle_mod.objective_grad(P, ds.truth.astype(np.float64))
    got = ctx.objective_grad(img)
    assert abs(got[1] - chi2) <= 1e-5 * chi2
    g = got[3].cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - grad) <= 1e-4 * np.linalg.norm(grad)
    # the adjoint's assembly takes the same kernel, without the scalars
    y = S.random_complex(ds.Z, 9).astype(np.complex64)
    back = ctx.adjoint(torch.from_numpy(np.stack([y.real, y.imag], 1)).cuda()).cpu().numpy().astype(np.float64)
    c = len(z) - 1
    s = P.sl(c)
    ref = P.pb[c] * oracle_mod.adjoint(N, P.dx, P.dy, P.u[s], P.v[s], y[s].astype(np.complex128))
    assert np.linalg.norm(back[c] - ref) <= 1e-4 * np.linalg.norm(ref)
    ctx.close()
