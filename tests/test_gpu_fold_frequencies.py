"""The folded kernels (FP16X3, resident and streamed, and FP64) at the frequencies where
their closed forms and signed half phases can go wrong: zero (the table sums divide by
sin(pi b)), half a turn per pixel (the phase's sign wraps), whole turns and aliases of
small frequencies, next to them, and every pair of these as (u, v)."""
import dataclasses

import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

CASES = [("fp16x3", 64, None), ("fp16x3", 64, ("stream", 64, 4, 3)), ("fp16x3", 128, None), ("fp16x3", 256, None),
         ("fp16x3", 256, ("resident", 256, 4, 2)), ("fp64_direct", 48, None), ("fp64_direct", 64, None),
         ("fp64_direct", 128, None)]


@pytest.mark.parametrize("form,N,tiling", CASES, ids=lambda v: str(v[0]) if isinstance(v, tuple) else str(v))
def test_special_frequencies(oracle_mod, form, N, tiling):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    base = S.random_problem(N, 10, 67, lam=1.0)
    f = np.array([0.0, 1e-18, -1e-18, 1e-9, -1e-7, 0.5, -0.5, 0.5 - 1e-9, 0.25, 1.0, -1.0, 1.0 + 1.0 / 64, 2.5, -1.5,
                  1.0 / N, -2.0 / N, 0.3, 100.25])
    fu, fv = (g.ravel() for g in np.meshgrid(f, f))
    z = fu.size
    rng = np.random.default_rng(5)
    ds = dataclasses.replace(base, u=fu / base.dx, v=fv / base.dy, vo=S.random_complex(z, 3), sigma=np.ones(z),
                             offsets=np.array([0, z], dtype=np.int64))
    # the oracle at the same reduced frequencies, so that both see the same phases
    red = lambda w, d: ((w * d) - np.rint(w * d)) / d  # noqa: E731
    u, v = red(ds.u, ds.dx), red(ds.v, ds.dy)
    img = rng.uniform(0.5, 1.0, (1, N, N)).astype(np.float32)
    B = ds.pb[0].astype(np.float64) * img[0].astype(np.float64)
    ctx = ms.Context(ds, precision=form)
    if tiling is not None:
        ctx.set_tiling(*tiling)
    V = ctx.forward(torch.from_numpy(img).cuda()).cpu().numpy().astype(np.float64)
    ref = oracle_mod.forward(N, ds.dx, ds.dy, u, v, B, "direct")
    tol = 2e-7 if form == "fp64_direct" else 1e-5
    assert np.max(np.abs(V[:, 0] + 1j * V[:, 1] - ref)) <= tol * np.max(np.abs(ref))
    # beside the largest (zero frequency): every value against its own terms' size
    assert np.max(np.abs(V[0, 0] + 1j * V[0, 1] - B.sum())) <= tol * B.sum()
    y = S.random_complex(z, 7).astype(np.complex64)
    G = ctx.adjoint(torch.from_numpy(np.stack([y.real, y.imag], 1)).cuda()).cpu().numpy()[0].astype(np.float64)
    want = ds.pb[0] * oracle_mod.adjoint(N, ds.dx, ds.dy, u, v, y.astype(np.complex128))
    assert np.linalg.norm(G - want) <= (2e-7 if form == "fp64_direct" else 1e-4) * np.linalg.norm(want)
    ctx.close()
