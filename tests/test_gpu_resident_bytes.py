"""What a context keeps per visibility: 68 bytes of data, and under two of tile lists,
partials and units.  u and v are not among them."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu


def test_bytes_per_visibility(oracle_mod, monkeypatch):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = S.random_problem(64, 400000, 31, lam=1.0)
    # beside the visibilities: FP32 form, 64 x 64, at most 64 shares of an FP64 image
    monkeypatch.setenv("MEMSYNTH_MAX_BYTES", str(70 * ds.Z + 64 * 64 * 64 * 8 + 2 ** 20))
    ctx = ms.Context(ds, precision="fp32_direct")
    got = ctx.forward(torch.from_numpy(ds.truth).cuda())[:500].cpu().numpy()
    ctx.close()
    ref = oracle_mod.forward(64, ds.dx, ds.dy, ds.u[:500], ds.v[:500],
                             ds.pb[0].astype(np.float64) * ds.truth[0].astype(np.float64), "direct")
    assert np.max(np.abs(got[:, 0] + 1j * got[:, 1] - ref)) <= 1e-5 * np.max(np.abs(ref))
