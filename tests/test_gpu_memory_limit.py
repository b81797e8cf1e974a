"""Contexts at a device memory limit (MEMSYNTH_MAX_BYTES, a failure made on the host):
what fits is taken, what does not is refused, and a refused call leaves the context
usable."""
import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ms():
    from paper_1703_02920_gb300 import memsynth
    memsynth.load()
    return memsynth


def _least(ms, monkeypatch, ds, form):
    """The smallest limit (to 256 bytes) that lets a context be created."""
    lo, hi = 0, 1 << 28
    while hi - lo > 256:
        mid = (lo + hi) // 2
        monkeypatch.setenv("MEMSYNTH_MAX_BYTES", str(mid))
        try:
            ms.Context(ds, precision=form).close()
            hi = mid
        except ms.MemError as e:
            assert e.status == 2
            lo = mid
    return hi


@pytest.mark.parametrize("N", [64, 80])
def test_fp64_form_shares_its_work_by_what_fits(ms, monkeypatch, N):
    """The FP64 form needs no more than the FP32 form, whose shares are fewer, and its
    own FP64 operand and residual; with fewer shares its sums are the same to the
    order of FP64 additions."""
    import torch
    ds = S.random_problem(N, 900, 37, lam=1.0)
    img = torch.from_numpy(ds.truth).cuda()
    monkeypatch.delenv("MEMSYNTH_MAX_BYTES", raising=False)
    ctx = ms.Context(ds, precision="fp64_direct")
    want = ctx.objective_grad(img)
    ctx.close()
    limit = _least(ms, monkeypatch, ds, "fp32_direct") + 16 * ds.Z + 8 * N * (N + 16) + 4096
    for cap in (limit, _least(ms, monkeypatch, ds, "fp64_direct")):
        monkeypatch.setenv("MEMSYNTH_MAX_BYTES", str(cap))
        ctx = ms.Context(ds, precision="fp64_direct")
        for _ in range(3):
            got = ctx.objective_grad(img)
            for a, b in zip(got[:3], want[:3]):
                assert abs(a - b) <= 1e-11 * abs(b)
            assert torch.linalg.norm(got[3] - want[3]) <= 2e-7 * torch.linalg.norm(want[3])
        ctx.close()


def test_other_forms_keep_their_shares_after_a_limited_fp64(ms, monkeypatch):
    """An FP64 context with few shares switched to the FP32 form: either its own shares
    fit, or it is refused; never the FP64 form's smaller block."""
    import torch
    ds = S.random_problem(64, 900, 41, lam=1.0)
    img = torch.from_numpy(ds.truth).cuda()
    monkeypatch.delenv("MEMSYNTH_MAX_BYTES", raising=False)
    ctx = ms.Context(ds, precision="fp32_direct")
    want = ctx.objective_grad(img)
    ctx.close()
    least = _least(ms, monkeypatch, ds, "fp64_direct")
    for cap in (least, least + (1 << 20), least + (3 << 20), least + (8 << 20)):
        monkeypatch.setenv("MEMSYNTH_MAX_BYTES", str(cap))
        ctx = ms.Context(ds, precision="fp64_direct")
        first = ctx.objective_grad(img)
        try:
            ctx.set_precision("fp32_direct")
        except ms.MemError as e:
            assert e.status == 2
        else:
            got = ctx.objective_grad(img)
            assert got[:3] == want[:3] and torch.equal(got[3], want[3])
        ctx.set_precision("fp64_direct")
        again = ctx.objective_grad(img)
        assert again[0] == first[0] and torch.equal(again[3], first[3])
        ctx.close()


def test_gridded_buffers_that_do_not_fit_are_given_back(ms, monkeypatch, oracle_mod):
    """Row spectra of a padding whose 2-D spectra do not fit are not kept: the next
    padding has its own."""
    import torch
    N = 64
    ds = S.random_problem(N, 100, 43, lam=1.0)
    least = _least(ms, monkeypatch, ds, "fp32_direct")
    rows = lambda pad: (pad * N // 2 + 1) * N * 8  # noqa: E731
    whole = lambda pad: (pad * N // 2 + 1) * pad * N * 8  # noqa: E731
    cap = least + rows(1) + whole(1) + 2048
    assert rows(2) < cap - least < rows(2) + whole(1)
    monkeypatch.setenv("MEMSYNTH_MAX_BYTES", str(cap))
    ctx = ms.Context(ds, precision="fp32_direct")
    img = torch.from_numpy(ds.truth).cuda()
    for _ in range(2):
        with pytest.raises(ms.MemError) as e:
            ctx.forward_gridded(img, 2)
        assert e.value.status == 2
        got = ctx.forward_gridded(img, 1).cpu().numpy().astype(np.float64)
        ref = oracle_mod.forward_gridded(N, ds.dx, ds.dy, ds.u, ds.v, ds.pb[0].astype(np.float64) * ds.truth[0], 1)
        assert np.max(np.abs(got[:, 0] + 1j * got[:, 1] - ref)) <= 2e-5 * np.max(np.abs(ref))
    ctx.close()


def test_solve_after_a_history_that_did_not_fit(ms, monkeypatch):
    import torch
    ds = S.random_problem(64, 900, 47, lam=1.0)
    start = torch.full((1, 64, 64), ds.G, dtype=torch.float32, device="cuda")
    monkeypatch.delenv("MEMSYNTH_MAX_BYTES", raising=False)
    ctx = ms.Context(ds, precision="fp16x3")
    want = ctx.solve(start, 3)
    ctx.close()
    monkeypatch.setenv("MEMSYNTH_MAX_BYTES", str(_least(ms, monkeypatch, ds, "fp16x3") + (4 << 20)))
    ctx = ms.Context(ds, precision="fp16x3")
    for _ in range(2):
        got = ctx.solve(start, 3)
        assert torch.equal(got[0], want[0]) and np.array_equal(got[2], want[2])
        with pytest.raises(ms.MemError) as e:
            ctx.solve(start, 200000)  # a history of 9.6 MB
        assert e.value.status == 2
    ctx.close()
