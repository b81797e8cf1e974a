"""Tilings saved by earlier versions (MEMSYNTH_TUNE_CACHE): BF16X3 entries apply with
and without the suffix that marks the folded FP16X3 kernels, FP16X3 entries only with
it, and what mem_autotune saves is read back."""
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,prec,suffix,applies", [("bf16x3", 2, "", True), ("bf16x3", 2, "|folded", True),
                                                      ("fp16x3", 3, "", False), ("fp16x3", 3, "|folded", True)])
def test_saved_entries(tmp_path, monkeypatch, form, prec, suffix, applies):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = S.random_problem(256, 700, 59, lam=1.0)
    name = torch.cuda.get_device_name().replace(" ", "_")
    cache = tmp_path / "tune.txt"
    cache.write_text(f"{name}|N=256|z=9|C=1|prec={prec}{suffix} 0 128 3 2\n")
    monkeypatch.setenv("MEMSYNTH_TUNE_CACHE", str(cache))
    ctx = ms.Context(ds, precision=form)
    assert (ctx.tiling() == ("stream", 128, 3, 2)) == applies
    img = torch.from_numpy(ds.truth).cuda()
    chosen = ctx.autotune(img, 1)
    ctx.close()
    ctx = ms.Context(ds, precision=form)
    assert ctx.tiling() == chosen
    ctx.close()
