"""The FP16X3 adjoint's beam factor is applied in FP64: a beam in FP32's subnormal
range (the far wing of a Gaussian) scales the result of a beam of one, to the rounding
of the two FP32 results."""
import dataclasses

import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [64, 128, 256])
@pytest.mark.parametrize("beam", [3 * 2.0 ** -149, 2.0 ** -140, 0.75])
def test_beam_factor(N, beam):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    base = S.random_problem(N, 3, 19, lam=1.0)
    y = torch.full((3, 2), 1e30, dtype=torch.float32, device="cuda")
    out = []
    for b in (1.0, beam):
        ctx = ms.Context(dataclasses.replace(base, pb=np.full((1, N, N), b, dtype=np.float32)), precision="fp16x3")
        out.append(ctx.adjoint(y).cpu().numpy().astype(np.float64))
        ctx.close()
    want = out[0] * float(np.float32(beam))
    assert np.all(np.abs(out[1] - want) <= 2.0 ** -23 * np.abs(want))
