"""log(I/G) of the tensor-core forms, read off the entropy of a constant image (whose
terms are equal, so their sum has the one logarithm's error) against extended
precision: no further off than FP64's quotient and logarithm, rounded once each."""
import dataclasses

import numpy as np
import pytest

from paper_1703_02920_gb300 import synth as S

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _entropies(form, G, values):
    import torch
    from paper_1703_02920_gb300 import memsynth as ms
    ds = dataclasses.replace(S.random_problem(64, 10, 3, lam=1.0), G=G)
    ctx = ms.Context(ds, precision=form)
    out = []
    for x in values:
        img = torch.full(ctx.image_shape(), float(x), dtype=torch.float32, device="cuda")
        out.append(-ctx.objective_grad(img)[2] / 64 ** 2 / float(x))
    ctx.close()
    return np.array(out)


@pytest.mark.parametrize("form", ["fp16x3", "bf16x3"])
@pytest.mark.parametrize("G", [1e-4, 6.25e-6, 3e-31, 1e-305])
def test_logarithm_of_the_entropy(form, G):
    near = np.linspace(0.98, 1.02, 41) * G if G > 1e-40 else []
    far = np.exp(np.linspace(-13.8, 20.0, 40)) * G if G > 1e-40 else np.array([1e-38, 1e-3])
    values = np.concatenate([near, far]).astype(np.float32)
    want = np.array([np.log(np.longdouble(x) / np.longdouble(G)) for x in values])
    err = np.abs((_entropies(form, G, values).astype(np.longdouble) - want).astype(np.float64))
    # the quotient's rounding; the logarithm's, the product's with x, the sum's (four
    # at most: the terms are equal) and the two divisions' here
    assert np.all(err <= EPS + 8 * EPS * np.abs(want.astype(np.float64)))


def test_quotients_near_one():
    """G within 2 % of the pixels' value: the error is at most half a unit of the
    quotient's last place, and the roundings of the logarithm, of its product with x,
    of the sum (three: the terms are equal) and of the division here."""
    x = float(np.float32(1.2345e-4))
    for G in x * np.random.default_rng(4).uniform(0.98, 1.02, 48):
        want = float(np.log(np.longdouble(x) / np.longdouble(G)))
        got = _entropies("fp16x3", float(G), [x])[0]
        assert abs(got - want) <= np.spacing(x / G) / 2 + 6 * EPS * abs(want), (G, got, want)


def test_image_at_the_bound_has_no_entropy():
    x = np.float32(1.0 / 3)
    assert _entropies("fp16x3", float(x), [x])[0] == 0.0
