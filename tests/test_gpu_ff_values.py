"""Conversion between complex128 and float-float spinors (``ff_split`` / ``ff_join``)
at the values where integer arithmetic on the bits can go wrong.

With kappa = 0 the float-float operator returns its input through both
conversions: 48 significant bits survive, so a value may move by 2^-48 of itself.
"""

import numpy as np
import pytest

import gen
from gpu_util import to_device


@pytest.mark.gpu
def test_values_pass_through_both_conversions():
    import torch

    import paper_2303_08609_gb300 as weo

    dims = (8, 8, 8, 8)
    n = 12 * 2048
    rng = np.random.default_rng(5)
    vals = [0.0]
    for k in (-80, -74, -73, -72, -40, -1, 0, 1, 24, 60, 100, 116, 117, 118):
        for m in (1.0, 1 + 2.0 ** -52, 1 + 2.0 ** -24, 1 + 2.0 ** -25, 1 + 3 * 2.0 ** -25, 2 - 2.0 ** -52, 2 - 2.0 ** -24,
                  2 - 2.0 ** -25, 2 - 3.4e-8, 2 - 2.0 ** -30, 1.5 + 2.0 ** -28):
            vals += [m * 2.0 ** k, -m * 2.0 ** k]
    vals = np.array(vals)
    re = np.concatenate([vals, rng.normal(size=n - len(vals)) * 2.0 ** rng.integers(-30, 30, n - len(vals))])
    x = (re + 1j * re[::-1]).reshape(4, 3, 2048)
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    with weo.WilsonEO(dims, 0.0, to_device(gen.gauge_field(dims, "haar", seed=6)), prec="f64") as op:
        y = op.apply_ff64(xd).cpu().numpy()
    for got, want in ((y.real, x.real), (y.imag, x.imag)):
        # below 2^-73 the low part runs into FP32's range: absolute there
        assert np.all(np.abs(got - want) <= 2.0 ** -48 * np.abs(want) + 2.0 ** -140)
