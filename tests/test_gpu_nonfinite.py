"""Infinities and NaN in a source reach the same sites whatever kernel runs: the split
hops, the 16-bit store that exchanges its norm between three threads, and the
float-float operator with its conversions on integer arithmetic."""

import numpy as np
import pytest

import gen
from gpu_util import to_device, to_planar

DIMS = (8, 6, 4, 10)


def source(value, nrhs):
    x = to_planar(gen.gaussian_spinor(DIMS, nrhs=nrhs, seed=1302))
    x[0, 0, 1, 17] = complex(value, 0.5)
    x[0, 3, 2, 400] = complex(-1.0, value)
    return x


@pytest.mark.gpu
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("prec,fmt", [("f32", 18), ("f32", 12), ("f16", 18), ("bf16", 12)])
def test_split_hops_as_one_site_per_thread(prec, fmt, value):
    import paper_2303_08609_gb300 as weo

    x = to_device(source(value, 2), prec)
    with weo.WilsonEO(DIMS, 0.13, to_device(gen.gauge_field(DIMS, "haar", seed=1301)), prec=prec, linkfmt=fmt) as op:
        split = op.apply(x).cpu().numpy()
        weo.wilson_eo_set_launch(op.handle, 128, 2)  # two right-hand sides per thread
        one = op.apply(x).cpu().numpy()
    assert not np.isfinite(split[0]).all() and np.isfinite(split[1]).all()
    assert np.array_equal(split.view(np.float32), one.view(np.float32), equal_nan=True)


@pytest.mark.gpu
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_float_float_as_fp64(value):
    import paper_2303_08609_gb300 as weo

    x = to_device(source(value, 1)[0])
    with weo.WilsonEO(DIMS, 0.13, to_device(gen.gauge_field(DIMS, "haar", seed=1301)), prec="f64") as op:
        want = np.isfinite(op.apply(x).cpu().numpy())
        y = op.apply_ff64(x).cpu().numpy()
    assert not want.all() and want.any()
    assert np.array_equal(np.isfinite(y), want)
