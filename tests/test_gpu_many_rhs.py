"""More right-hand sides in one call than a grid has rows (65535): 2^4, 65541 of them,
of which the first, the last and those around the limit are compared with single calls."""

import pytest

import gen
from gpu_util import to_device


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["ff64", "f64", "f32", "f16"])
def test_right_hand_sides_beyond_a_grid_dimension(prec):
    import torch

    import paper_2303_08609_gb300 as weo

    dims, n = (2, 2, 2, 2), 65541
    wide = prec in ("ff64", "f64")
    g = torch.Generator(device="cuda").manual_seed(701)
    x = torch.randn(n, 4, 3, 8, dtype=torch.complex128 if wide else torch.complex64, device="cuda", generator=g)
    with weo.WilsonEO(dims, 0.13, to_device(gen.gauge_field(dims, "haar", seed=702)),
                      prec="f64" if wide else prec) as op:
        apply = op.apply_ff64 if prec == "ff64" else op.apply
        y = apply(x)
        for r in (0, 1, 65534, 65535, 65536, n - 1):
            assert torch.equal(y[r], apply(x[r].contiguous())), r
