"""Mixed solves whose |b|^2 lies outside FP32's range, while every element is well
inside it: the norms are summed in FP64. A solve of s b takes the steps of the solve
of b when s is a power of two."""

import pytest

import gen
from gpu_util import to_device, to_planar


@pytest.mark.gpu
@pytest.mark.parametrize("prec,fmt", [("f32", 18), ("f16", 12)])
@pytest.mark.parametrize("power", [61, -50])
def test_solve_of_a_scaled_right_hand_side(prec, fmt, power):
    import torch

    import paper_2303_08609_gb300 as weo

    dims = (8, 8, 8, 8)
    b = to_device(to_planar(gen.gaussian_spinor(dims, seed=502)[0]))
    with weo.WilsonEO(dims, 0.13, to_device(gen.gauge_field(dims, "smooth", seed=501, eps=0.4)), prec=prec,
                      linkfmt=fmt) as op:
        x, info = op.solve(b, tol=1e-10)
        y, scaled = op.solve(b * 2.0 ** power, tol=1e-10)
    assert info["converged"] and scaled["converged"], scaled
    assert scaled["iterations"] == info["iterations"]
    assert torch.equal(y, x * 2.0 ** power)


@pytest.mark.gpu
def test_each_right_hand_side_has_its_own_scale():
    import torch

    import paper_2303_08609_gb300 as weo

    dims = (8, 8, 8, 8)
    b = to_device(to_planar(gen.gaussian_spinor(dims, nrhs=3, seed=503)))
    s = torch.tensor([2.0 ** 61, 1.0, 2.0 ** -50], dtype=torch.float64, device="cuda")[:, None, None, None]
    with weo.WilsonEO(dims, 0.13, to_device(gen.gauge_field(dims, "smooth", seed=501, eps=0.4)), prec="f16") as op:
        x, info = op.solve(b, tol=1e-10)
        y, scaled = op.solve(b * s, tol=1e-10)
    assert info["converged"] and scaled["converged"]
    assert torch.equal(y, x * s)
