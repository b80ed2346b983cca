"""A handle's captured solver iterations after something they hold has changed: kappa,
the launch settings, link blocks given back, work vectors that another solve made
larger. Each solve equals that of a handle which never solved before, bit by bit."""

import pytest

import gen
from gpu_util import to_device, to_planar

DIMS = (8, 8, 8, 8)


@pytest.fixture(scope="module")
def data():
    U = to_device(gen.gauge_field(DIMS, "smooth", seed=1001, eps=0.4))
    return U, to_device(to_planar(gen.gaussian_spinor(DIMS, nrhs=4, seed=1002)))


def fresh(U, kappa, prec, b, mixed):
    import paper_2303_08609_gb300 as weo

    with weo.WilsonEO(DIMS, kappa, U, prec=prec) as op:
        x, info = op.solve(b, tol=1e-10, mixed=mixed)
    assert info["converged"]
    return x


@pytest.mark.gpu
@pytest.mark.parametrize("prec,mixed", [("f32", True), ("f16", True), ("f64", False)])
def test_kappa_between_solves(data, prec, mixed):
    import torch

    import paper_2303_08609_gb300 as weo

    U, b = data[0], data[1][0].contiguous()
    with weo.WilsonEO(DIMS, 0.13, U, prec=prec) as op:
        op.solve(b, tol=1e-10, mixed=mixed)
        op.set_kappa(0.12)
        x, info = op.solve(b, tol=1e-10, mixed=mixed)
    assert info["converged"]
    assert torch.equal(x, fresh(U, 0.12, prec, b, mixed))


@pytest.mark.gpu
def test_vectors_that_another_solve_made_larger(data):
    import torch

    import paper_2303_08609_gb300 as weo

    U, many = data
    one = many[0].contiguous()
    with weo.WilsonEO(DIMS, 0.13, U, prec="f32") as op:
        first = op.solve(one, tol=1e-10, mixed=False)[0]
        op.solve(many, tol=1e-10, mixed=True)
        again = op.solve(one, tol=1e-10, mixed=False)[0]
        mixed = op.solve(one, tol=1e-10, mixed=True)[0]
    assert torch.equal(first, again)
    assert torch.equal(mixed, fresh(U, 0.13, "f32", one, True))


@pytest.mark.gpu
def test_staging_turned_off_between_solves(data):
    import torch

    import paper_2303_08609_gb300 as weo

    U, b = data[0], data[1][0].contiguous()
    with weo.WilsonEO(DIMS, 0.13, U, prec="f32") as op:
        weo.wilson_eo_set_staging(op.handle, True)
        op.solve(b, tol=1e-10)
        weo.wilson_eo_set_staging(op.handle, False)
        assert torch.equal(op.solve(b, tol=1e-10)[0], fresh(U, 0.13, "f32", b, True))
