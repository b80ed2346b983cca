"""meo() where no link gradient can follow: 16-bit handles, which compute the forward
pass and the source's gradient, and evaluations under no_grad, which keep nothing."""

import pytest

import gen
from gpu_util import to_device, to_planar

DIMS = (8, 8, 8, 8)


def setup(prec):
    import torch

    import paper_2303_08609_gb300 as weo

    U = to_device(gen.gauge_field(DIMS, "smooth", seed=801, eps=0.3)).to(torch.complex64).requires_grad_()
    phi = to_device(to_planar(gen.gaussian_spinor(DIMS, seed=802)[0]), "f32").requires_grad_()
    return U, phi, weo.WilsonEO(DIMS, 0.13, U.detach(), prec=prec)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f16", "bf16"])
def test_16_bit_handle_with_links_that_require_a_gradient(prec):
    import torch

    import paper_2303_08609_gb300 as weo
    from paper_2303_08609_gb300.autograd import MeoFunction, meo

    U, phi, op = setup(prec)
    want = op.apply(phi.detach())
    for y in (meo(phi, U, op), MeoFunction.apply(phi, U, op), MeoFunction.apply(phi, U, op, False)):
        assert torch.equal(y, want)
    with torch.no_grad():
        assert torch.equal(meo(phi, U, op), want)
    with pytest.raises(weo.WilsonEOError):  # there is no link gradient in 16 bits
        meo(phi, U, op).abs().sum().backward()
    g = torch.ones_like(want)
    (grad,) = torch.autograd.grad(meo(phi, U.detach(), op), phi, g)
    assert torch.equal(grad, op.apply(g, dag=True))
    op.close()


@pytest.mark.gpu
def test_no_grad_keeps_no_intermediate():
    import torch

    from paper_2303_08609_gb300.autograd import MeoFunction, meo

    U, phi, op = setup("f32")
    want = op.apply(phi.detach())
    with torch.no_grad():
        torch.cuda.synchronize()
        torch.cuda.reset_peak_memory_stats()
        before = torch.cuda.memory_allocated()
        y = meo(phi, U, op, False)
        assert torch.cuda.max_memory_allocated() - before == y.numel() * y.element_size()
    assert torch.equal(y, want)
    # the three- and four-argument forms still differentiate
    for extra in ((), (None,)):
        gp, gu = torch.autograd.grad(MeoFunction.apply(phi, U, op, *extra).abs().sum(), (phi, U))
        assert gp.shape == phi.shape and gu.shape == U.shape
    op.close()
