"""The hops that forward and backward of M_eo share (``wilson_eo_grad_*``).

The same kernels run on the same fields as in the separate entry points, so results
are bitwise those of ``apply``, ``link_grad`` and ``apply(dag=True)``; lattices are
ragged against the 16-, 32- and 128-site blocks of the kernels involved.
"""

import ctypes

import numpy as np
import pytest

import gen
from gpu_util import to_device, to_planar


@pytest.fixture(scope="module")
def weo():
    import paper_2303_08609_gb300 as weo

    weo.library()
    return weo


def test_null_arguments_are_refused(weo):
    lib = weo.library()
    n = ctypes.c_void_p(None)
    assert lib.wilson_eo_grad_forward(n, n, n, n, n) < 0
    assert lib.wilson_eo_grad_backward(n, n, n, n, n, n, n) < 0


@pytest.mark.gpu
@pytest.mark.parametrize("prec,fmt", [("f64", 18), ("f64", 12), ("f32", 18), ("f32", 12)])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 10, 2, 4), (4, 2, 6, 10)])
def test_shared_hops_match_separate_calls(weo, dims, prec, fmt):
    import torch

    U = to_device(gen.gauge_field(dims, "haar", seed=311))
    phi, g = (to_device(to_planar(gen.gaussian_spinor(dims, seed=s)[0]), prec) for s in (312, 313))
    op = weo.WilsonEO(dims, 0.13, U, prec=prec, linkfmt=fmt)
    out, t, dphi = torch.empty_like(phi), torch.empty_like(phi), torch.empty_like(phi)
    dU = torch.empty((4, int(np.prod(dims)), 3, 3), dtype=phi.dtype, device="cuda")
    weo.wilson_eo_grad_forward(op.handle, out, t, phi)
    weo.wilson_eo_grad_backward(op.handle, dphi, dU, g, phi, t)
    dU_only = torch.empty_like(dU)
    weo.wilson_eo_grad_backward(op.handle, None, dU_only, g, phi, t)
    assert torch.equal(out, op.apply(phi))
    assert torch.equal(dphi, op.apply(g, dag=True))
    assert torch.equal(dU, op.link_grad(g, phi)) and torch.equal(dU, dU_only)
    # host arrays and aliased ones are refused
    host = np.empty(1, dtype=np.complex128)
    lib = weo.library()
    ptr = ctypes.c_void_p
    assert lib.wilson_eo_grad_forward(op.handle, ptr(out.data_ptr()), ptr(host.ctypes.data), ptr(phi.data_ptr()), ptr(None)) < 0
    assert lib.wilson_eo_grad_forward(op.handle, ptr(out.data_ptr()), ptr(out.data_ptr()), ptr(phi.data_ptr()), ptr(None)) < 0
    op.close()
