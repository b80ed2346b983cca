"""Arguments that the two halves of the differentiable M_eo refuse: outputs that
overlap an input or one another, wholly or in part, and host arrays."""

import ctypes

import pytest

import gen
from gpu_util import to_device


@pytest.mark.gpu
def test_overlapping_and_host_arrays_are_refused():
    import torch

    import paper_2303_08609_gb300 as weo

    dims, lib = (4, 4, 4, 4), weo.library()
    sb = 12 * 128 * 8
    gb = 4 * 256 * 9 * 8
    mem = torch.zeros(4 * sb + gb, dtype=torch.uint8, device="cuda")
    base = mem.data_ptr()
    a, b, c, d, g = (base + k * sb for k in range(5))  # four spinors and a gauge field
    host = torch.zeros(gb, dtype=torch.uint8).data_ptr()
    with weo.WilsonEO(dims, 0.13, to_device(gen.gauge_field(dims, "haar", seed=901)), prec="f32") as op:
        def forward(*p):
            return lib.wilson_eo_grad_forward(op.handle, *map(ctypes.c_void_p, p), ctypes.c_void_p(None))

        def backward(*p):
            return lib.wilson_eo_grad_backward(op.handle, *map(ctypes.c_void_p, p), ctypes.c_void_p(None))

        # out, t, in
        assert forward(a, b, c) == 0
        for bad in ((a, b, a), (a, b, b), (a, a, c), (a, b, b + 16), (a, a + sb - 16, c), (host, b, c), (a, host, c),
                    (a, b, host)):
            assert forward(*bad) == -1, bad
        # grad_phi, grad_gauge, g, phi, t
        assert backward(a, g, b, c, d) == 0
        assert backward(None, g, b, c, d) == 0
        for bad in ((b, g, b, c, d), (c, g, b, c, d), (d, g, b, c, d), (a, b, b, c, d), (a, c, b, c, d), (None, d, b, c, d),
                    (a, a, b, c, d), (g, g, b, c, d), (g + gb - sb, g, b, c, d), (a, d + 16, b, c, d), (b + 16, g, b, c, d),
                    (a, g, g + gb - 16, c, d), (host, g, b, c, d), (a, host, b, c, d), (a, g, host, c, d)):
            assert backward(*bad) == -1, bad
    torch.cuda.synchronize()
