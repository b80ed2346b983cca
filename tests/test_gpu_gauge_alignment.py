"""Device gauge fields that start anywhere: on 16 bytes (vector loads in the packing
kernel), on their reals' size (scalar loads), and between (a copy first). The packed
links, and so the results, do not depend on it."""

import ctypes

import numpy as np
import pytest

import gen
from gpu_util import to_device, to_planar


@pytest.mark.gpu
@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("offset", [0, 2, 4, 8])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 14)])  # below and above one 128-site block
def test_field_at_an_offset(dims, offset, f64):
    import torch

    import paper_2303_08609_gb300 as weo

    U = gen.gauge_field(dims, "haar", seed=601).astype(np.complex128 if f64 else np.complex64)
    x = to_device(to_planar(gen.gaussian_spinor(dims, seed=602)[0]), "f32")
    raw = torch.zeros(U.nbytes + 16, dtype=torch.uint8, device="cuda")
    raw[offset:offset + U.nbytes] = torch.from_numpy(U.reshape(-1).view(np.uint8)).cuda()
    with weo.WilsonEO(dims, 0.13, to_device(U)) as op, weo.WilsonEO(dims, 0.13, to_device(np.ones_like(U))) as moved:
        p = ctypes.c_void_p
        assert weo.library().wilson_eo_set_gauge(moved.handle, p(raw.data_ptr() + offset), int(f64), p(None)) == 0
        assert torch.equal(moved.apply(x), op.apply(x))
        # the handle's own copy, which later packs read
        assert torch.equal(moved.apply_ff64(x.to(torch.complex128)), op.apply_ff64(x.to(torch.complex128)))
