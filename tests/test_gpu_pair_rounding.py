"""FP64 hops: the lower spin rows, differences of the forward and the backward hop,
are rounded on their own. With P = 2^53 - 1 and Q = 2 the sum of the upper rows has
to round (2^53 + 1) and the difference does not (2^53 - 3): a difference derived from
the rounded sum is off by one. Unit links, so every other operation is exact."""

import numpy as np
import pytest

from gpu_util import to_device
from lattice_ref import GAMMA, parity_sites, shift_index


@pytest.mark.gpu
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 16)])  # 16-site and 32-site CTAs
@pytest.mark.parametrize("mu", range(4))
@pytest.mark.parametrize("dag", [False, True])
def test_difference_is_not_taken_from_the_sum(dims, mu, dag):
    import paper_2303_08609_gb300 as weo

    V = int(np.prod(dims))
    here, there = parity_sites(dims, 1), parity_sites(dims, 0)
    k = len(here) // 2  # an odd site, and the compact indices of its two neighbours
    fwd, bwd = (int(np.searchsorted(there, shift_index(dims, mu, s)[here[k]])) for s in (1, -1))
    P, Q = 2 ** 53 - 1, 2
    psi = np.zeros((4, 3, V // 2), dtype=np.complex128)
    psi[0, 0, fwd], psi[0, 0, bwd] = P, Q
    with weo.WilsonEO(dims, 0.13, to_device(np.broadcast_to(np.eye(3, dtype=complex), (4, V, 3, 3))), prec="f64") as op:
        got = op.hop(to_device(psi), 1, dag=dag).cpu().numpy()[:, 0, k]
    s = -1 if dag else 1
    for row in range(4):
        g = GAMMA[mu][row, 0] * s
        f, b = (row == 0) - g, (row == 0) + g
        want = complex(float(int(f.real) * P + int(b.real) * Q), float(int(f.imag) * P + int(b.imag) * Q))
        assert got[row] == want, (row, got[row], want)
