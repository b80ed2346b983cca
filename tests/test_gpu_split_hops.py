"""Hops with a site's directions on different warps (``csrc/weo_split.cuh``).

The index rules are checked on the CPU by a model of the kernels' arithmetic; on
the GPU M_eo and M_eo^dag are compared with the FP64 oracle where these kernels
can go wrong: V/2 below, at and above one and several 32-site (FP64: 16-site)
blocks, extents of 2, Lx/2 = 1, and both sides of the size where FP64 changes
its kernel (V/2 = 4864). The bounds are those of every parity test here.
"""

import numpy as np
import pytest

import gen
from gpu_util import TOL, from_planar, rel_l2, to_device, to_planar


def fastdiv(d):
    """(m, s) of the kernels' division by d: n // d == (n * m) >> s for n < 2^31."""
    if d < 2:
        return 1, 0
    lg = (d - 1).bit_length()
    return ((1 << (31 + lg)) + d - 1) // d, 31 + lg


def test_division_by_multiplication():
    rng = np.random.default_rng(0)
    ds = list(range(1, 300)) + [2 ** k + e for k in range(9, 31) for e in (-1, 0, 1)] + \
        [int(x) for x in rng.integers(1, 2 ** 31, 300)]
    for d in ds:
        m, s = fastdiv(d)
        assert 0 < m < 2 ** 32
        top = (2 ** 31 - 1) // d * d
        for n in {0, 1, d - 1, d, d + 1, 2 * d - 1, top - 1, top, 2 ** 31 - 1, *map(int, rng.integers(0, 2 ** 31, 8))}:
            if 0 <= n < 2 ** 31:
                assert (n * m) >> s == n // d, (n, d)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 2), (4, 2, 2, 6), (6, 4, 2, 4), (10, 6, 4, 2)])
def test_neighbour_of_each_direction(dims):
    """dir_neighbour's compact index is lex/2 of x +- mu."""
    lx, ly, lz, lt = dims
    ext = dims
    lxh = lx // 2
    step = (0, lxh, lxh * ly, lxh * ly * lz)
    for op in (0, 1):
        for i in range(lx * ly * lz * lt // 2):
            xh, y, z, t = i % lxh, i // lxh % ly, i // (lxh * ly) % lz, i // (lxh * ly * lz)
            par = (y + z + t + op) & 1
            x = [2 * xh + par, y, z, t]
            for mu in range(4):
                for fwd in (True, False):
                    if mu == 0:
                        if fwd:
                            got = (i - xh if xh + 1 == lxh else i + 1) if par else i
                        else:
                            got = i if par else (i + lxh - 1 if xh == 0 else i - 1)
                    else:
                        c, n = x[mu], ext[mu]
                        if fwd:
                            got = i - (n - 1) * step[mu] if c + 1 == n else i + step[mu]
                        else:
                            got = i + (n - 1) * step[mu] if c == 0 else i - step[mu]
                    q = list(x)
                    q[mu] = (q[mu] + (1 if fwd else -1)) % ext[mu]
                    assert got == (((q[3] * lz + q[2]) * ly + q[1]) * lx + q[0]) // 2


@pytest.mark.gpu
@pytest.mark.parametrize("prec,fmt", [("f64", 18), ("f64", 12), ("f32", 18), ("f32", 12), ("f16", 18), ("f16", 12),
                                      ("bf16", 12)])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 2, 4), (2, 8, 2, 2), (2, 6, 4, 10), (6, 10, 2, 4),
                                  (8, 6, 10, 20), (8, 4, 8, 38)])
def test_split_hops_match_oracle(weo, oracle_lib, dims, prec, fmt):
    U = gen.gauge_field(dims, "haar", seed=301)
    psi = gen.gaussian_spinor(dims, seed=302)[0]
    op = weo.WilsonEO(dims, 0.13, to_device(U), prec=prec, linkfmt=fmt)
    x = to_device(to_planar(psi), prec)
    for dag in (False, True):
        want = (oracle_lib.meo_dag if dag else oracle_lib.meo)(U, 0.13, psi, dims)
        y = op.apply(x, dag=dag)
        assert rel_l2(from_planar(y.cpu().numpy()), want) <= TOL[prec]


@pytest.mark.gpu
@pytest.mark.parametrize("prec,fmt", [("f64", 18), ("f32", 18), ("f32", 12), ("f16", 18), ("f16", 12)])
@pytest.mark.parametrize("dims", [(2, 6, 4, 10), (16, 16, 16, 32)])
def test_several_right_hand_sides_equal_single_ones(weo, dims, prec, fmt):
    """Whatever kernel the size selects (split hops, tiles with their links in shared
    memory, one site per thread), each right-hand side is bitwise the single one:
    V/2 = 65536 lies on both sides of every rule for 2 to 13 right-hand sides."""
    import torch

    op = weo.WilsonEO(dims, 0.13, to_device(gen.gauge_field(dims, "smooth", seed=311, eps=0.4)), prec=prec,
                      linkfmt=fmt)
    x = to_device(to_planar(gen.gaussian_spinor(dims, nrhs=13, seed=312)), prec)
    for dag in (False, True):
        one = torch.stack([op.apply(x[r].contiguous(), dag=dag) for r in range(13)])
        for n in (2, 3, 5, 7, 8, 13):
            assert torch.equal(op.apply(x[:n].contiguous(), dag=dag), one[:n])


@pytest.fixture(scope="module")
def weo():
    import paper_2303_08609_gb300 as w

    return w
