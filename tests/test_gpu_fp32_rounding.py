"""FP32 and 16-bit M_eo against a model that rounds as the kernels do, bit by bit.

Where a result is rounded to 16 bits again, an FP32 rounding taken in another order
moves single elements by a whole step of the format (2^-8 of the site's norm with
BF16), far inside the bounds against the oracle. The model is plain numpy in FP32
with exactly rounded fused operations, so the outputs have to be equal. Extents of
2, where both neighbours of an axis are one site, add such steps up.
"""

from fractions import Fraction

import numpy as np
import pytest

import gen
from gpu_util import to_device, to_planar
from lattice_ref import parity_sites, shift_index

F, D = np.float32, np.float64


def fma(a, b, c):
    """a b + c of FP32 arrays, rounded once: the product is exact in FP64, and the sum
    is rounded to odd there, so that the step to FP32 rounds as from the exact value."""
    p, c = D(a) * D(b), D(c)
    s = p + c
    t = s - p
    e = (p - (s - t)) + (c - t)
    even = (s.view(np.int64) & 1) == 0
    return F(np.where((e != 0) & even, np.nextafter(s, np.where(e > 0, np.inf, -np.inf)), s))


def test_fused_operation_of_the_model():
    rng = np.random.default_rng(1)
    a, b = (F(rng.normal(size=20000)) for _ in range(2))
    # sums next to a midpoint of FP32, where rounding twice goes wrong
    c = F(rng.normal(size=20000) * 2.0 ** rng.integers(-30, 30, 20000))
    for x, y, z, r in zip(a, b, c, fma(a, b, c)):
        want = Fraction(float(x)) * Fraction(float(y)) + Fraction(float(z))
        err = abs(Fraction(float(r)) - want)
        for q in (np.nextafter(r, F(np.inf)), np.nextafter(r, F(-np.inf))):
            assert err <= abs(Fraction(float(q)) - want)


def round16(v, prec):
    if prec == "f16":
        return F(np.float16(v))
    u = np.ascontiguousarray(v, dtype=F).view(np.uint32).astype(np.uint64)  # to nearest, ties to even
    return ((u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(F)


class C:
    """Complex FP32 arrays as the kernels hold them."""

    def __init__(self, r, i):
        self.r, self.i = r, i

    def __add__(self, o):
        return C(self.r + o.r, self.i + o.i)

    def __sub__(self, o):
        return C(self.r - o.r, self.i - o.i)

    def times_i(self):
        return C(-self.i, self.r)

    def conj(self):
        return C(self.r, -self.i)


def cfma(a, b, acc, conj=False):
    ai = -a.i if conj else a.i
    return C(fma(-ai, b.i, fma(a.r, b.r, acc.r)), fma(ai, b.r, fma(a.r, b.i, acc.i)))


ZERO = C(F(0), F(0))


def cmul(a, b):
    return cfma(a, b, ZERO)


def links(U, prec, fmt):
    """Stored links as 3x3 of C over (mu, lex)."""
    f = U.astype(np.complex64)
    r, i = F(f.real), F(f.imag)
    if prec in ("f16", "bf16"):
        r, i = round16(r, prec), round16(i, prec)
    L = [[C(r[..., a, b], i[..., a, b]) for b in range(3)] for a in range(3)]
    if fmt == 12:
        L[2] = [(cmul(L[0][(c + 1) % 3], L[1][(c + 2) % 3]) - cmul(L[0][(c + 2) % 3], L[1][(c + 1) % 3])).conj()
                for c in range(3)]
    return L


def scaled(a, b, plus, n):
    """(a +- b) n: the second value times n rounded, the first added in one operation."""
    if n is None:
        return a + b if plus else a - b
    s = F(1) if plus else F(-1)
    return C(fma(a.r, n, s * (b.r * n)), fma(a.i, n, s * (b.i * n)))


# per direction: does row k take i times its partner (else 1), the partner of rows 0 and 1,
# and their signs for the projector 1 - gamma
RULE = [(True, (3, 2), (1, 1)), (False, (3, 2), (1, -1)), (True, (2, 3), (1, -1)), (False, (2, 3), (-1, -1))]


def hop(v, L, dims, out_parity, dag, norm=None):
    """Sum over the directions, in the kernels' order, of one site's [spin][colour]."""
    here, there = parity_sites(dims, out_parity), parity_sites(dims, out_parity ^ 1)
    index = np.empty(int(np.prod(dims)), dtype=int)
    index[there] = np.arange(len(there))
    out = [[C(np.zeros(len(here), F), np.zeros(len(here), F)) for _ in range(3)] for _ in range(4)]
    for mu in range(4):
        rot, partner, sign = RULE[mu]
        for fwd in (True, False):
            nb = shift_index(dims, mu, 1 if fwd else -1)[here]
            at = index[nb]
            S = 1 if fwd != dag else -1
            n = None if norm is None else norm[at]
            get = lambda s, c: C(v[s][c].r[at], v[s][c].i[at])
            h = [[None] * 3 for _ in range(2)]
            for k in range(2):
                for c in range(3):
                    q = get(partner[k], c)
                    h[k][c] = scaled(get(k, c), q.times_i() if rot else q, sign[k] * S > 0, n)
            base = here if fwd else nb
            W = [[C(L[a][b].r[mu][base], L[a][b].i[mu][base]) for b in range(3)] for a in range(3)]
            for k in range(2):
                for a in range(3):
                    z = ZERO
                    for b in range(3):
                        z = cfma(W[a][b], h[k][b], z) if fwd else cfma(W[b][a], h[k][b], z, conj=True)
                    out[k][a] = out[k][a] + z
                    # the lower rows: A^dag of the projection, with its unit and sign
                    low = partner[k]
                    down = z.times_i() if rot else z
                    plus = (sign[k] * S > 0) != rot
                    out[low][a] = out[low][a] + down if plus else out[low][a] - down
    return out


def meo_model(U, kappa, psi, dims, prec, fmt, dag):
    L = links(U, prec, fmt)
    x = psi.astype(np.complex64)
    v = [[C(F(x[s, c].real), F(x[s, c].imag)) for c in range(3)] for s in range(4)]
    odd = hop(v, L, dims, 1, dag)
    norm = None
    if prec in ("f16", "bf16"):
        flat = [p for row in odd for z in row for p in (z.r, z.i)]
        norm = np.max(np.abs(flat), axis=0)
        s = F(1) / norm
        odd = [[C(round16(z.r * s, prec), round16(z.i * s, prec)) for z in row] for row in odd]
    out = hop(odd, L, dims, 0, dag, norm)
    a = F(-kappa * kappa)
    return np.stack([np.stack([fma(a, out[s][c].r, v[s][c].r) + 1j * fma(a, out[s][c].i, v[s][c].i) for c in range(3)])
                     for s in range(4)]).astype(np.complex64)


def inputs(dims):
    return gen.gauge_field(dims, "haar", seed=401), to_planar(gen.gaussian_spinor(dims, seed=402)[0])


@pytest.mark.parametrize("fmt", [18, 12])
def test_model_is_the_operator(oracle_lib, fmt):
    """The model against the oracle: 1e-5, the bound of FP32 results."""
    dims = (2, 4, 2, 6)
    U, psi = inputs(dims)
    site_major = np.moveaxis(psi, -1, 0)
    for dag in (False, True):
        want = to_planar((oracle_lib.meo_dag if dag else oracle_lib.meo)(U, 0.13, np.ascontiguousarray(site_major), dims))
        got = meo_model(U, 0.13, psi, dims, "f32", fmt, dag)
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.gpu
@pytest.mark.parametrize("prec,fmt", [("bf16", 18), ("bf16", 12), ("f16", 18), ("f16", 12), ("f32", 18), ("f32", 12)])
@pytest.mark.parametrize("dims", [(2, 4, 2, 6), (6, 2, 10, 2), (8, 6, 4, 10)])
def test_bitwise_the_model(dims, prec, fmt):
    import paper_2303_08609_gb300 as weo

    U, psi = inputs(dims)
    with weo.WilsonEO(dims, 0.13, to_device(U), prec=prec, linkfmt=fmt) as op:
        x = to_device(psi, prec)
        for dag in (False, True):
            got = op.apply(x, dag=dag).cpu().numpy()
            want = meo_model(U, 0.13, psi, dims, prec, fmt, dag)
            assert np.array_equal(got, want), np.mean(got != want)
