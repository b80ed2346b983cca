"""What a user of this package has it do, as cases that can be timed.

Each case is one pass through the public entry points (``WilsonEO``, the batch
call and the differentiable action) on inputs made on the GPU from a seed: links
exp(i eps H) or Haar-random, Gaussian sources, the lattices of this repository's
benchmark, workload table and tests, and ragged ones between them.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes the inputs and the handle, ``run`` is the pass, ``work`` the bytes
and operations that the pass cannot do without, and ``exact`` the result in
64-bit arithmetic written out in plain torch.
"""

from __future__ import annotations

import torch

import paper_2303_08609_gb300 as weo
from paper_2303_08609_gb300 import autograd as weo_autograd

FLOP_PER_SITE = 1344  # one M_eo per lattice site: two hops of 1320 per output site, and the diagonal term


def _case(name, kind, dims, prec, **more):
    c = {"name": name, "kind": kind, "dims": dims, "prec": prec, "linkfmt": 18, "nrhs": 1, "kappa": 0.13,
         "links": "smooth", "dag": False, "staged": False, "tol": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: the parity workload of the operator, FP64 on Haar links, latency alone
        _case("meo_8x8x8x8_f64", "meo", "8x8x8x8", "f64", kappa=0.125, links="haar"),
        # a small ragged lattice, the adjoint, compressed links: extents that no tile divides
        _case("meo_10x6x14x18_f32_l12", "meo", "10x6x14x18", "f32", linkfmt=12, dag=True),
        # M^dag M on an ordinary lattice with the default handle: what a user's own Krylov solver calls
        _case("normal_16x16x16x32_f32", "normal", "16x16x16x32", "f32"),
        # the benchmark's main line: M^dag M on the large lattice, hops staged by TMA
        _case("normal_32x32x32x64_f32_staged", "normal", "32x32x32x64", "f32", staged=True),
        # the largest lattice, that of the solve, with the 16-bit operator that the mixed solver iterates
        _case("normal_48x48x48x96_f16_l12", "normal", "48x48x48x96", "f16", linkfmt=12, kappa=0.135),
        # the FP64 operator on an ordinary lattice: references, and the plain solver's operator
        _case("normal_16x16x16x32_f64", "normal", "16x16x16x32", "f64"),
        # FP64-class accuracy from FP32 arithmetic: the residuals of a user's own refinement loop
        _case("ff64_24x24x24x48", "ff64", "24x24x24x48", "f64"),
        # a propagator's 12 spin-colour right-hand sides in one call
        _case("meo_12rhs_24x24x24x48_f32", "meo", "24x24x24x48", "f32", nrhs=12),
        # one molecular-dynamics step of HMC: new links, then the pseudofermion force and dS/dphi
        _case("force_24x24x24x48_f32", "force", "24x24x24x48", "f32"),
        # the differentiable action in a training loop, FP64: forward, and gradients of source and links
        _case("autograd_16x16x16x32_f64", "autograd", "16x16x16x32", "f64"),
        # an ensemble of different lattices in one launch (the mixed batch of the workload table)
        _case("batch_16_24_32_f32", "batch", "16x16x16x16,24x24x24x48,32x32x32x64", "f32", links="haar"),
        # a whole mixed-precision solve with 16-bit links, to the residual that HMC's energies need
        _case("solve_16x16x16x32_f16_l12", "solve", "16x16x16x32", "f16", linkfmt=12, tol=1e-12),
    ]


# ------------------------------------------------------------------ drawing --
def _draw_dims(rng, lo, hi):
    """Even extents with a volume between lo and hi, spread over its logarithm."""
    while True:
        want = lo * (hi / lo) ** rng.random()
        d = [2 * rng.randint(2, 24) for _ in range(3)]
        lt = 2 * round(want / (d[0] * d[1] * d[2]) / 2)
        if 2 <= lt <= 96:
            v = d[0] * d[1] * d[2] * lt
            if lo * 0.9 <= v <= hi:
                return d + [lt], v


def _text(d):
    return "x".join(str(x) for x in d)


def draw(rng):
    kind = rng.choice(["meo", "meo", "normal", "normal", "meo", "ff64", "rhs", "force", "autograd", "batch", "solve"])
    links = rng.choice(["smooth", "haar"])
    kappa = round(rng.uniform(0.12, 0.135), 4)
    fmt = rng.choice([18, 12])
    dag = rng.random() < 0.5
    top = 32 ** 3 * 64
    if kind in ("meo", "normal"):
        prec = rng.choice(["f32", "f32", "f16", "bf16", "f64"])
        d, _ = _draw_dims(rng, 2 ** 11, top // 8 if prec == "f64" else 2 * top if prec != "f32" else top)
        c = _case("", kind, _text(d), prec, linkfmt=fmt)
        rows = [r for r in range(2, d[1] + 1) if d[1] % r == 0 and r * (d[0] // 2) <= 64]
        if prec == "f32" and fmt == 18 and d[0] % 4 == 0 and rows and rng.random() < 0.5:
            c["staged"] = True
    elif kind == "ff64":
        d, _ = _draw_dims(rng, 2 ** 12, 24 ** 3 * 48)
        c = _case("", "ff64", _text(d), "f64")
    elif kind == "rhs":  # several right-hand sides in one call
        n = rng.randint(2, 16)
        prec = rng.choice(["f32", "f32", "f16", "bf16"])
        d, _ = _draw_dims(rng, 2 ** 12, min(top, 24 ** 3 * 48 * 12 // n))
        c = _case("", "meo", _text(d), prec, linkfmt=fmt, nrhs=n)
    elif kind == "force":
        d, _ = _draw_dims(rng, 2 ** 12, 24 ** 3 * 48)
        c = _case("", "force", _text(d), rng.choice(["f32", "f32", "f64"]), linkfmt=fmt)
        if c["prec"] == "f64":
            d, _ = _draw_dims(rng, 2 ** 12, 16 ** 3 * 32)
            c["dims"] = _text(d)
    elif kind == "autograd":
        prec = rng.choice(["f64", "f32"])
        d, _ = _draw_dims(rng, 2 ** 12, 16 ** 3 * 32 if prec == "f64" else 24 ** 3 * 48)
        c = _case("", "autograd", _text(d), prec, linkfmt=fmt)
    elif kind == "batch":
        ds = [_draw_dims(rng, 2 ** 12, 24 ** 3 * 48)[0] for _ in range(rng.randint(2, 5))]
        c = _case("", "batch", ",".join(_text(d) for d in ds), "f32", linkfmt=fmt)
    else:
        n = rng.choice([1, 1, 1, 2, 4])
        d, _ = _draw_dims(rng, 2 ** 12, 16 ** 3 * 32 // n)
        c = _case("", "solve", _text(d), rng.choice(["f16", "bf16", "f32"]), linkfmt=fmt, nrhs=n, tol=1e-12)
    c.update(links=links, kappa=kappa, dag=dag)
    if c["kind"] == "solve":  # the smooth field and kappa of the benchmark's batched solve: they converge
        c.update(links="smooth", kappa=0.13, dag=False)
    if c["kind"] != "meo" and c["kind"] != "batch" and c["kind"] != "ff64":
        c["dag"] = False
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs --
def _dims(text):
    return [tuple(int(x) for x in d.split("x")) for d in text.split(",")]


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _mm(a, b):
    """Products of 3x3 matrices, elementwise over the leading axes."""
    return sum(a[..., :, k:k + 1] * b[..., k:k + 1, :] for k in range(3))


def _gaussian(gen, shape):
    """Complex normal numbers with E|z|^2 = 1."""
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda", dtype=torch.float64) * 0.5 ** 0.5)


def _links(gen, n, kind):
    """n SU(3) matrices: exp(i 0.4 H), H random traceless Hermitian, or Haar."""
    z = _gaussian(gen, (n, 3, 3))
    if kind == "smooth":
        h = 0.5 * (z + z.transpose(1, 2).conj())
        h = h - torch.diagonal(h, dim1=1, dim2=2).real.mean(1)[:, None, None] * torch.eye(3, device="cuda")
        x = (0.4j / 8) * h  # scaling and squaring
        u = torch.eye(3, device="cuda", dtype=torch.complex128) + x
        term = x
        for k in range(2, 11):
            term = _mm(term, x) / k
            u = u + term
        for _ in range(3):
            u = _mm(u, u)
        return u
    cols = []  # Gram-Schmidt with a positive diagonal, then determinant 1
    for k in range(3):
        v = z[:, :, k]
        for q in cols:
            v = v - (q.conj() * v).sum(1, keepdim=True) * q
        cols.append(v / torch.linalg.vector_norm(v, dim=1, keepdim=True))
    u = torch.stack(cols, 2)
    return u / torch.exp(1j * torch.angle((u[:, :, 0] * torch.linalg.cross(u[:, :, 1], u[:, :, 2])).sum(1)) / 3)[:, None, None]


def _gauge(gen, dims, case):
    v = _volume(dims)
    dtype = torch.complex128 if case["prec"] == "f64" else torch.complex64
    u = torch.empty(4, v, 3, 3, device="cuda", dtype=dtype)
    for mu in range(4):
        for a in range(0, v, 1 << 21):
            n = min(1 << 21, v - a)
            u[mu, a:a + n] = _links(gen, n, case["links"])
    return u


def _spinor(gen, dims, case, wide=False):
    shape = (4, 3, _volume(dims) // 2)
    if case["nrhs"] > 1:
        shape = (case["nrhs"],) + shape
    x = _gaussian(gen, shape)
    return x if wide or case["prec"] == "f64" else x.to(torch.complex64)


def _inputs(case, seed):
    """(dims, links, spinor) of every lattice of the case."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    got = []
    for dims in _dims(case["dims"]):
        u = _gauge(gen, dims, case)
        got.append((dims, u, _spinor(gen, dims, case, wide=case["kind"] == "solve")))
    return got


def _kappa(case, k):
    """The lattices of a batch have hopping parameters of their own."""
    return case["kappa"] - 0.004 * k


def prepare(case, seed):
    got = _inputs(case, seed)
    ops = []
    for k, (dims, u, _) in enumerate(got):
        op = weo.WilsonEO(dims, _kappa(case, k), u, prec=case["prec"], linkfmt=case["linkfmt"])
        if case["staged"]:
            weo.wilson_eo_set_staging(op.handle, True)
        ops.append(op)
    kind = case["kind"]
    s = {"kind": kind, "case": case, "op": ops[0], "x": got[0][2]}
    if kind == "force":
        s["u"] = got[0][1]
    elif kind == "autograd":
        s["u"] = got[0][1].requires_grad_()
        s["x"].requires_grad_()
    elif kind == "batch":
        s["ops"] = ops
        s["handles"] = [op.handle for op in ops]
        s["ins"] = [x for _, _, x in got]
        s["outs"] = [torch.empty_like(x) for x in s["ins"]]
    return s


def run(s):
    kind, case, op, x = s["kind"], s["case"], s["op"], s["x"]
    if kind == "meo":
        return op.apply(x, dag=case["dag"])
    if kind == "normal":
        y = op.apply(x)
        return y, op.apply(y, dag=True)
    if kind == "ff64":
        return op.apply_ff64(x, dag=case["dag"])
    if kind == "force":
        op.set_gauge(s["u"])
        return op.force(x, want_dphi=True)
    if kind == "autograd":
        action = weo_autograd.pseudofermion_action(x, s["u"], op)
        return (action.detach(),) + torch.autograd.grad(action, (x, s["u"]))
    if kind == "batch":
        weo.wilson_eo_apply_batch(s["handles"], s["outs"], s["ins"], dag=case["dag"])
        return s["outs"]
    x, _ = op.solve(x, tol=case["tol"], mixed=True)
    return x


# --------------------------------------------------------------------- work --
def work(case):
    """Each input read once and each output written once, and the operations of
    the hopping sums (1344 per lattice site and M_eo)."""
    kind, n = case["kind"], case["nrhs"]
    wide = case["prec"] == "f64"
    link = {"f64": 144, "f32": 72, "f16": 36, "bf16": 36}[case["prec"]] * (2 if case["linkfmt"] == 12 else 3) // 3
    sp = 192 if wide or kind == "solve" else 96  # bytes of a spinor
    v = sum(_volume(d) for d in _dims(case["dims"]))
    vh = v // 2
    if kind == "meo" or kind == "batch":
        return {"bytes": v * 4 * link + 2 * n * vh * sp, "flops": n * v * FLOP_PER_SITE}
    if kind == "normal":
        return {"bytes": v * 4 * link + 3 * n * vh * sp, "flops": 2 * n * v * FLOP_PER_SITE}
    if kind == "ff64":
        return {"bytes": v * 4 * 144 + 2 * vh * 192, "flops": v * FLOP_PER_SITE}
    if kind in ("force", "autograd"):
        # links in, force or gradient out, phi in, dS/dphi out; M, M^dag and per link
        # two outer products of 2-spinors (2 x 144) and, for the force, a 3x3 product
        links = 4 * v * (144 if wide else 72)
        return {"bytes": 2 * links + 2 * vh * sp,
                "flops": 2 * v * FLOP_PER_SITE + 4 * v * (2 * 144 + 48 + (216 if kind == "force" else 0))}
    # about 140 iterations of M^dag M take the residual to 1e-12 at kappa = 0.13;
    # the fields are read and written once, as a lattice that stays on chip would
    return {"bytes": v * 4 * 144 + 2 * n * vh * 192, "flops": 140 * 2 * n * v * FLOP_PER_SITE}


# -------------------------------------------------------------------- exact --
def _gamma():
    s = [[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]]
    g = []
    for k in range(3):
        m = torch.zeros(4, 4, dtype=torch.complex128, device="cuda")
        sk = torch.tensor(s[k], dtype=torch.complex128, device="cuda")
        m[:2, 2:], m[2:, :2] = -1j * sk, 1j * sk
        g.append(m)
    m = torch.zeros(4, 4, dtype=torch.complex128, device="cuda")
    m[0, 2] = m[1, 3] = m[2, 0] = m[3, 1] = 1
    return g + [m]


def _hop(u, psi, sign):
    """sum_mu (1 - s g) U_mu(x) psi(x+mu) + (1 + s g) U_mu^dag(x-mu) psi(x-mu) on the
    whole lattice; u (4, T, Z, Y, X, 3, 3), psi (T, Z, Y, X, 4, 3)."""
    one = torch.eye(4, dtype=torch.complex128, device="cuda")
    out = None
    for mu, g in enumerate(_gamma()):
        ax = 3 - mu
        h = torch.einsum("st,xyzwtc->xyzwsc", one - sign * g, torch.roll(psi, -1, ax))
        f = sum(u[mu][..., None, :, b] * h[..., :, b, None] for b in range(3))
        h = torch.einsum("st,xyzwtc->xyzwsc", one + sign * g, psi)
        w = sum(u[mu].conj()[..., None, b, :] * h[..., :, b, None] for b in range(3))
        f = f + torch.roll(w, 1, ax)
        out = f if out is None else out + f
    return out


class _Exact:
    """M_eo of one lattice in 64 bits on full-lattice fields."""

    def __init__(self, dims, u, kappa):
        lx, ly, lz, lt = dims
        self.shape = (lt, lz, ly, lx)
        self.u, self.kappa = u.to(torch.complex128).reshape(4, *self.shape, 3, 3), kappa
        c = [torch.arange(n, device="cuda") for n in self.shape]
        par = (c[0][:, None, None, None] + c[1][None, :, None, None] + c[2][None, None, :, None] + c[3]) % 2
        self.even = torch.nonzero(par.reshape(-1) == 0)[:, 0]

    def meo(self, x, dag=False):
        """x: (4, 3, V/2) complex128."""
        full = torch.zeros(self.shape[0] * self.shape[1] * self.shape[2] * self.shape[3], 4, 3,
                           dtype=torch.complex128, device="cuda").index_copy(0, self.even, x.permute(2, 0, 1))
        psi = full.reshape(*self.shape, 4, 3)
        sign = -1.0 if dag else 1.0
        r = psi - self.kappa ** 2 * _hop(self.u, _hop(self.u, psi, sign), sign)
        return r.reshape(-1, 4, 3)[self.even].permute(1, 2, 0).contiguous()


def _cg(m, b):
    """x with M^dag M x = b, as far as 64 bits go."""
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), float((r.abs() ** 2).sum())
    stop = 1e-30 * rr
    for _ in range(600):
        q = m.meo(p)
        a = rr / float((q.abs() ** 2).sum())
        x = x + a * p
        r = r - a * m.meo(q, True)
        new = float((r.abs() ** 2).sum())
        if new <= stop:
            break
        p, rr = r + (new / rr) * p, new
    return x


def exact(case, seed):
    kind = case["kind"]
    got = _inputs(case, seed)
    if kind == "batch":
        return [_Exact(d, u, _kappa(case, k)).meo(x.to(torch.complex128), case["dag"]) for k, (d, u, x) in enumerate(got)]
    dims, u, x = got[0]
    x = x.to(torch.complex128)
    m = _Exact(dims, u, case["kappa"])
    each = x if x.dim() == 4 else x[None]
    if kind in ("meo", "ff64"):
        y = torch.stack([m.meo(v, case["dag"]) for v in each])
        return y.reshape(x.shape)
    if kind == "normal":
        y = m.meo(x)
        return y, m.meo(y, True)
    if kind == "solve":
        return torch.stack([_cg(m, v) for v in each]).reshape(x.shape)
    x = x.detach().requires_grad_()
    m.u = m.u.detach().requires_grad_()
    y = m.meo(x)
    action = (y.real ** 2 + y.imag ** 2).sum()
    gx, gu = torch.autograd.grad(action, (x, m.u))
    gu = gu.reshape(4, -1, 3, 3)
    if kind == "autograd":
        return action.detach(), gx, gu
    w = _mm(gu, m.u.detach().reshape(4, -1, 3, 3).transpose(2, 3).conj())
    w = 0.5 * (w - w.transpose(2, 3).conj())
    tr = torch.diagonal(w, dim1=2, dim2=3).sum(2) / 3
    return w - tr[..., None, None] * torch.eye(3, device="cuda"), gx
