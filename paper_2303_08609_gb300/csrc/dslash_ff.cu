// Float-float hopping kernel: Eq. 1 with every real carried as hi + lo of two
// floats (about 48 significant bits from FP32 operations), spinors in SpFF and
// links in LkFF18. FP64-class accuracy without the FP64 pipe.
//
// Both parts of a complex number are kept as (real, imaginary) pairs, the layout
// they have in memory, and all arithmetic uses the two-wide FP32 instructions: half
// the instructions of the scalar form (9.0 k FP32 operations per site and hop),
// which was bound by their issue (70 %). As in weo_split.cuh a CTA of 128 threads
// takes 32 output sites and warp mu the directions +-mu; three warps add the four
// pairs, and the second hop writes complex128 itself. us per M_eo on complex128
// spinors, one site per thread -> here: 8^4 41.9 -> 14.3, 16^3 x 32 119 -> 67.2,
// 24^3 x 48 430 -> 299, 32^3 x 64 1304 -> 915; relative error 2.4e-15 -> 2.3e-15.
// Of the 299, 38 are the conversion of the input and 261 the two hops: issue 45-50 %
// of cycles, bound by the latency of the loads at 16 warps per SM (117 registers;
// three CTAs per SM 301, five or six with spills 314 and 329). Loading both links
// again for each spin row was 344; fetching the next row's values ahead 313.
#include "weo_internal.h"
#include "weo_split.cuh"

namespace weo {

// A complex number in float-float, value h + l
struct FC {
    float2 h, l;
};

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f), a); }

// s + e = a + sg b exactly, sg = +-1 (or +-2) in each half (Knuth's two-sum; sg b
// is exact inside the fused operations)
__device__ __forceinline__ float2 two_sum2(float2 a, float2 b, float2 sg, float2 &e)
{
    const float2 s = fma2(b, sg, a);
    const float2 nb = sub2(a, s);  // -(part of b that reached s)
    e = add2(sub2(a, add2(s, nb)), fma2(b, sg, nb));
    return s;
}

// i z or -i z without the sign: the halves exchanged
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }

// a + sg b, unnormalised
__device__ __forceinline__ FC add_pair(FC a, FC b, float2 sg)
{
    FC r;
    float2 e;
    r.h = two_sum2(a.h, b.h, sg, e);
    r.l = add2(fma2(b.l, sg, a.l), e);
    return r;
}
// z += u v for a real u = uh + ul, in the twice-working-precision manner of
// Ogita, Rump and Oishi (2005): -p is the rounded -uh vh, so e = uh vh - p needs
// no negated operand, and while the products are summed z keeps their negated sum
// in h and every rounding error in l (value l - h)
template <bool FIRST>
__device__ __forceinline__ void ff_product(FC &z, float uh, float ul, FC v)
{
    const float2 u = f2(uh);
    const float2 np = mul2(f2(-uh), v.h);
    float2 e = fma2(u, v.h, np);
    e = fma2(u, v.l, e);
    e = fma2(f2(ul), v.h, e);
    if (FIRST) {
        z.h = np;
        z.l = e;
    } else {
        float2 r;
        const float2 s = two_sum2(z.h, np, f2(1.f), r);
        z.l = add2(z.l, sub2(e, r));
        z.h = s;
    }
}

struct FFLink {
    float r[3][3], i[3][3], rl[3][3], il[3][3];
};

__device__ __forceinline__ void load_ff_link(const char *base, long long vh, uint32_t i, FFLink &U)
{
    cx<float> H[3][3], L[3][3];
    LkF32_18::load(base, vh, i, H);
    LkF32_18::load(base + 72 * vh, vh, i, L);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            U.r[a][b] = H[a][b].r;
            U.i[a][b] = H[a][b].i;
            U.rl[a][b] = L[a][b].r;
            U.il[a][b] = L[a][b].i;
        }
}

__device__ __forceinline__ FC load_fc(const float2 *in, long long vh, int k, uint32_t i)
{
    return {ld_keep(at(in + k * vh, i)), ld_keep(at(in + (12 + k) * vh, i))};
}

// three colours of a spin row and of the row that its projection adds to it
struct FCRows {
    FC a[3], b[3];
};

__device__ __forceinline__ FCRows load_rows(const float2 *a, const float2 *b, long long vh, uint32_t i)
{
    FCRows r;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        r.a[c] = load_fc(a, vh, c, i);
        r.b[c] = load_fc(b, vh, c, i);
    }
    return r;
}

// w = W h of one spin row in one direction (W = U or U^dag), h = psi_row + sg u
// psi_partner with the unit u = i (ROT) or 1
template <bool ROT, bool FWD>
__device__ __forceinline__ void ff_row(const FCRows &r, float sg, const FFLink &U, FC w[3])
{
    FC h[3], g[3];  // g = i h (forward) or -i h
    const float2 s = ROT ? make_float2(-sg, sg) : f2(sg);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const FC y = ROT ? FC{swap2(r.b[c].h), swap2(r.b[c].l)} : r.b[c];
        h[c] = add_pair(r.a[c], y, s);
        g[c] = FWD ? FC{make_float2(-h[c].h.y, h[c].h.x), make_float2(-h[c].l.y, h[c].l.x)}
                   : FC{make_float2(h[c].h.y, -h[c].h.x), make_float2(h[c].l.y, -h[c].l.x)};
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int x = FWD ? k : c, y = FWD ? c : k;
            if (c == 0) ff_product<true>(w[k], U.r[x][y], U.rl[x][y], h[c]);
            else ff_product<false>(w[k], U.r[x][y], U.rl[x][y], h[c]);
            ff_product<false>(w[k], U.i[x][y], U.il[x][y], g[c]);
        }
    // l - h as an ordinary pair, renormalised: without it the low parts of the sums
    // that follow are a few ulps long and the result 7 % further off
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float2 h = w[k].h;
        w[k].h = two_sum2(w[k].l, h, f2(-1.f), w[k].l);
    }
}

// Both hops of direction mu for one site: P + Q (three colours of spin rows 0, 1)
// and P - Q, left in `out` (P waits there for Q, so each link is loaded once for
// both rows). One copy of this code serves two of the directions and
// both spin rows: unrolled over all of them the kernel is 6000 instructions, and
// warps waited for instructions 40 % of the time.
template <bool ROT>
__device__ __forceinline__ void ff_pair(const HopParams &p, const float2 *in, int mu, float s0, uint32_t i, uint32_t nf,
                                        uint32_t nb, float4 *out)
{
    const char *gf = p.gauge + (2 * mu + p.out_parity) * p.gauge_pb;
    const char *gb = p.gauge + (2 * mu + (p.out_parity ^ 1)) * p.gauge_pb;
    // project<MU, S>: the sign of x, y, z, t for spin row s, and the partner's spin
    auto sign = [&](int s) { return mu == 3 || ((mu == 1 || mu == 2) && s) ? -s0 : s0; };
    auto row = [&](int s) { return in + 3ll * s * p.vh; };
    auto partner = [&](int s) { return in + 3ll * (mu < 2 ? 3 - s : 2 + s) * p.vh; };
    FFLink U;
    load_ff_link(gf, p.vh, i, U);
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        FC P[3];
        ff_row<ROT, true>(load_rows(row(s), partner(s), p.vh, nf), sign(s), U, P);
#pragma unroll
        for (int k = 0; k < 3; ++k) out[32 * (3 * s + k)] = make_float4(P[k].h.x, P[k].h.y, P[k].l.x, P[k].l.y);
    }
    load_ff_link(gb, p.vh, nb, U);
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        FC Q[3];
        ff_row<ROT, false>(load_rows(row(s), partner(s), p.vh, nb), -sign(s), U, Q);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float4 f = out[32 * (3 * s + k)];
            const FC P = {make_float2(f.x, f.y), make_float2(f.z, f.w)};
            const FC u = add_pair(P, Q[k], f2(1.f)), d = add_pair(P, Q[k], f2(-1.f));
            out[32 * (3 * s + k)] = make_float4(u.h.x, u.h.y, u.l.x, u.l.y);
            out[32 * (6 + 3 * s + k)] = make_float4(d.h.x, d.h.y, d.l.x, d.l.y);
        }
    }
}

template <bool Dag, bool Axpy, bool OutF64>
__global__ void __launch_bounds__(128, 4) hop_kernel_ff(const HopParams p)
{
    constexpr int S0 = Dag ? -1 : 1;
    __shared__ float4 part[4 * 12 * 32];
    const int lane = (int)threadIdx.x & 31, w = warp_id();
    pdl_wait();
    const int r = (int)blockIdx.y;
    const int b = p.reverse ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x;
    const int i_raw = b * 32 + lane;
    const bool valid = i_raw < p.vh;
    const int i = valid ? i_raw : p.vh - 1;
    int xh, y, z;
    const int t = p.dz.div(p.dy.div(p.dx.div(i, xh), y), z);
    const float2 *in = reinterpret_cast<const float2 *>(static_cast<const char *>(p.in) + r * p.in_stride);
    uint32_t nf, nb;
    switch (w) {
    case 0: nf = dir_neighbour<0, true>(p, i, xh, y, z, t), nb = dir_neighbour<0, false>(p, i, xh, y, z, t); break;
    case 1: nf = dir_neighbour<1, true>(p, i, xh, y, z, t), nb = dir_neighbour<1, false>(p, i, xh, y, z, t); break;
    case 2: nf = dir_neighbour<2, true>(p, i, xh, y, z, t), nb = dir_neighbour<2, false>(p, i, xh, y, z, t); break;
    default: nf = dir_neighbour<3, true>(p, i, xh, y, z, t), nb = dir_neighbour<3, false>(p, i, xh, y, z, t); break;
    }
    if (w & 1) ff_pair<false>(p, in, w, (float)S0, (uint32_t)i, nf, nb, part + w * 12 * 32 + lane);
    else ff_pair<true>(p, in, w, (float)S0, (uint32_t)i, nf, nb, part + w * 12 * 32 + lane);
    FC xv[4];
    if (Axpy && w < 3) {
        const float2 *x = reinterpret_cast<const float2 *>(static_cast<const char *>(p.x) + r * p.x_stride);
#pragma unroll
        for (int k = 0; k < 4; ++k) xv[k] = load_fc(x, p.vh, 3 * k + w, (uint32_t)i);
    }
    __syncthreads();
    pdl_next();
    if (w >= 3 || !valid) return;
    auto read = [&](int m, int k) {
        const float4 q = part[(12 * m + 3 * k + w) * 32 + lane];
        return FC{make_float2(q.x, q.y), make_float2(q.z, q.w)};
    };
    auto turn = [](FC a) { return FC{swap2(a.h), swap2(a.l)}; };
    const float2 one = f2(1.f);
    constexpr float S = (float)S0;
    // spin rows 0, 1: + (P + Q); spin rows 2, 3: - S A^dag (P - Q), row k of it in slot 2 + k
    FC o[4];
    o[0] = add_pair(add_pair(add_pair(read(0, 0), read(1, 0), one), read(2, 0), one), read(3, 0), one);
    o[1] = add_pair(add_pair(add_pair(read(0, 1), read(1, 1), one), read(2, 1), one), read(3, 1), one);
    // x: -S i (d1, d0); y: -S (d1, -d0); z: -S i (d0, -d1); t: -S (d0, d1)
    const float2 ri = make_float2(S, -S), rim = make_float2(-S, S);
    o[2] = add_pair(add_pair(FC{mul2(f2(-S), read(1, 3).h), mul2(f2(-S), read(1, 3).l)}, read(3, 2), f2(-S)), turn(read(0, 3)), ri);
    o[2] = add_pair(o[2], turn(read(2, 2)), ri);
    o[3] = add_pair(add_pair(FC{mul2(f2(S), read(1, 2).h), mul2(f2(S), read(1, 2).l)}, read(3, 3), f2(-S)), turn(read(0, 2)), ri);
    o[3] = add_pair(o[3], turn(read(2, 3)), rim);
    const ff a(p.a);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float2 lo;
        float2 hi = two_sum2(o[k].h, o[k].l, one, lo);  // renormalise
        if (Axpy) {  // x + a H
            const float2 np = mul2(f2(-a.hi), hi);
            float2 e = fma2(f2(a.hi), hi, np), q;
            e = fma2(f2(a.hi), lo, e);
            e = fma2(f2(a.lo), hi, e);
            const float2 s = two_sum2(xv[k].h, np, f2(-1.f), q);
            const float2 u = add2(q, add2(e, xv[k].l));
            hi = add2(s, u);
            lo = sub2(u, sub2(hi, s));
        }
        char *out = static_cast<char *>(p.out) + r * p.out_stride;
        if (OutF64) {
            double2 *q = reinterpret_cast<double2 *>(out) + (long long)(3 * k + w) * p.vh;
            *const_cast<double2 *>(at(q, (uint32_t)i)) = make_double2(ff_join(hi.x, lo.x), ff_join(hi.y, lo.y));
        } else {
            float2 *q = reinterpret_cast<float2 *>(out) + (long long)(3 * k + w) * p.vh;
            *const_cast<float2 *>(at(q, (uint32_t)i)) = hi;
            *const_cast<float2 *>(at(q + 12ll * p.vh, (uint32_t)i)) = lo;
        }
    }
}

template <bool Dag, bool Axpy, bool OutF64>
static int launch_ff(const HopParams &p, cudaStream_t s)
{
    const unsigned nsb = (unsigned)((p.vh + 31) / 32);
    HopParams q = p;
    for (long long r = 0; r < p.nrhs; r += kGridRows) {
        q.nrhs = (int)(p.nrhs - r < kGridRows ? p.nrhs - r : kGridRows);
        q.in = static_cast<const char *>(p.in) + r * p.in_stride;
        q.out = static_cast<char *>(p.out) + r * p.out_stride;
        if (Axpy) q.x = static_cast<const char *>(p.x) + r * p.x_stride;
        WEO_TRY(launch_dependent(hop_kernel_ff<Dag, Axpy, OutF64>, dim3(nsb, (unsigned)q.nrhs), 128, s, q));
    }
    return WEO_OK;
}

int launch_hop_ff(bool dag, bool axpy, const HopParams &p, const LaunchCfg &, cudaStream_t s)
{
    if (axpy && p.out_f64) return dag ? launch_ff<true, true, true>(p, s) : launch_ff<false, true, true>(p, s);
    if (dag) return axpy ? launch_ff<true, true, false>(p, s) : launch_ff<true, false, false>(p, s);
    return axpy ? launch_ff<false, true, false>(p, s) : launch_ff<false, false, false>(p, s);
}

}  // namespace weo
