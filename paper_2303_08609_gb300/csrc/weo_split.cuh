// Hopping kernels that spread a site's eight directions over the warps of a CTA:
// hop_site's sums, term by term in its order, so the results are bitwise its.
//
// With one site per thread a thread walks the eight directions one after the
// other: eight dependent rounds of loads, 24 accumulators and the index
// arithmetic of all neighbours in registers (spilled at the 64 that half
// occupancy allows), and on a small lattice a handful of warps per SM. Here a CTA
// of 128 threads takes 32 consecutive output sites, and warp mu of it the
// directions +-mu of all 32: it projects, multiplies and leaves the two spin rows
// of each direction in shared memory; three warps then add the directions, one
// colour each, apply the axpy and store. All loads of a site are in flight at
// once, and a thread needs 48 to 64 registers. The plane bases are the same for
// the whole warp and the offsets 32 bits (at()), so a load needs no address
// arithmetic of its own: with 64-bit offsets the same kernel ran 14 % slower at
// 32^3 x 64 and 45 % slower with 16-bit storage.
//
// us per M_eo on one GB300, one site per thread -> split:
//   lattice        FP32 18-real     FP32 12-real     FP16 18-real     FP64 18-real
//   8^4            10.9 -> 3.7       8.6 -> 4.1       9.4 -> 4.3      63.7 -> 12.6
//   16^3 x 32      25.4 -> 15.5     19.0 -> 13.5     20.0 -> 13.2      243 -> 207
//   24^3 x 48       104 -> 77       77.0 -> 65.2     68.9 -> 56.6     1070 -> 996
//   32^3 x 64       278 -> 240       227 -> 196       181 -> 171
//   48^3 x 96      1358 -> 1205     1109 -> 977       867 -> 848
// CTAs of 64 or 128 sites measured slower (249 and 261 us at 32^3 x 64, FP32
// 18-real), and so did both spin rows of a colour as one 16-byte value (257:
// spills).
// FP32 18-real links: bound by HBM (7.1 TB/s of the two passes' 816 B per site at
// 32^3 x 64; the copy bandwidth is 6.8, part of the intermediate stays in L2).
// 12-real and 16-bit links: instruction issue (68-72 % of cycles at 32^3 x 32 with
// FP16) and the L1 / shared-memory path (57-76 %) together. FP64: the FP64 pipe.
#pragma once

#include "weo_dslash.cuh"
#include "weo_route.h"

namespace weo {

// chi = W h of one direction for one site, two spin rows x three colours
template <int MU, bool FWD, int S0, class N>
__device__ __forceinline__ void dir_chi(const cx<float> U[3][3], const cx<float> v[12], N scale, float2 *out)
{
    constexpr int S = FWD ? S0 : -S0;
    cx<float> h[2][3], w[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) project<MU, S>(v[c], v[3 + c], v[6 + c], v[9 + c], h[0][c], h[1][c], scale);
    link_mul<FWD>(U, h, w);
#pragma unroll
    for (int k = 0; k < 6; ++k) out[32 * k] = make_float2(w[k / 3][k % 3].r, w[k / 3][k % 3].i);
}

// add direction (MU, FWD) of one colour to the four spin rows
template <int MU, bool FWD, int S0>
__device__ __forceinline__ void dir_add(cx<float> o[4], const float2 *chi)
{
    const float2 a = chi[0], b = chi[32 * 3];
    reconstruct<MU, FWD ? S0 : -S0>(o[0], o[1], o[2], o[3], cx<float>{a.x, a.y}, cx<float>{b.x, b.y});
}

// wait for the other two warps that finish the same right-hand side
__device__ __forceinline__ void finish_sync() { asm volatile("bar.sync 1, 96;" ::: "memory"); }

// The 16-bit store of one site whose spinor is spread over three threads (one
// colour each): the site's norm and the packed words are exchanged through
// shared memory (mx: 3 x 32 floats, wd: 12 x 32 words), and each thread writes
// one of the three uint4 planes.
template <class Tr>
__device__ __forceinline__ void store16_split(const cx<float> o[4], int c, int lane, void *base, long long vh,
                                              long long i, bool valid, float *mx, uint32_t *wd)
{
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) m = fmaxf(m, fmaxf(fabsf(o[k].r), fabsf(o[k].i)));
    mx[32 * c + lane] = m;
    finish_sync();
    m = fmaxf(fmaxf(mx[lane], mx[32 + lane]), mx[64 + lane]);
    const float s = m > 0.f ? 1.0f / m : 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) wd[32 * (3 * k + c) + lane] = Tr::from_f2(o[k].r * s, o[k].i * s);
    finish_sync();
    if (!valid) return;
    uint4 *p = static_cast<uint4 *>(base);
    const uint32_t *q = wd + 32 * 4 * c + lane;
    p[c * vh + i] = make_uint4(q[0], q[32], q[64], q[96]);
    if (c == 0) reinterpret_cast<float *>(p + 3 * vh)[i] = m;
}

template <class S>
struct Is16 {
    static constexpr bool value = false;
    using traits = void;
};
template <class Tr>
struct Is16<Sp16<Tr>> {
    static constexpr bool value = true;
    using traits = Tr;
};

// neighbour of site i in direction (MU, FWD), from the site's coordinates
template <int MU, bool FWD>
__device__ __forceinline__ uint32_t dir_neighbour(const HopParams &p, int i, int xh, int y, int z, int t)
{
    if (MU == 0) {
        const int par = (y + z + t + p.out_parity) & 1;
        if (FWD) return (uint32_t)(par ? (xh + 1 == p.lxh ? i - xh : i + 1) : i);
        return (uint32_t)(par ? i : (xh == 0 ? i + p.lxh - 1 : i - 1));
    }
    const int c = MU == 1 ? y : MU == 2 ? z : t, n = MU == 1 ? p.ly : MU == 2 ? p.lz : p.lt;
    const int step = MU == 1 ? p.lxh : MU == 2 ? p.lxh * p.ly : p.lxh * p.ly * p.lz;
    if (FWD) return (uint32_t)(c + 1 == n ? i - (n - 1) * step : i + step);
    return (uint32_t)(c == 0 ? i + (n - 1) * step : i - step);
}

__device__ __forceinline__ uint32_t neighbour_of(const HopParams &p, int d, int i)
{
    int xh, y, z;
    const int t = p.dz.div(p.dy.div(p.dx.div(i, xh), y), z);
    switch (d) {
    case 0: return dir_neighbour<0, true>(p, i, xh, y, z, t);
    case 1: return dir_neighbour<0, false>(p, i, xh, y, z, t);
    case 2: return dir_neighbour<1, true>(p, i, xh, y, z, t);
    case 3: return dir_neighbour<1, false>(p, i, xh, y, z, t);
    case 4: return dir_neighbour<2, true>(p, i, xh, y, z, t);
    case 5: return dir_neighbour<2, false>(p, i, xh, y, z, t);
    case 6: return dir_neighbour<3, true>(p, i, xh, y, z, t);
    default: return dir_neighbour<3, false>(p, i, xh, y, z, t);
    }
}

// the warp's number, known to the compiler to be the same in all its lanes
__device__ __forceinline__ int warp_id() { return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0); }

// three warps add the eight directions of one colour each, apply the axpy and store
template <class SOut, bool Dag, bool Axpy>
__device__ __forceinline__ void finish_site(const HopParams &p, char *out, const float2 *cb, int c, int lane, uint32_t i,
                                            bool valid, const float2 xv[4], float *mx, uint32_t *wd)
{
    constexpr int S0 = Dag ? -1 : 1;
    cx<float> o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = {0.f, 0.f};
    dir_add<0, true, S0>(o, cb);
    dir_add<0, false, S0>(o, cb + 1 * 192);
    dir_add<1, true, S0>(o, cb + 2 * 192);
    dir_add<1, false, S0>(o, cb + 3 * 192);
    dir_add<2, true, S0>(o, cb + 4 * 192);
    dir_add<2, false, S0>(o, cb + 5 * 192);
    dir_add<3, true, S0>(o, cb + 6 * 192);
    dir_add<3, false, S0>(o, cb + 7 * 192);
    if (Axpy) {
        const float a = float(p.a);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            o[k].r = fmaf(a, o[k].r, xv[k].x);
            o[k].i = fmaf(a, o[k].i, xv[k].y);
        }
    }
    if constexpr (Is16<SOut>::value) {
        store16_split<typename Is16<SOut>::traits>(o, c, lane, out, p.vh, i, valid, mx, wd);
    } else if (valid) {
        float2 *q = reinterpret_cast<float2 *>(out) + (long long)c * p.vh;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            *const_cast<float2 *>(at(q + 3ll * k * p.vh, i)) = make_float2(o[k].r, o[k].i);
    }
}

// scratch of one 32-site block
template <bool OUT16>
struct DirsShared {
    float2 chi[8 * 6 * 32];
    float mx[OUT16 ? 96 : 1];
    uint32_t wd[OUT16 ? 384 : 1];
};

// The 32 sites from 32 b on, for right-hand side r, by the 128 threads of a CTA
template <class SIn, class SOut, class SX, class Lk, bool Dag, bool Axpy, bool MULTI>
__device__ __forceinline__ void dirs_block(const HopParams &p, int b, int r, DirsShared<Is16<SOut>::value> &sh)
{
    constexpr int S0 = Dag ? -1 : 1;
    const int lane = (int)threadIdx.x & 31, w = warp_id();
    const char *in = static_cast<const char *>(p.in) + (MULTI ? r * p.in_stride : 0);
    const int i_raw = b * 32 + lane;
    const bool valid = i_raw < p.vh;
    const int i = valid ? i_raw : p.vh - 1;  // the last block's spare lanes repeat its last site
    int xh, y, z;
    const int t = p.dz.div(p.dy.div(p.dx.div(i, xh), y), z);
    auto dir = [&](auto mu, auto fwd) {
        constexpr int MU = decltype(mu)::value;
        constexpr bool FWD = decltype(fwd)::value;
        const uint32_t nb = dir_neighbour<MU, FWD>(p, i, xh, y, z, t);
        cx<float> U[3][3], v[12];
        const auto n = SIn::load(in, p.vh, nb, v);
        Lk::load(p.gauge + (2 * MU + (FWD ? p.out_parity : p.out_parity ^ 1)) * p.gauge_pb, p.vh,
                 FWD ? (uint32_t)i : nb, U);
        dir_chi<MU, FWD, S0>(U, v, n, sh.chi + (2 * MU + !FWD) * 192 + lane);
    };
    auto both = [&](auto mu) {
        dir(mu, std::true_type());
        dir(mu, std::false_type());
    };
    switch (w) {
    case 0: both(std::integral_constant<int, 0>()); break;
    case 1: both(std::integral_constant<int, 1>()); break;
    case 2: both(std::integral_constant<int, 2>()); break;
    default: both(std::integral_constant<int, 3>()); break;
    }
    float2 xv[4];
    if (Axpy && w < 3) {
        const float2 *x = reinterpret_cast<const float2 *>(static_cast<const char *>(p.x) + (MULTI ? r * p.x_stride : 0)) +
                          (long long)w * p.vh;
#pragma unroll
        for (int k = 0; k < 4; ++k) xv[k] = ld_keep(at(x + 3ll * k * p.vh, (uint32_t)i));
    }
    __syncthreads();
    pdl_next();
    if (w < 3)
        finish_site<SOut, Dag, Axpy>(p, static_cast<char *>(p.out) + (MULTI ? r * p.out_stride : 0),
                                     sh.chi + 32 * w + lane, w, lane, (uint32_t)i, valid, xv, sh.mx, sh.wd);
}

// MINB: resident CTAs per SM that the registers are held to
// MULTI: several right-hand sides, which vary fastest in the grid, so that the
// CTAs that read the same links run side by side
template <class SIn, class SOut, class SX, class Lk, bool Dag, bool Axpy, int MINB, bool MULTI>
__global__ void __launch_bounds__(128, MINB) hop_kernel_dirs(const HopParams p)
{
    __shared__ DirsShared<Is16<SOut>::value> sh;
    pdl_wait();
    const int r = MULTI ? (int)blockIdx.x % p.nrhs : 0;
    int b = MULTI ? (int)blockIdx.x / p.nrhs : (int)blockIdx.x;
    if (p.reverse) b = (MULTI ? (p.vh + 31) / 32 : (int)gridDim.x) - 1 - b;
    dirs_block<SIn, SOut, SX, Lk, Dag, Axpy, MULTI>(p, b, r, sh);
}

// FP64: warp mu of a 128-thread CTA takes the pair of directions +-mu of 32
// sites (hop_pair); three warps then add the four pairs, one colour each.
template <class Lk, bool Dag, bool Axpy>
__device__ __forceinline__ void pairs_block(const HopParams &p, int b, int r, double2 *part)
{
    constexpr int S0 = Dag ? -1 : 1;
    const int lane = (int)threadIdx.x & 31, w = warp_id();
    const int i_raw = b * 32 + lane;
    const bool valid = i_raw < p.vh;
    const int i = valid ? i_raw : p.vh - 1;
    int xh, y, z;
    const int t = p.dz.div(p.dy.div(p.dx.div(i, xh), y), z);
    const char *in = static_cast<const char *>(p.in) + r * p.in_stride;
    auto pair = [&](auto mu) {
        constexpr int MU = decltype(mu)::value;
        cx<double> sum[2][3], dif[2][3];
        hop_pair<SpF64, Lk, MU, S0>(p, in, dir_neighbour<MU, true>(p, i, xh, y, z, t),
                                    dir_neighbour<MU, false>(p, i, xh, y, z, t), (uint32_t)i, sum, dif);
        double2 *o = part + MU * 12 * 32 + lane;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            o[32 * k] = make_double2(sum[k / 3][k % 3].r, sum[k / 3][k % 3].i);
            o[32 * (6 + k)] = make_double2(dif[k / 3][k % 3].r, dif[k / 3][k % 3].i);
        }
    };
    switch (w) {
    case 0: pair(std::integral_constant<int, 0>()); break;
    case 1: pair(std::integral_constant<int, 1>()); break;
    case 2: pair(std::integral_constant<int, 2>()); break;
    default: pair(std::integral_constant<int, 3>()); break;
    }
    double2 xv[4];
    if (Axpy && w < 3) {
        const double2 *x = reinterpret_cast<const double2 *>(static_cast<const char *>(p.x) + r * p.x_stride) + (long long)w * p.vh;
#pragma unroll
        for (int k = 0; k < 4; ++k) xv[k] = ld_keep(at(x + 3ll * k * p.vh, (uint32_t)i));
    }
    __syncthreads();
    if (w >= 3 || !valid) return;
    cx<double> o[4];
    auto add = [&](auto mu) {
        constexpr int MU = decltype(mu)::value;
        const double2 *q = part + MU * 12 * 32 + lane + 32 * w;
        const double2 s0 = q[0], s1 = q[32 * 3], d0 = q[32 * 6], d1 = q[32 * 9];
        reconstruct_pair<MU, S0>(o[0], o[1], o[2], o[3], cx<double>{s0.x, s0.y}, cx<double>{s1.x, s1.y},
                                 cx<double>{d0.x, d0.y}, cx<double>{d1.x, d1.y});
    };
    add(std::integral_constant<int, 0>());
    add(std::integral_constant<int, 1>());
    add(std::integral_constant<int, 2>());
    add(std::integral_constant<int, 3>());
    if (Axpy) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            o[k].r = fma(p.a, o[k].r, xv[k].x);
            o[k].i = fma(p.a, o[k].i, xv[k].y);
        }
    }
    double2 *q = reinterpret_cast<double2 *>(static_cast<char *>(p.out) + r * p.out_stride) + (long long)w * p.vh;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        *const_cast<double2 *>(at(q + 3ll * k * p.vh, (uint32_t)i)) = make_double2(o[k].r, o[k].i);
}

template <class Lk, bool Dag, bool Axpy>
__global__ void __launch_bounds__(128, 3) hop_kernel_pairs(const HopParams p)
{
    __shared__ double2 part[4 * 12 * 32];
    pdl_wait();
    const int r = (int)blockIdx.x % p.nrhs;
    int b = (int)blockIdx.x / p.nrhs;
    if (p.reverse) b = (p.vh + 31) / 32 - 1 - b;
    pairs_block<Lk, Dag, Axpy>(p, b, r, part);
}

// FP64: a 128-thread CTA takes 16 sites; warp mu of it the forward and backward
// hop of direction mu (as hop_pair), lanes 0..15 the first spin row of the
// projected spinors, lanes 16..31 the second.
template <int MU, int S0>
__device__ __forceinline__ void pair_rows(const HopParams &p, const char *in, const cx<double> Uf[3][3],
                                          const cx<double> Ub[3][3], uint32_t nf, uint32_t nbk, int row,
                                          double2 *part)
{
    constexpr bool kRot = MU == 0 || MU == 2;           // unit factor +-i or +-1
    const int partner = MU < 2 ? 3 - row : 2 + row;     // spin added to row `row`
    // h_row = psi_row + sg u psi_partner, u = i or 1 (project<MU, S>)
    const double sg = (double)((MU == 3 ? -S0 : S0) * ((MU == 1 || MU == 2) && row ? -1 : 1));
    const double2 *a = reinterpret_cast<const double2 *>(in) + 3ll * row * p.vh;
    const double2 *b = reinterpret_cast<const double2 *>(in) + 3ll * partner * p.vh;
    cx<double> h[3], g[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double2 u = ld_keep(at(a + (long long)c * p.vh, nf)), v = ld_keep(at(b + (long long)c * p.vh, nf));
        h[c] = kRot ? cx<double>{fma(-sg, v.y, u.x), fma(sg, v.x, u.y)} : cx<double>{fma(sg, v.x, u.x), fma(sg, v.y, u.y)};
        const double2 s = ld_keep(at(a + (long long)c * p.vh, nbk)), t = ld_keep(at(b + (long long)c * p.vh, nbk));
        g[c] = kRot ? cx<double>{fma(sg, t.y, s.x), fma(-sg, t.x, s.y)} : cx<double>{fma(-sg, t.x, s.x), fma(-sg, t.y, s.y)};
    }
    // the lower spin row that (P - Q)_row goes to, and its unit factor -S A^dag
    const int down = MU < 2 ? 3 - row : 2 + row;
    const bool neg = MU == 0 || MU == 3 ? S0 > 0 : (S0 > 0) == (MU == 1 ? row == 1 : row == 0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        cx<double> P = {0.0, 0.0};
#pragma unroll
        for (int c = 0; c < 3; ++c) P = cfma(Uf[k][c], h[c], P);
        cx<double> Q = {0.0, 0.0};
#pragma unroll
        for (int c = 0; c < 3; ++c) Q = cfmaconj(Ub[c][k], g[c], Q);
        const cx<double> z = cadd(P, Q), d = csub(P, Q);
        part[16 * (3 * row + k)] = make_double2(z.r, z.i);
        cx<double> l = kRot ? cmuli(d) : d;
        if (neg) l = cneg(l);
        part[16 * (3 * down + k)] = make_double2(l.r, l.i);
    }
}

template <class Lk, bool Dag, bool Axpy>
__global__ void __launch_bounds__(128, 4) hop_kernel_rows(const HopParams p)
{
    constexpr int S0 = Dag ? -1 : 1;
    __shared__ double2 part[4][12 * 16];
    pdl_wait();
    const int lane = (int)threadIdx.x & 31, w = warp_id();
    const int r = (int)blockIdx.x % p.nrhs;
    int b = (int)blockIdx.x / p.nrhs;
    if (p.reverse) b = (p.vh + 15) / 16 - 1 - b;
    const int s = lane & 15, row = lane >> 4;
    const int i_raw = b * 16 + s;
    const bool valid = i_raw < p.vh;
    const int i = valid ? i_raw : p.vh - 1;
    const uint32_t nf = neighbour_of(p, 2 * w, i), nbk = neighbour_of(p, 2 * w + 1, i);
    const char *in = static_cast<const char *>(p.in) + r * p.in_stride;
    cx<double> Uf[3][3], Ub[3][3];
    Lk::load(p.gauge + (2 * w + p.out_parity) * p.gauge_pb, p.vh, (uint32_t)i, Uf);
    Lk::load(p.gauge + (2 * w + (p.out_parity ^ 1)) * p.gauge_pb, p.vh, nbk, Ub);
    double2 *o = part[w] + s;
    switch (w) {
    case 0: pair_rows<0, S0>(p, in, Uf, Ub, nf, nbk, row, o); break;
    case 1: pair_rows<1, S0>(p, in, Uf, Ub, nf, nbk, row, o); break;
    case 2: pair_rows<2, S0>(p, in, Uf, Ub, nf, nbk, row, o); break;
    default: pair_rows<3, S0>(p, in, Uf, Ub, nf, nbk, row, o); break;
    }
    __syncthreads();
    pdl_next();
    // 12 spin-colour components x 16 sites over four warps, the last four over two
    for (int k = 2 * w + row; k < 12; k += 8) {
        double2 xv = make_double2(0.0, 0.0);
        if (Axpy)
            xv = ld_keep(at(reinterpret_cast<const double2 *>(static_cast<const char *>(p.x) + r * p.x_stride) + (long long)k * p.vh, (uint32_t)i));
        double2 acc = part[0][16 * k + s];
#pragma unroll
        for (int m = 1; m < 4; ++m) {
            const double2 v = part[m][16 * k + s];
            acc.x += v.x;
            acc.y += v.y;
        }
        if (Axpy) {
            acc.x = fma(p.a, acc.x, xv.x);
            acc.y = fma(p.a, acc.y, xv.y);
        }
        double2 *q = reinterpret_cast<double2 *>(static_cast<char *>(p.out) + r * p.out_stride) + (long long)k * p.vh;
        if (valid) *const_cast<double2 *>(at(q, (uint32_t)i)) = acc;
    }
}

}  // namespace weo
