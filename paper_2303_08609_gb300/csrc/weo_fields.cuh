// Device-side storage formats of spinor and link fields, and complex helpers.
//
// Spinor formats (one parity, one right-hand side; site index i = lex/2):
//   SpF64  [12][vh] double2   planar complex128 (the canonical FP64 layout)
//   SpF32  [12][vh] float2    planar complex64  (the canonical FP32 layout)
//   SpH16  [3][vh] uint4 + [vh] float   16-bit values scaled by a per-site norm:
//          uint4 plane q holds spin-colour components 4q..4q+3 as half2 (re, im);
//          norm[i] = max |real or imaginary part| over the site's 24 reals
//   SpB16  like SpH16 with bfloat16 values
// Link formats (one direction mu, one base-site parity; 3x3 complex per site):
//   LkF64_18 [9][vh] double2            row-major U_ab
//   LkF64_12 [6][vh] double2            rows 0, 1; row 2 = conj(row0 x row1)
//   LkF32_18 [4][vh] float4 + [vh] float2
//   LkF32_12 [3][vh] float4
//   LkH16_18 [2][vh] uint4 + [vh] uint32 (half2 per complex)
//   LkH16_12 [vh] uint4 + [vh] uint2
//   LkB16_*  like LkH16_* with bfloat16
// Every plane starts on a 16-byte boundary because vh = V/2 is a multiple of 8.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace weo {

template <typename T>
struct cx {
    T r, i;
};

// ---------------------------------------------------------- float-float --
// A float-float number hi + lo (|lo| <= half an ulp of hi) carries about 48
// significant bits, enough for FP64-class accuracy, with FP32 arithmetic only
// (double-float arithmetic as in Dekker 1971). On GB300 the FP32 pipes issue 64
// times as many operations per cycle as the FP64 pipe.
struct ff {
    float hi, lo;
    ff() = default;
    __device__ explicit ff(double v) : hi(float(v)), lo(float(v - double(float(v)))) {}
};

// hi + lo as a double, correctly rounded, by integer arithmetic (conversions and
// additions of doubles would run on the FP64 pipe, at 1/64 of the FP32 rate); out
// of the range of the scale factor, and for infinities and NaN, by the FP64 pipe
__device__ __forceinline__ double ff_join(float hi, float lo)
{
    const uint32_t b = __float_as_uint(hi), E = (b >> 23) & 255u;
    if (E - 53u > 201u || fabsf(lo) > fabsf(hi)) return double(hi) + double(lo);
    // lo in units of the result's last place: 2^-52 of hi's binade, or of the one
    // below when hi is a power of two that lo reduces
    const uint32_t below = (b & 0x7fffffu) == 0 && (int)(b ^ __float_as_uint(lo)) < 0;
    const int L = __float2int_rn(lo * __uint_as_float((306u - E + below) << 23));
    const long long m = (((long long)(b & 0x7fffffffu) + (896ll << 23)) << 29) + ((int)b < 0 ? -L : L);
    return __longlong_as_double(m | ((long long)(b & 0x80000000u) << 32));
}

// d as hi + lo, the inverse of ff_join
__device__ __forceinline__ float2 ff_split(double d)
{
    const long long x = __double_as_longlong(d), a = x & 0x7fffffffffffffffll;
    const uint32_t E = (uint32_t)(a >> 52);
    if (E - 950u > 190u) {  // outside 2^-73 .. 2^117
        const float h = float(d);
        return make_float2(h, float(d - double(h)));
    }
    const long long hi = (a + (1ll << 28)) >> 29;  // rounded to 24 bits, exponent + 896
    const int r = (int)(a - (hi << 29));           // remainder in units of d's 2^-52
    const uint32_t s = (uint32_t)(x >> 32) & 0x80000000u;
    const float lo = __int2float_rn(r) * __uint_as_float((E - 948u) << 23);
    return make_float2(__uint_as_float((uint32_t)(hi - (896ll << 23)) | s), __uint_as_float(__float_as_uint(lo) ^ s));
}

template <typename T>
__device__ __forceinline__ cx<T> cadd(cx<T> a, cx<T> b) { return {a.r + b.r, a.i + b.i}; }
template <typename T>
__device__ __forceinline__ cx<T> csub(cx<T> a, cx<T> b) { return {a.r - b.r, a.i - b.i}; }
// i * a
template <typename T>
__device__ __forceinline__ cx<T> cmuli(cx<T> a) { return {-a.i, a.r}; }
template <typename T>
__device__ __forceinline__ cx<T> cneg(cx<T> a) { return {-a.r, -a.i}; }
// acc + a * b
template <typename T>
__device__ __forceinline__ cx<T> cfma(cx<T> a, cx<T> b, cx<T> acc)
{
    acc.r = fma(a.r, b.r, acc.r);
    acc.r = fma(-a.i, b.i, acc.r);
    acc.i = fma(a.r, b.i, acc.i);
    acc.i = fma(a.i, b.r, acc.i);
    return acc;
}
// acc + conj(a) * b
template <typename T>
__device__ __forceinline__ cx<T> cfmaconj(cx<T> a, cx<T> b, cx<T> acc)
{
    acc.r = fma(a.r, b.r, acc.r);
    acc.r = fma(a.i, b.i, acc.r);
    acc.i = fma(a.r, b.i, acc.i);
    acc.i = fma(-a.i, b.r, acc.i);
    return acc;
}
template <typename T>
__device__ __forceinline__ cx<T> cmul(cx<T> a, cx<T> b) { return cfma(a, b, cx<T>{0, 0}); }
template <typename T>
__device__ __forceinline__ cx<T> cconj(cx<T> a) { return {a.r, -a.i}; }
template <typename T>
__device__ __forceinline__ cx<T> cscale(cx<T> a, T s) { return {a.r * s, a.i * s}; }

// ------------------------------------------------------------ loads/stores --
// Spinor neighbour reads are re-used by up to eight output sites: loads cached in
// L1 and L2. Not the read-only path (__ldg): it is for memory that nobody writes
// while the kernel runs, and a hop launched as a programmatic dependent is resident
// while its predecessor still writes the spinor that it reads after pdl_wait; the
// batch's second hop reads what its first hop wrote in the same launch. Links are
// used once per pass: streaming loads (evict-first) so they do not push the spinor
// working set out of L2.

template <typename T>
__device__ __forceinline__ T ld_keep(const T *p) { return __ldca(p); }
template <typename T>
__device__ __forceinline__ T ld_stream(const T *p) { return __ldcs(p); }


// Load policies of the link fields. LdStream: the links are read once per pass
// (evict first). LdL2: another CTA reads the same links again shortly (the
// second hop of the fused M_eo): keep them in L2 at normal priority and skip L1.
struct LdStream {
    template <typename T>
    __device__ static __forceinline__ T ld(const T *p) { return __ldcs(p); }
};
struct LdL2 {
    template <typename T>
    __device__ static __forceinline__ T ld(const T *p) { return __ldcg(p); }
};

// Element i of a plane. With a 32-bit index the byte offset is formed in 32
// bits, so that a load is one instruction on a warp-uniform base (callers
// guarantee i * sizeof(T) < 2^32); with a 64-bit index it is ordinary pointer
// arithmetic.
template <typename T, typename I>
__device__ __forceinline__ const T *at(const T *plane, I i)
{
    if constexpr (std::is_same<I, uint32_t>::value)
        return reinterpret_cast<const T *>(reinterpret_cast<const char *>(plane) + i * (uint32_t)sizeof(T));
    else
        return plane + i;
}

// ---------------------------------------------------------------- spinors --
// load() returns the factor that the values still need: none, or the site's norm
// of the 16-bit formats, which the projection applies (project in weo_dslash.cuh).
struct NoScale {};

// (a + b) n and (a - b) n. With a norm n the value b n is rounded first and a n
// added to it in one fused operation, spelled out so that every kernel rounds
// alike: where a result is rounded to 16 bits again, another order of these
// operations moves single elements by a whole step of the format, 2^-8 of the
// site's norm with BF16. The 24 operations per direction are as many as the
// projection and a multiplication of its 12 results would take.
template <typename R>
__device__ __forceinline__ cx<R> cadd(cx<R> a, cx<R> b, NoScale) { return cadd(a, b); }
template <typename R>
__device__ __forceinline__ cx<R> csub(cx<R> a, cx<R> b, NoScale) { return csub(a, b); }
__device__ __forceinline__ cx<float> cadd(cx<float> a, cx<float> b, float n)
{
    return {fmaf(a.r, n, __fmul_rn(b.r, n)), fmaf(a.i, n, __fmul_rn(b.i, n))};
}
__device__ __forceinline__ cx<float> csub(cx<float> a, cx<float> b, float n)
{
    return {fmaf(a.r, n, -__fmul_rn(b.r, n)), fmaf(a.i, n, -__fmul_rn(b.i, n))};
}

struct SpF64 {
    using real = double;
    static constexpr int kBytesPerSite = 192;
    template <typename R, typename I>
    __device__ static __forceinline__ NoScale load(const void *base, long long vh, I i,
                                                cx<R> v[12])
    {
        const double2 *p = static_cast<const double2 *>(base);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            double2 d = ld_keep(at(p + k * vh, i));
            v[k] = {R(d.x), R(d.y)};
        }
        return NoScale();
    }
    template <typename R>
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<R> v[12])
    {
        double2 *p = static_cast<double2 *>(base);
#pragma unroll
        for (int k = 0; k < 12; ++k) p[k * vh + i] = make_double2(double(v[k].r), double(v[k].i));
    }
};

struct SpF32 {
    using real = float;
    static constexpr int kBytesPerSite = 96;
    template <typename R, typename I>
    __device__ static __forceinline__ NoScale load(const void *base, long long vh, I i,
                                                cx<R> v[12])
    {
        const float2 *p = static_cast<const float2 *>(base);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            float2 d = ld_keep(at(p + k * vh, i));
            v[k] = {R(d.x), R(d.y)};
        }
        return NoScale();
    }
    template <typename R>
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<R> v[12])
    {
        float2 *p = static_cast<float2 *>(base);
#pragma unroll
        for (int k = 0; k < 12; ++k) p[k * vh + i] = make_float2(float(v[k].r), float(v[k].i));
    }
};

struct H16Traits {
    using scalar2 = __half2;
    __device__ static __forceinline__ float2 to_f2(uint32_t u)
    {
        __half2 h = *reinterpret_cast<__half2 *>(&u);
        return __half22float2(h);
    }
    __device__ static __forceinline__ uint32_t from_f2(float a, float b)
    {
        __half2 h = __floats2half2_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    }
};

struct B16Traits {
    using scalar2 = __nv_bfloat162;
    __device__ static __forceinline__ float2 to_f2(uint32_t u)
    {
        __nv_bfloat162 h = *reinterpret_cast<__nv_bfloat162 *>(&u);
        return __bfloat1622float2(h);
    }
    __device__ static __forceinline__ uint32_t from_f2(float a, float b)
    {
        __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    }
};

// 16-bit spinor with per-site FP32 norm; Tr = H16Traits or B16Traits.
template <class Tr>
struct Sp16 {
    using real = float;
    static constexpr int kBytesPerSite = 52;
    template <typename R, typename I>
    __device__ static __forceinline__ float load(const void *base, long long vh, I i,
                                                cx<R> v[12])
    {
        const uint4 *p = static_cast<const uint4 *>(base);
        const float *nrm = reinterpret_cast<const float *>(p + 3 * vh);
        const float n = ld_keep(at(nrm, i));
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            uint4 w = ld_keep(at(p + q * vh, i));
            float2 a = Tr::to_f2(w.x), b = Tr::to_f2(w.y), c = Tr::to_f2(w.z), d = Tr::to_f2(w.w);
            v[4 * q + 0] = {R(a.x), R(a.y)};
            v[4 * q + 1] = {R(b.x), R(b.y)};
            v[4 * q + 2] = {R(c.x), R(c.y)};
            v[4 * q + 3] = {R(d.x), R(d.y)};
        }
        return n;
    }
    template <typename R>
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<R> v[12])
    {
        uint4 *p = static_cast<uint4 *>(base);
        float *nrm = reinterpret_cast<float *>(p + 3 * vh);
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 12; ++k) m = fmaxf(m, fmaxf(fabsf(float(v[k].r)), fabsf(float(v[k].i))));
        const float s = m > 0.f ? 1.0f / m : 0.f;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            uint4 w;
            w.x = Tr::from_f2(float(v[4 * q + 0].r) * s, float(v[4 * q + 0].i) * s);
            w.y = Tr::from_f2(float(v[4 * q + 1].r) * s, float(v[4 * q + 1].i) * s);
            w.z = Tr::from_f2(float(v[4 * q + 2].r) * s, float(v[4 * q + 2].i) * s);
            w.w = Tr::from_f2(float(v[4 * q + 3].r) * s, float(v[4 * q + 3].i) * s);
            p[q * vh + i] = w;
        }
        nrm[i] = m;
    }
};
using SpH16 = Sp16<H16Traits>;
using SpB16 = Sp16<B16Traits>;

// ------------------------------------------------------------------ links --

// conj(a b - c d) in eight operations, for the FP64 pipe
__device__ __forceinline__ cx<double> cross_conj(cx<double> a, cx<double> b, cx<double> c, cx<double> d)
{
    return {fma(c.i, d.i, fma(-c.r, d.r, fma(-a.i, b.i, __dmul_rn(a.r, b.r)))),
            fma(c.i, d.r, fma(c.r, d.i, fma(-a.i, b.r, __dmul_rn(-a.r, b.i))))};
}
// FP32, also under 16-bit storage: the two products rounded apart, then subtracted.
// The eight operations of the FP64 form round otherwise, which 16-bit results
// multiply (see cadd with a norm above).
__device__ __forceinline__ cx<float> cross_conj(cx<float> a, cx<float> b, cx<float> c, cx<float> d)
{
    return cconj(csub(cmul(a, b), cmul(c, d)));
}

template <typename R>
__device__ __forceinline__ void reconstruct_row2(cx<R> U[3][3])
{
    // row2 = conj(row0 x row1), exact for SU(3)
    U[2][0] = cross_conj(U[0][1], U[1][2], U[0][2], U[1][1]);
    U[2][1] = cross_conj(U[0][2], U[1][0], U[0][0], U[1][2]);
    U[2][2] = cross_conj(U[0][0], U[1][1], U[0][1], U[1][0]);
}

struct LkF64_18 {
    static constexpr int kBytesPerSite = 144;
    template <typename R, typename I>
    __device__ static __forceinline__ void load(const void *base, long long vh, I i,
                                                cx<R> U[3][3])
    {
        const double2 *p = static_cast<const double2 *>(base);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            double2 d = ld_stream(at(p + k * vh, i));
            U[k / 3][k % 3] = {R(d.x), R(d.y)};
        }
    }
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<double> U[3][3])
    {
        double2 *p = static_cast<double2 *>(base);
#pragma unroll
        for (int k = 0; k < 9; ++k) p[k * vh + i] = make_double2(U[k / 3][k % 3].r, U[k / 3][k % 3].i);
    }
};

struct LkF64_12 {
    static constexpr int kBytesPerSite = 96;
    template <typename R, typename I>
    __device__ static __forceinline__ void load(const void *base, long long vh, I i,
                                                cx<R> U[3][3])
    {
        const double2 *p = static_cast<const double2 *>(base);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            double2 d = ld_stream(at(p + k * vh, i));
            U[k / 3][k % 3] = {R(d.x), R(d.y)};
        }
        reconstruct_row2(U);
    }
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<double> U[3][3])
    {
        double2 *p = static_cast<double2 *>(base);
#pragma unroll
        for (int k = 0; k < 6; ++k) p[k * vh + i] = make_double2(U[k / 3][k % 3].r, U[k / 3][k % 3].i);
    }
};

template <class Ld = LdStream>
struct LkF32_18T {
    static constexpr int kBytesPerSite = 72;
    template <typename R, typename I>
    __device__ static __forceinline__ void load(const void *base, long long vh, I i,
                                                cx<R> U[3][3])
    {
        const float4 *p = static_cast<const float4 *>(base);
        float4 a = Ld::ld(at(p, i)), b = Ld::ld(at(p + vh, i)), c = Ld::ld(at(p + 2 * vh, i)),
               d = Ld::ld(at(p + 3 * vh, i));
        float2 e = Ld::ld(at(reinterpret_cast<const float2 *>(p + 4 * vh), i));
        U[0][0] = {R(a.x), R(a.y)};
        U[0][1] = {R(a.z), R(a.w)};
        U[0][2] = {R(b.x), R(b.y)};
        U[1][0] = {R(b.z), R(b.w)};
        U[1][1] = {R(c.x), R(c.y)};
        U[1][2] = {R(c.z), R(c.w)};
        U[2][0] = {R(d.x), R(d.y)};
        U[2][1] = {R(d.z), R(d.w)};
        U[2][2] = {R(e.x), R(e.y)};
    }
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<double> U[3][3])
    {
        float4 *p = static_cast<float4 *>(base);
        p[i] = make_float4(U[0][0].r, U[0][0].i, U[0][1].r, U[0][1].i);
        p[vh + i] = make_float4(U[0][2].r, U[0][2].i, U[1][0].r, U[1][0].i);
        p[2 * vh + i] = make_float4(U[1][1].r, U[1][1].i, U[1][2].r, U[1][2].i);
        p[3 * vh + i] = make_float4(U[2][0].r, U[2][0].i, U[2][1].r, U[2][1].i);
        reinterpret_cast<float2 *>(p + 4 * vh)[i] = make_float2(U[2][2].r, U[2][2].i);
    }
};

template <class Ld = LdStream>
struct LkF32_12T {
    static constexpr int kBytesPerSite = 48;
    template <typename R, typename I>
    __device__ static __forceinline__ void load(const void *base, long long vh, I i,
                                                cx<R> U[3][3])
    {
        const float4 *p = static_cast<const float4 *>(base);
        float4 a = Ld::ld(at(p, i)), b = Ld::ld(at(p + vh, i)), c = Ld::ld(at(p + 2 * vh, i));
        U[0][0] = {R(a.x), R(a.y)};
        U[0][1] = {R(a.z), R(a.w)};
        U[0][2] = {R(b.x), R(b.y)};
        U[1][0] = {R(b.z), R(b.w)};
        U[1][1] = {R(c.x), R(c.y)};
        U[1][2] = {R(c.z), R(c.w)};
        reconstruct_row2(U);
    }
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<double> U[3][3])
    {
        float4 *p = static_cast<float4 *>(base);
        p[i] = make_float4(U[0][0].r, U[0][0].i, U[0][1].r, U[0][1].i);
        p[vh + i] = make_float4(U[0][2].r, U[0][2].i, U[1][0].r, U[1][0].i);
        p[2 * vh + i] = make_float4(U[1][1].r, U[1][1].i, U[1][2].r, U[1][2].i);
    }
};

template <class Tr, class Ld = LdStream>
struct Lk16_18 {
    static constexpr int kBytesPerSite = 36;
    template <typename R, typename I>
    __device__ static __forceinline__ void load(const void *base, long long vh, I i,
                                                cx<R> U[3][3])
    {
        const uint4 *p = static_cast<const uint4 *>(base);
        uint4 a = Ld::ld(at(p, i)), b = Ld::ld(at(p + vh, i));
        uint32_t e = Ld::ld(at(reinterpret_cast<const unsigned int *>(p + 2 * vh), i));
        const uint32_t w[9] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, e};
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            float2 f = Tr::to_f2(w[k]);
            U[k / 3][k % 3] = {R(f.x), R(f.y)};
        }
    }
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<double> U[3][3])
    {
        uint32_t w[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) w[k] = Tr::from_f2(float(U[k / 3][k % 3].r), float(U[k / 3][k % 3].i));
        uint4 *p = static_cast<uint4 *>(base);
        p[i] = make_uint4(w[0], w[1], w[2], w[3]);
        p[vh + i] = make_uint4(w[4], w[5], w[6], w[7]);
        reinterpret_cast<unsigned int *>(p + 2 * vh)[i] = w[8];
    }
};

template <class Tr, class Ld = LdStream>
struct Lk16_12 {
    static constexpr int kBytesPerSite = 24;
    template <typename R, typename I>
    __device__ static __forceinline__ void load(const void *base, long long vh, I i,
                                                cx<R> U[3][3])
    {
        const uint4 *p = static_cast<const uint4 *>(base);
        uint4 a = Ld::ld(at(p, i));
        uint2 b = Ld::ld(at(reinterpret_cast<const uint2 *>(p + vh), i));
        const uint32_t w[6] = {a.x, a.y, a.z, a.w, b.x, b.y};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            float2 f = Tr::to_f2(w[k]);
            U[k / 3][k % 3] = {R(f.x), R(f.y)};
        }
        reconstruct_row2(U);
    }
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<double> U[3][3])
    {
        uint32_t w[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] = Tr::from_f2(float(U[k / 3][k % 3].r), float(U[k / 3][k % 3].i));
        uint4 *p = static_cast<uint4 *>(base);
        p[i] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint2 *>(p + vh)[i] = make_uint2(w[4], w[5]);
    }
};

// FP64-class links in float-float: the high parts in the LkF32_18 layout,
// then the low parts in the same layout (144 bytes per site, as FP64).
struct LkFF18 {
    static constexpr int kBytesPerSite = 144;
    __device__ static __forceinline__ void store(void *base, long long vh, long long i,
                                                 const cx<double> U[3][3])
    {
        cx<double> H[3][3], L[3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const ff r(U[a][b].r), m(U[a][b].i);
                H[a][b] = {double(r.hi), double(m.hi)};
                L[a][b] = {double(r.lo), double(m.lo)};
            }
        LkF32_18T<>::store(base, vh, i, H);
        LkF32_18T<>::store(static_cast<char *>(base) + 72 * vh, vh, i, L);
    }
};

using LkF32_18 = LkF32_18T<>;
using LkF32_12 = LkF32_12T<>;
using LkH16_18 = Lk16_18<H16Traits>;
using LkH16_12 = Lk16_12<H16Traits>;
using LkB16_18 = Lk16_18<B16Traits>;
using LkB16_12 = Lk16_12<B16Traits>;

}  // namespace weo
