// Float-float operator support: conversions between canonical complex128
// spinors and the SpFF layout, and the lazily packed float-float gauge field.
#include "weo_internal.h"

namespace weo {

// src: nrhs x [12][vh] double2 ; dst: nrhs x ([12][vh] float2 high parts, [12][vh] low parts).
// One right-hand side per blockIdx.y; ff_split keeps it off the FP64 pipe.
constexpr int kSplitPer = 4;  // values per thread, all loads in flight together
__global__ void __launch_bounds__(256) k_f64_to_ff(float2 *__restrict__ dst, const double2 *__restrict__ src, long long per)
{
    const long long k0 = blockIdx.x * (256ll * kSplitPer) + threadIdx.x;
    const double2 *s = src + blockIdx.y * per;
    float2 *d = dst + blockIdx.y * 2 * per;
    double2 v[kSplitPer];
#pragma unroll
    for (int j = 0; j < kSplitPer; ++j)
        if (k0 + 256 * j < per) v[j] = __ldcs(s + k0 + 256 * j);
#pragma unroll
    for (int j = 0; j < kSplitPer; ++j) {
        const long long k = k0 + 256 * j;
        if (k >= per) break;
        const float2 a = ff_split(v[j].x), b = ff_split(v[j].y);
        d[k] = make_float2(a.x, b.x);
        d[per + k] = make_float2(a.y, b.y);
    }
}

int ff_from_f64(void *dst, const void *src, long long vh, int nrhs, cudaStream_t s)
{
    const long long per = 12 * vh;
    const unsigned blocks = (unsigned)((per + 256 * kSplitPer - 1) / (256 * kSplitPer));
    for (long long r = 0; r < nrhs; r += kGridRows) {
        const dim3 grid(blocks, (unsigned)(nrhs - r < kGridRows ? nrhs - r : kGridRows));
        k_f64_to_ff<<<grid, 256, 0, s>>>(static_cast<float2 *>(dst) + r * 2 * per,
                                         static_cast<const double2 *>(src) + r * per, per);
        WEO_CUDA(cudaGetLastError());
    }
    return WEO_OK;
}

int ff_gauge(wilson_eo_s *h, const PackedGauge **g, cudaStream_t s)
{
    if (!h->gauge_ff.valid)
        WEO_TRY(pack_gauge(h, h->gauge_ff, kPrecFF, WEO_LINK18, h->canon_gauge.ptr, h->canon_is_f64, s));
    *g = &h->gauge_ff;
    return WEO_OK;
}

}  // namespace weo
