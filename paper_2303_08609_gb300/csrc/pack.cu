// Gauge packing (canonical lexicographic AoS -> per-(mu, parity) planar formats),
// device buffers and error reporting.
#include <stdio.h>

#include <string>
#include <type_traits>

#include "weo_internal.h"

namespace weo {

// ------------------------------------------------------------------ errors --

static thread_local std::string g_last_error;

int set_error(int status, const std::string &msg)
{
    g_last_error = msg;
    return status;
}

const char *last_error_message() { return g_last_error.c_str(); }

int fail_cuda(cudaError_t e, const char *what, const char *file, int line)
{
    char buf[512];
    snprintf(buf, sizeof(buf), "%s failed: %s (%s) at %s:%d", what, cudaGetErrorName(e),
             cudaGetErrorString(e), file, line);
    (void)cudaGetLastError();  // clear a non-sticky error so later calls can proceed
    return set_error(e == cudaErrorMemoryAllocation ? WEO_ERR_OOM : WEO_ERR_CUDA, buf);
}

// ----------------------------------------------------------------- buffers --

int Buffer::ensure(size_t n)
{
    if (n <= bytes && ptr) return WEO_OK;
    release();
    if (n == 0) return WEO_OK;
    cudaError_t e = cudaMalloc(&ptr, n);
    if (e != cudaSuccess) {
        ptr = nullptr;
        bytes = 0;
        return fail_cuda(e, "cudaMalloc", __FILE__, __LINE__);
    }
    bytes = n;
    return WEO_OK;
}

void Buffer::release()
{
    if (ptr) cudaFree(ptr);
    ptr = nullptr;
    bytes = 0;
}

// ----------------------------------------------------------------- packing --

// A CTA takes the links of one direction based at 128 consecutive sites: it reads
// their contiguous 3x3 matrices as 16-byte vectors, writes the handle's canonical
// copy of them on the way (copy, may be null), and stores each parity's links as
// contiguous planes. One thread per link read 72-byte records at their stride, after
// a separate copy: set_gauge at 24^3 x 48 (FP32) took 58 + 66 us, now 83 us for
// 573 MB of traffic (6.9 TB/s).
constexpr int kPackSites = 128;

template <class Lk, typename In>
__global__ void __launch_bounds__(kPackSites) pack_gauge_kernel(const In *__restrict__ src, In *__restrict__ copy,
                                                                char *__restrict__ out, long long pb, unsigned lx,
                                                                unsigned ly, unsigned lz, long long V)
{
    using V4 = typename std::conditional<sizeof(In) == 4, float4, double2>::type;
    constexpr int kPer = 16 / sizeof(In);
    __shared__ __align__(16) In sh[18 * kPackSites];
    const int mu = (int)blockIdx.y;
    const long long lex0 = blockIdx.x * (long long)kPackSites;
    const int n = (int)(V - lex0 < kPackSites ? V - lex0 : kPackSites);  // even
    const long long first = 18 * (mu * V + lex0);
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        const V4 *s4 = reinterpret_cast<const V4 *>(src + first);
        V4 *c4 = reinterpret_cast<V4 *>(copy + first);
        for (int k = threadIdx.x; k < 18 * n / kPer; k += kPackSites) {
            const V4 v = s4[k];
            reinterpret_cast<V4 *>(sh)[k] = v;
            if (copy) c4[k] = v;
        }
    } else {
        for (int k = threadIdx.x; k < 18 * n; k += kPackSites) {
            const In v = src[first + k];
            sh[k] = v;
            if (copy) copy[first + k] = v;
        }
    }
    __syncthreads();
    if ((int)threadIdx.x >= n) return;
    // the first n / 2 threads take the even sites, the others the odd ones: sites
    // 2 j and 2 j + 1 lie in one row and have one of each parity
    const int par = (int)threadIdx.x >= n / 2, j = (int)threadIdx.x - (par ? n / 2 : 0);
    const unsigned row = (unsigned)(lex0 + 2 * j) / lx;
    const unsigned y = row % ly, zt = row / ly;
    const int l = 2 * j + (int)((y + zt % lz + zt / lz + par) & 1u);
    cx<double> U[3][3];
#pragma unroll
    for (int k = 0; k < 9; ++k) U[k / 3][k % 3] = {double(sh[18 * l + 2 * k]), double(sh[18 * l + 2 * k + 1])};
    Lk::store(out + (2 * mu + par) * pb, V / 2, (lex0 >> 1) + j, U);
}

template <class Lk>
static int pack_with(PackedGauge &g, const wilson_eo_s *h, const void *src, void *copy, int is_f64, cudaStream_t s)
{
    const long long V = 2 * h->vh;
    const dim3 grid((unsigned)((V + kPackSites - 1) / kPackSites), 4);
    char *out = static_cast<char *>(g.buf.ptr);
    const unsigned lx = h->dims[0], ly = h->dims[1], lz = h->dims[2];
    if (is_f64)
        pack_gauge_kernel<Lk, double><<<grid, kPackSites, 0, s>>>(static_cast<const double *>(src),
                                                                  static_cast<double *>(copy), out, g.pb, lx, ly, lz, V);
    else
        pack_gauge_kernel<Lk, float><<<grid, kPackSites, 0, s>>>(static_cast<const float *>(src),
                                                                 static_cast<float *>(copy), out, g.pb, lx, ly, lz, V);
    WEO_CUDA(cudaGetLastError());
    return WEO_OK;
}

int pack_gauge(wilson_eo_s *h, PackedGauge &g, int prec, int fmt, const void *canon, int is_f64,
               cudaStream_t s, void *copy)
{
    g.valid = false;
    g.prec = prec;
    g.fmt = fmt;
    g.pb = h->vh * link_site_bytes(prec, fmt);
    WEO_TRY(g.buf.ensure((size_t)(8 * g.pb)));
    const bool c = fmt == WEO_LINK12;
    int st;
    switch (prec) {
    case WEO_F64: st = c ? pack_with<LkF64_12>(g, h, canon, copy, is_f64, s) : pack_with<LkF64_18>(g, h, canon, copy, is_f64, s); break;
    case WEO_F32: st = c ? pack_with<LkF32_12>(g, h, canon, copy, is_f64, s) : pack_with<LkF32_18>(g, h, canon, copy, is_f64, s); break;
    case WEO_F16: st = c ? pack_with<LkH16_12>(g, h, canon, copy, is_f64, s) : pack_with<LkH16_18>(g, h, canon, copy, is_f64, s); break;
    case WEO_BF16: st = c ? pack_with<LkB16_12>(g, h, canon, copy, is_f64, s) : pack_with<LkB16_18>(g, h, canon, copy, is_f64, s); break;
    case kPrecFF: st = pack_with<LkFF18>(g, h, canon, copy, is_f64, s); break;
    default: return set_error(WEO_ERR_ARG, "unknown precision");
    }
    if (st == WEO_OK) {
        g.valid = true;
        ++g.gen;
    }
    return st;
}

int launch_hop(int prec, int fmt, int io, bool dag, bool axpy, const HopParams &p,
               const LaunchCfg &cfg, cudaStream_t s)
{
    if (p.vh == 0 || p.nrhs == 0) return WEO_OK;
    switch (prec) {
    case WEO_F64: return launch_hop_f64(fmt, dag, axpy, p, cfg, s);
    case WEO_F32: return launch_hop_f32(fmt, dag, axpy, p, cfg, s);
    case WEO_F16: return launch_hop_h16(fmt, io, dag, axpy, p, cfg, s);
    case WEO_BF16: return launch_hop_b16(fmt, io, dag, axpy, p, cfg, s);
    case kPrecFF: return launch_hop_ff(dag, axpy, p, cfg, s);
    default: return set_error(WEO_ERR_ARG, "unknown precision");
    }
}

}  // namespace weo
