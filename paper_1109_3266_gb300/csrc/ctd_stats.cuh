// ctd_stats.cuh -- device parts of the precision measures (Sec. 3.1) shared by the
// statistics kernels and the allocation-free entry point: the mean of s/D over
// D > 0.1 D_max and the sum of s over D > 0.2 D_max, inside rho >= 0.1 g/cm^3.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

#include "ctd_internal.h"

namespace ctd {
namespace stats {

constexpr int kThreads = 256;
constexpr int kMaxStatBlocks = 152 * 8;   // resident blocks of 256 threads
constexpr int kPerThread = 4;             // voxels a thread holds in flight

static_assert(kPartialCells == 6 * kMaxStatBlocks, "six partials per block");

inline int stat_blocks(size_t n, int per_thread)
{
    const size_t per_block = static_cast<size_t>(kThreads) * per_thread;
    const size_t g = (n + per_block - 1) / per_block;
    return static_cast<int>(g < 1 ? 1 : g > kMaxStatBlocks ? kMaxStatBlocks : g);
}

// 1/x for a positive normal x: the hardware's approximate reciprocal (relative
// error below 2^-22) and two Newton-Raphson steps y <- y + y (1 - x y), each of
// which squares the relative error, so the result is within an ulp or two of 1/x.
__device__ __forceinline__ double recip(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double e = fma(-x, y, 1.0);
    y = fma(y, e, y);
    e = fma(-x, y, 1.0);
    return fma(y, e, y);
}

// sqrt(x) for finite x >= 2^-1000: Goldschmidt's coupled iteration for sqrt and
// 1/(2 sqrt) from the hardware's approximate reciprocal square root, then one correction
// by the residual x - g^2 (Markstein, IBM J. Res. Dev. 34, 1990).  With an approximation
// within 2^-20 the iteration leaves relative errors near 2^-39 in g and h, so what the
// correction rounds is within 2^-77 of sqrt(x): the nearest double but where sqrt(x) lies
// that close to the middle of two.
__device__ __forceinline__ double root(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double g = x * y, h = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));   // y / 2
    const double r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    h = fma(h, r, h);
    return fma(fma(-g, g, x), h, g);
}

// A non-negative double's bits order like its value; negative numbers come below
// every one of them and NaNs above infinity.
constexpr long long kInfBits = 0x7ff0000000000000ll;

__device__ __forceinline__ long long max_dose(long long m, double dose)
{
    const long long b = __double_as_longlong(dose);
    return b > m && b <= kInfBits ? b : m;
}

__device__ __forceinline__ long long warp_max(long long m)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m ? y : m;
    }
    return m;
}

// block-wide maximum, in every thread
__device__ __forceinline__ long long block_max(long long m)
{
    __shared__ long long sh[kThreads / 32];
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    m = warp_max(sh[threadIdx.x & (kThreads / 32 - 1)]);
    __syncthreads();
    return m;
}

// maximum of n bit patterns written by an earlier kernel, in every thread
__device__ __forceinline__ long long max_of(const long long *p, int n)
{
    long long m = 0;
    for (int i = threadIdx.x; i < n; i += kThreads) m = p[i] > m ? p[i] : m;
    return block_max(m);
}

// block-wide sums of K doubles, in thread 0
template <int K>
__device__ __forceinline__ void block_sum(double (&x)[K])
{
    __shared__ double sh[K][kThreads / 32];
#pragma unroll
    for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x[k] += __shfl_down_sync(0xffffffffu, x[k], o);
        if ((threadIdx.x & 31) == 0) sh[k][threadIdx.x >> 5] = x[k];
    }
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            x[k] = 0.0;
            for (int w = 0; w < kThreads / 32; ++w) x[k] += sh[k][w];
        }
    __syncthreads();
}

// One block's partial sums of the precision measures, to sums[4][stride] at this
// block's place: s/D and its count over D > 0.1 D_max, s and its count over
// D > 0.2 D_max.
//
// GB300's FP64 pipe (about two multiply-adds per cycle and SM), not memory, bounds
// a division per voxel.  Four quotients share one reciprocal: s0/D0 + s1/D1 =
// (s0 D1 + s1 D0) / (D0 D1), and again for two such pairs, 3.5 FP64 operations a
// voxel instead of 6 with a reciprocal each.  The doses are first scaled by a power
// of two (on their exponent bits, exactly) that takes D_max to [2^-4, 2^-3), so products
// of doses stay in range; those with an error, down to 2^-22 of it, do while the error is
// above 2^-1000.  D_max outside [2^-500, 2^500] divides voxel by voxel: inside, a smaller
// error is below 2^-490 of its dose.
__device__ __forceinline__ void rsd_sums(const double *__restrict__ dose, const double *__restrict__ sd,
                                         const float *__restrict__ rho, size_t nvox, double dmax, double *sums,
                                         int stride_out)
{
    const long long lo1 = __double_as_longlong(0.1 * dmax), lo2 = __double_as_longlong(0.2 * dmax);
    const bool scaled = dmax >= 0x1p-500 && dmax <= 0x1p500;
    const int shift = (__double2hiint(dmax) & 0x7ff00000) - ((1023 - 4) << 20);
    double rel = 0.0, s2 = 0.0;
    unsigned n1 = 0, n2 = 0;
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    for (size_t v0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x; v0 < nvox; v0 += kPerThread * stride) {
        float r[kPerThread];
        double d[kPerThread], s[kPerThread];
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) {
            const size_t v = v0 + k * stride;
            r[k] = v < nvox ? rho[v] : 0.0f;
            d[k] = v < nvox ? dose[v] : 0.0;
        }
        bool any = false;
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) {
            const long long b = __double_as_longlong(d[k]);
            const bool in1 = r[k] >= 0.1f && b > lo1 && b <= kInfBits, in2 = in1 && b > lo2;
            s[k] = in1 ? sd[v0 + k * stride] : 0.0;
            if (in2) s2 += s[k];
            n1 += in1;
            n2 += in2;
            any |= in1;
            // (a voxel outside the mask adds 0/1)
            const double x = scaled ? __hiloint2double(__double2hiint(d[k]) - shift, __double2loint(d[k])) : d[k];
            d[k] = in1 ? x : 1.0;
        }
        if (!any) continue;
        if (scaled) {
            const double n01 = fma(s[0], d[1], s[1] * d[0]), d01 = d[0] * d[1];
            const double n23 = fma(s[2], d[3], s[3] * d[2]), d23 = d[2] * d[3];
            rel = fma(fma(n01, d23, n23 * d01), recip(d01 * d23), rel);
        } else {
#pragma unroll
            for (int k = 0; k < kPerThread; ++k) rel += s[k] / d[k];
        }
    }
    // s/D of a scaled dose D' = D 2^-e is s/D' 2^-e
    if (scaled) rel *= __hiloint2double((1023 << 20) - shift, 0);
    double x[2] = {rel, s2};
    block_sum<2>(x);
    const unsigned w1 = __reduce_add_sync(0xffffffffu, n1), w2 = __reduce_add_sync(0xffffffffu, n2);
    __shared__ unsigned sh[2][kThreads / 32];
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = w1;
        sh[1][threadIdx.x >> 5] = w2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned c1 = 0, c2 = 0;
        for (int w = 0; w < kThreads / 32; ++w) {
            c1 += sh[0][w];
            c2 += sh[1][w];
        }
        sums[blockIdx.x] = x[0];
        sums[stride_out + blockIdx.x] = c1;
        sums[2 * stride_out + blockIdx.x] = x[1];
        sums[3 * stride_out + blockIdx.x] = c2;
    }
}

// Whether this block is the grid's last to get here; it then sees what every block
// wrote before.  `done` counts from 0 and is left at 0.
__device__ __forceinline__ bool last_block(unsigned *done)
{
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(done, 1u) == gridDim.x - 1;
        if (last) *done = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Sum of n partials in a fixed order by the block, in thread 0.
__device__ __forceinline__ double total_of(const double *p, int n)
{
    double x[1] = {0.0};
    for (int i = threadIdx.x; i < n; i += kThreads) x[0] += __ldcg(p + i);
    block_sum<1>(x);
    return x[0];
}

// result[0..2] = avg RSD, sigma-bar, D_max from n blocks' partial sums, and with extra
// partials (n_extra of them) result[3] = their sum; the sums are reduced side by side
template <bool kExtra>
__device__ __forceinline__ void rsd_result(const double *sums, int stride, int n, double dmax, const double *extra,
                                           int n_extra, double *result)
{
    double s[kExtra ? 5 : 4] = {};
    for (int i = threadIdx.x; i < n; i += kThreads)
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] += __ldcg(sums + k * stride + i);
    if (kExtra)
        for (int i = threadIdx.x; i < n_extra; i += kThreads) s[kExtra ? 4 : 0] += __ldcg(extra + i);
    block_sum<kExtra ? 5 : 4>(s);
    if (threadIdx.x == 0) {
        result[0] = s[1] > 0.0 ? s[0] / s[1] : 0.0;
        result[1] = (s[3] > 0.0 && dmax > 0.0) ? s[2] / (s[3] * dmax) : 0.0;
        result[2] = dmax;
        if (kExtra) result[3] = s[kExtra ? 4 : 0];
    }
}

}  // namespace stats
}  // namespace ctd
