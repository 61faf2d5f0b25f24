// ctd_stats.cu -- batch statistics of the dose engine (Sec. 2.2.1) and the
// precision measures of Sec. 3.1, as streaming kernels over the FP64 grids.
#include <cuda_runtime.h>

#include "ctd_internal.h"
#include "ctd_stats.cuh"

namespace ctd {
namespace {

using namespace stats;

// GB300's binary64 pipe is narrow (about two multiply-adds per cycle and SM), so
// these kernels divide by nothing per voxel and keep the operations per batch and
// voxel few: the fold multiplies by the voxel's 1/rho (correctly rounded once, when
// the phantom is created) once for all batches, the mean and variance by 1/nb and
// 1/(nb (nb - 1)) from the host; quotients and roots: ctd_stats.cuh.

// Fold of one request's batch in the multi-request fold: d = E_b / (m_v n_b) in Gy per
// history; accumulate d and d^2, keep the raw energy, clear the tally.  rinv = 1 / rho
// (0 where rho = 0).
__device__ __forceinline__ void fold_voxel(double t, size_t v, double *__restrict__ tally,
                                           const double *__restrict__ rinv, double *__restrict__ sum_d,
                                           double *__restrict__ sum_d2, double *__restrict__ edep, double scale)
{
    const double d = (t * scale) * rinv[v];
    edep[v] += t;
    tally[v] = 0.0;
    sum_d[v] += d;
    sum_d2[v] += d * d;
}

// Mean over nb batches and its standard error: s^2 = (sum d^2 - nb D^2) / (nb (nb - 1)),
// nb D^2 as D sum d, with inv_nb = 1/nb and inv_nn = 1/(nb (nb - 1)).  (A comparison of
// doubles is FP64 work too: the variance's sign and size are read from its bits.  What is
// not a normal number above 2^-1000, such as an infinity or a NaN of tallies that are not
// finite, takes the comparison.)
__device__ __forceinline__ void mean_sd(double s1, double s2, double inv_nb, double inv_nn, double &D, double &sd)
{
    D = s1 * inv_nb;
    const double var = fma(-D, s1, s2) * inv_nn;
    const int hi = __double2hiint(var), lo = (1023 - 1000) << 20;
    sd = static_cast<unsigned>(hi - lo) < static_cast<unsigned>(0x7ff00000 - lo) ? root(var) : var > 0.0 ? sqrt(var) : 0.0;
}

// Fold of a request's batches in one pass, and with kLast the mean, the standard
// error and the blocks' partial maxima of the dose (inside rho >= 0.1) and sums of the
// deposited energy as well.  With d_b = w t_b (w = scale / rho) a batch costs two
// binary64 operations a voxel, sum t and sum t^2 (fused), and the weights are applied
// to the sums: sum d = w sum t, sum d^2 = w^2 sum t^2, for the larger and the smaller
// batches apart.  kFirst: the sums start here.  Bound by the binary64 pipe (about
// 2 nb + 15 operations) and by memory (8 bytes a batch and at most 84 once): 8.4 M voxels
// and ten batches 0.68 ms, where a fold per batch and a kernel for the mean took 1.49.
template <bool kFirst, bool kLast>
__global__ void __launch_bounds__(kThreads) fold_kernel(const FoldBatches f, const double *__restrict__ rinv,
                                                        double *__restrict__ sum_d, double *__restrict__ sum_d2,
                                                        double *__restrict__ edep, size_t nvox, const FoldLast last)
{
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    long long dmax = 0;
    double total[1] = {0.0};
    for (size_t v = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x; v < nvox; v += stride) {
        double t1[2] = {0.0, 0.0}, t2[2] = {0.0, 0.0};   // sum t and sum t^2 of either size of batch
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int hi = g == 0 ? f.n_first : f.nb;
            for (int b = g == 0 ? 0 : f.n_first; b < hi; b += kPerThread) {
                double t[kPerThread];
#pragma unroll
                for (int k = 0; k < kPerThread; ++k) t[k] = b + k < hi ? f.tally[(b + k) * nvox + v] : 0.0;
#pragma unroll
                for (int k = 0; k < kPerThread; ++k)
                    if (__double_as_longlong(t[k]) != 0) {
                        t1[g] += t[k];
                        t2[g] = fma(t[k], t[k], t2[g]);
                        if (f.clear) f.tally[(b + k) * nvox + v] = 0.0;
                    }
            }
        }
        double e = kFirst ? 0.0 : edep[v], s1 = kFirst ? 0.0 : sum_d[v], s2 = kFirst ? 0.0 : sum_d2[v];
        const double r = rinv[v];
        if (f.n_first > 0) {
            const double w = f.scale0 * r;
            e = kFirst ? t1[0] : e + t1[0];
            s1 = kFirst ? w * t1[0] : fma(w, t1[0], s1);
            s2 = kFirst ? (w * w) * t2[0] : fma(w * w, t2[0], s2);
        }
        if (f.n_first < f.nb) {
            const double w = f.scale1 * r;
            const bool start = kFirst && f.n_first == 0;
            e = start ? t1[1] : e + t1[1];
            s1 = fma(w, t1[1], s1);
            s2 = fma(w * w, t2[1], s2);
        }
        if (kFirst || f.nb > 0) edep[v] = e;
        if (!kLast || last.keep_sums) {
            sum_d[v] = s1;
            sum_d2[v] = s2;
        }
        if (kLast) {
            double D, s;
            mean_sd(s1, s2, last.inv_nb, last.inv_nn, D, s);
            last.dose[v] = D;
            last.sd[v] = s;
            if (last.rho[v] >= 0.1f) dmax = max_dose(dmax, D);
            total[0] += e;
        }
    }
    if (kLast) {
        dmax = block_max(dmax);
        block_sum<1>(total);
        if (threadIdx.x == 0) {
            reinterpret_cast<long long *>(last.partials)[blockIdx.x] = dmax;
            last.partials[kMaxStatBlocks + blockIdx.x] = total[0];
            if (blockIdx.x == 0) *reinterpret_cast<unsigned *>(last.partials + kPartialCells) = 0;
        }
    }
}

// The precision measures and the total deposit from the dose, its standard error and
// the partial maxima and sums n_fold blocks of fold_kernel left: result[0..3] = avg
// RSD, sigma-bar, D_max, total.  The last block to finish adds the blocks' sums up.
__global__ void __launch_bounds__(kThreads) rsd_kernel(const double *__restrict__ dose, const double *__restrict__ sd,
                                                       const float *__restrict__ rho, size_t nvox, double *partials,
                                                       int n_fold, double *result)
{
    const double dmax = __longlong_as_double(max_of(reinterpret_cast<const long long *>(partials), n_fold));
    double *sums = partials + 2 * kMaxStatBlocks;
    rsd_sums(dose, sd, rho, nvox, dmax, sums, kMaxStatBlocks);
    if (last_block(reinterpret_cast<unsigned *>(partials + kPartialCells)))
        rsd_result<true>(sums, kMaxStatBlocks, gridDim.x, dmax, partials + kMaxStatBlocks, n_fold, result);
}

// The same fold for several requests at once, one tile of kFoldTile voxels per step.
__global__ void fold_multi_kernel(const FoldDesc *__restrict__ descs, const uint64_t *__restrict__ tile_off, int n,
                                  uint64_t total_tiles)
{
    for (uint64_t tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tile_off[mid] <= tile) lo = mid;
            else hi = mid - 1;
        }
        const FoldDesc d = descs[lo];
        const uint64_t base = (tile - tile_off[lo]) * static_cast<uint64_t>(kFoldTile);
        const uint64_t end = base + kFoldTile < d.nvox ? base + kFoldTile : d.nvox;
        for (uint64_t v = base + threadIdx.x; v < end; v += blockDim.x) {
            const double t = d.tally[v];
            if (t != 0.0) fold_voxel(t, v, d.tally, d.rinv, d.sum_d, d.sum_d2, d.edep, d.scale);
        }
    }
}

// Sum of n doubles: blocks' partial sums, then one block's in a fixed order.
__global__ void __launch_bounds__(kThreads) sum_kernel(const double *__restrict__ x, size_t n, double *partials)
{
    double a[1] = {0.0};
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    for (size_t v0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x; v0 < n; v0 += kPerThread * stride) {
        double t[kPerThread];
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) t[k] = v0 + k * stride < n ? x[v0 + k * stride] : 0.0;
        a[0] += (t[0] + t[1]) + (t[2] + t[3]);
    }
    block_sum<1>(a);
    if (threadIdx.x == 0) partials[blockIdx.x] = a[0];
}

__global__ void __launch_bounds__(kThreads) sum_final_kernel(const double *partials, int n, double *result)
{
    const double s = total_of(partials, n);
    if (threadIdx.x == 0) *result = s;
}

// One pass over a new phantom's voxels (grid-stride): range checks and the
// per-material presence and largest density, reduced in shared memory, then one
// global atomic per block and quantity.  -0 densities count as +0.
__global__ void scan_phantom_kernel(const uint8_t *__restrict__ mat, const float *__restrict__ rho, size_t nvox,
                                    int n_mat, uint32_t *__restrict__ vox, double *__restrict__ rinv,
                                    PhantomScan *out)
{
    __shared__ unsigned int s_max[kMaxPhantomMaterials];
    __shared__ unsigned int s_mask;
    __shared__ unsigned long long s_bad_mat, s_bad_rho;
    if (threadIdx.x < kMaxPhantomMaterials) s_max[threadIdx.x] = 0u;
    if (threadIdx.x == 0) {
        s_mask = 0u;
        s_bad_mat = ~0ull;
        s_bad_rho = ~0ull;
    }
    __syncthreads();
    for (size_t v = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; v < nvox;
         v += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const int m = mat[v];
        const float r = rho[v];
        if (m >= n_mat) {
            atomicMin(&s_bad_mat, static_cast<unsigned long long>(v));
            continue;
        }
        const uint32_t f = __float_as_uint(r + 0.0f);   // -0 as +0
        const uint32_t ex = f >> 23;
        if (!(r >= 0.0f) || (f != 0u && (ex < kRhoExpLo || ex > kRhoExpHi))) {
            atomicMin(&s_bad_rho, static_cast<unsigned long long>(v));
            continue;
        }
        vox[v] = (static_cast<uint32_t>(m) << 28) | (f ? f - (kRhoExpBias << 23) : 0u);
        rinv[v] = f ? 1.0 / static_cast<double>(r) : 0.0;
        atomicMax(&s_max[m], f);
        atomicOr(&s_mask, 1u << m);
    }
    __syncthreads();
    if (threadIdx.x < n_mat && (s_mask >> threadIdx.x & 1u)) atomicMax(&out->max_bits[threadIdx.x], s_max[threadIdx.x]);
    if (threadIdx.x == 0) {
        if (s_mask) atomicOr(&out->present_mask, s_mask);
        if (s_bad_mat != ~0ull) atomicMin(&out->first_bad_mat, s_bad_mat);
        if (s_bad_rho != ~0ull) atomicMin(&out->first_bad_rho, s_bad_rho);
    }
}

// Angular surfaces [k][n_e][n_zeta] as cells [k][n_e - 1][n_zeta - 1] of float4: the
// corners S[j][i], S[j][i+1], S[j+1][i], S[j+1][i+1] of the bilinear lookup in cell
// (j, i).  One block per row of cells at a time; bound by the 16 bytes a cell written.
__global__ void cells_kernel(const float *__restrict__ rows, int n_rows, int n_e, int n_zeta, float4 *__restrict__ cells)
{
    for (int r = blockIdx.x; r < n_rows; r += gridDim.x) {
        const int m = r / (n_e - 1), j = r - m * (n_e - 1);
        const float *r0 = rows + (static_cast<size_t>(m) * n_e + j) * n_zeta, *r1 = r0 + n_zeta;
        float4 *out = cells + static_cast<size_t>(r) * (n_zeta - 1);
        for (int i = threadIdx.x; i + 1 < n_zeta; i += blockDim.x) out[i] = make_float4(r0[i], r0[i + 1], r1[i], r1[i + 1]);
    }
}

inline int ok() { return cudaGetLastError() == cudaSuccess ? CTD_OK : CTD_ECUDA; }

}  // namespace

int launch_fold(const FoldBatches &f, const double *rinv, double *sum_d, double *sum_d2, double *edep, size_t nvox,
                bool first, const FoldLast *last, void *stream)
{
    const int grid = stat_blocks(nvox, 1);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    FoldLast none{};
    const FoldLast &l = last ? *last : none;
    if (first && last) fold_kernel<true, true><<<grid, kThreads, 0, s>>>(f, rinv, sum_d, sum_d2, edep, nvox, l);
    else if (first) fold_kernel<true, false><<<grid, kThreads, 0, s>>>(f, rinv, sum_d, sum_d2, edep, nvox, l);
    else if (last) fold_kernel<false, true><<<grid, kThreads, 0, s>>>(f, rinv, sum_d, sum_d2, edep, nvox, l);
    else fold_kernel<false, false><<<grid, kThreads, 0, s>>>(f, rinv, sum_d, sum_d2, edep, nvox, l);
    return ok();
}

int launch_rsd(const FoldLast &l, size_t nvox, double *result, void *stream)
{
    rsd_kernel<<<stat_blocks(nvox, kPerThread), kThreads, 0, static_cast<cudaStream_t>(stream)>>>(
        l.dose, l.sd, l.rho, nvox, l.partials, stat_blocks(nvox, 1), result);
    return ok();
}

int launch_fold_multi(const FoldDesc *descs, const uint64_t *tile_off, int n, uint64_t total_tiles, void *stream)
{
    if (total_tiles == 0) return CTD_OK;
    const int grid = total_tiles < 152 * 16 ? static_cast<int>(total_tiles) : 152 * 16;
    fold_multi_kernel<<<grid, kThreads, 0, static_cast<cudaStream_t>(stream)>>>(descs, tile_off, n, total_tiles);
    return ok();
}

int launch_scan_phantom(const uint8_t *mat, const float *rho, size_t nvox, int n_mat, uint32_t *vox, double *rinv,
                        PhantomScan *out, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    PhantomScan init{};
    init.first_bad_mat = ~0ull;
    init.first_bad_rho = ~0ull;
    if (cudaMemcpyAsync(out, &init, sizeof(init), cudaMemcpyHostToDevice, s) != cudaSuccess) return CTD_ECUDA;
    scan_phantom_kernel<<<stat_blocks(nvox, 1), kThreads, 0, s>>>(mat, rho, nvox, n_mat, vox, rinv, out);
    return ok();
}

int launch_cells(const float *rows, int k, int n_e, int n_zeta, float *cells, void *stream)
{
    const int n_rows = k * (n_e - 1);
    cells_kernel<<<n_rows < kMaxStatBlocks ? n_rows : kMaxStatBlocks, kThreads, 0, static_cast<cudaStream_t>(stream)>>>(
        rows, n_rows, n_e, n_zeta, reinterpret_cast<float4 *>(cells));
    return ok();
}

int launch_sum(const double *x, size_t n, double *partials, double *result, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int grid = stat_blocks(n, kPerThread);
    sum_kernel<<<grid, kThreads, 0, s>>>(x, n, partials);
    sum_final_kernel<<<1, kThreads, 0, s>>>(partials, grid, result);
    return ok();
}

}  // namespace ctd
