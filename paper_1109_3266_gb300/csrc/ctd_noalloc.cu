// ctd_noalloc.cu -- an allocation-free variant of the avg-RSD reduction.
//
// Some callers cannot allocate device memory at the moment they need the
// precision measure, such as hosts that hand all device memory to their own
// pool allocator and forbid libraries from calling cudaMalloc.  For them,
// ctd_avg_rsd_noalloc reduces dose and stddev arrays that already live on the
// device, using per-block partial sums kept in a fixed file-scope device array
// instead of library-allocated scratch.
//
// The array (g_rsd_scratch, 5 * kMaxStatBlocks + 8 doubles = 48 KB) is part of the
// library image: every GPU that loads the library holds it until the process
// exits.  All calls share it; each call overwrites everything in it that it reads,
// so nothing is carried over from the previous call, but calls that overlap on
// the GPU (on different streams, or from different host threads) race on it.
#include <cuda_runtime.h>

#include <mutex>

#include "ctd_internal.h"
#include "ctd_stats.cuh"

namespace {

using namespace ctd::stats;

constexpr size_t kMaxVoxels = 67108864;
constexpr int kScratchDoubles = 5 * kMaxStatBlocks + 8;      // partials: 1 max + 4 sums per block, + 8 cells
constexpr int kMaxDevices = 64;

static __device__ __align__(256) double g_rsd_scratch[kScratchDoubles];

// layout inside the scratch array
constexpr int kOffMax = 0;                       // [kMaxStatBlocks] per-block maxima (bit patterns)
constexpr int kOffSums = kMaxStatBlocks;         // [4][kMaxStatBlocks] per-block sums
constexpr int kOffCells = 5 * kMaxStatBlocks;    // [0] = blocks done

// Two kernels, bound by memory: 12 bytes a voxel for the maximum, then 20 (8 less
// outside the mask) for the sums, 10.5 M voxels in 31 us at the measured copy rate
// if each byte came from HBM once.  The last block to finish adds the partial
// sums up.  With a division per voxel, single-thread final sums and four kernels the
// call took 421 us on such a head; now 145, of which 24 are the maximum's at 5.3 TB/s and
// the rest the sums', bound by the FP64 pipe (80 % busy).

// maximum dose over voxels with rho >= 0.1, per block
__global__ void __launch_bounds__(kThreads) na_dmax_kernel(const double *__restrict__ dose,
                                                           const float *__restrict__ rho, size_t nvox, double *scratch)
{
    long long m = 0;
    const size_t stride = static_cast<size_t>(gridDim.x) * kThreads;
    for (size_t v0 = blockIdx.x * static_cast<size_t>(kThreads) + threadIdx.x; v0 < nvox; v0 += kPerThread * stride) {
        float r[kPerThread];
        double d[kPerThread];
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) {
            const size_t v = v0 + k * stride;
            r[k] = v < nvox ? rho[v] : 0.0f;
            d[k] = v < nvox ? dose[v] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < kPerThread; ++k)
            if (r[k] >= 0.1f) m = max_dose(m, d[k]);
    }
    m = block_max(m);
    if (threadIdx.x == 0) {
        reinterpret_cast<long long *>(scratch + kOffMax)[blockIdx.x] = m;
        if (blockIdx.x == 0) *reinterpret_cast<unsigned *>(scratch + kOffCells) = 0;
    }
}

// sums of s/D over D > 0.1 D_max and of s over D > 0.2 D_max, with their counts, and
// the measures from them
__global__ void __launch_bounds__(kThreads) na_rsd_kernel(const double *__restrict__ dose,
                                                          const double *__restrict__ sd, const float *__restrict__ rho,
                                                          size_t nvox, double *scratch, double *result)
{
    const double dmax =
        __longlong_as_double(max_of(reinterpret_cast<const long long *>(scratch + kOffMax), gridDim.x));
    rsd_sums(dose, sd, rho, nvox, dmax, scratch + kOffSums, kMaxStatBlocks);
    if (last_block(reinterpret_cast<unsigned *>(scratch + kOffCells)))
        rsd_result<false>(scratch + kOffSums, kMaxStatBlocks, gridDim.x, dmax, nullptr, 0, result);
}

std::mutex g_mu;
double *g_scratch_ptr[kMaxDevices];   // device address of g_rsd_scratch, per device

int na_fail(int code, const char *msg)
{
    ctd::set_error(msg);
    return code;
}

}  // namespace

extern "C" {

int ctd_avg_rsd_noalloc(const double *dose_dev, const double *stddev_dev, const float *density_dev, size_t nvox,
                        double *result_dev, void *stream)
{
    ctd::set_error("");
    if (!dose_dev || !stddev_dev || !density_dev || !result_dev) return na_fail(CTD_EINVAL, "null device pointer");
    if (nvox == 0) return na_fail(CTD_EINVAL, "nvox must be positive");
    if (nvox > kMaxVoxels)
        return na_fail(CTD_EINVAL, "nvox exceeds the 67,108,864 voxels the fixed scratch array covers");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return na_fail(CTD_ECUDA, "no usable current CUDA device");
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // The scratch array's device address, looked up with the device current.  Outside
    // stream capture it is looked up on every call (a device reset reloads the module
    // and moves the array); during capture the address of this device's last lookup
    // is used.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
        cudaGetLastError();
        cap = cudaStreamCaptureStatusActive;   // unknown: take the cached address
    }
    double *scratch;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (cap == cudaStreamCaptureStatusNone || !g_scratch_ptr[dev]) {
            void *p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_rsd_scratch);
            if (e != cudaSuccess || !p) {
                cudaGetLastError();
                return na_fail(CTD_ECUDA, "cudaGetSymbolAddress of the scratch array failed");
            }
            g_scratch_ptr[dev] = static_cast<double *>(p);
        }
        scratch = g_scratch_ptr[dev];
    }
    const int nblocks = stat_blocks(nvox, kPerThread);
    na_dmax_kernel<<<nblocks, kThreads, 0, s>>>(dose_dev, density_dev, nvox, scratch);
    na_rsd_kernel<<<nblocks, kThreads, 0, s>>>(dose_dev, stddev_dev, density_dev, nvox, scratch, result_dev);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return na_fail(CTD_ECUDA, cudaGetErrorString(e));
    return CTD_OK;
}

}  // extern "C"
