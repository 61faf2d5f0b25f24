// Prints the launches of histories [h0, h1) of n in nb batches: for each its range, first
// batch, tally offset, the two sizes of claims and where the small ones begin.
// Arguments: n, nb, h0, h1, chunk, warps, alone.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "ctd_host.h"

namespace {
double *g_tally = reinterpret_cast<double *>(1 << 20);
int g_cleared = 0;
}  // namespace

extern "C" {
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t)
{
    ++g_cleared;
    return cudaSuccess;
}
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaMalloc(void **, size_t) { return cudaErrorMemoryAllocation; }
cudaError_t cudaGetDevice(int *) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
}

namespace ctd {
int launch_transport(const LaunchParams &p, int, int, int, void *, const L2Window *)
{
    const RequestDesc &q = p.one;
    std::printf("%llu %llu %d %td %d %d %llu %u %d\n", static_cast<unsigned long long>(q.h_begin),
                static_cast<unsigned long long>(q.h_end), q.b0, q.tally - g_tally, q.big, q.small,
                static_cast<unsigned long long>(q.h_big), q.h_hi, g_cleared);
    return CTD_OK;
}
namespace host {
int fail(int code, const char *, ...) { return code; }
}  // namespace host
}  // namespace ctd

int main(int, char **argv)
{
    auto u = [&](int i) { return std::strtoull(argv[i], nullptr, 10); };
    ctd_ctx ctx;
    ctx.chunk = static_cast<int>(u(5));
    const int warps = static_cast<int>(u(6));
    const bool alone = u(7) != 0;
    ctd::LaunchParams L;
    std::memset(&L, 0, sizeof(L));
    ctd::host::set_range(L.one, u(1), static_cast<int>(u(2)), u(3), u(4), g_tally, 1000, ctx.chunk, warps, alone);
    return ctd::host::launch_single(&ctx, L, {warps, 32, 32}, alone, nullptr);
}
