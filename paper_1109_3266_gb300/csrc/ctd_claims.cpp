// ctd_claims.cpp -- the histories of a single-request launch: batches, claims of the
// warps, and the pieces whose histories share the upper word of their index.
#include <cuda_runtime.h>

#include <algorithm>

#include "ctd_host.h"

namespace ctd {
namespace host {

// Claims: `chunk` histories each (for a launch that has the GPU to itself, a sixteenth of a
// warp's share of it raised to the next multiple of 32, at most `chunk`) until what is left
// is some 256 per warp, then 32, one round of source photons.  1e6 histories (a 51x51x32 head, 183 per warp) took 0.43 ms
// while half of them went in claims of 256, 0.23 in claims of 32; for 1e5 claims of 18, so
// that every warp has one, took 0.080 ms, claims of 32 0.057.
// With claims of 256 in every launch of more than 256 per warp the first round alone was
// 1.4e6 histories, and a warp that met a costly run of them (a batch's histories go from
// low energies to high) ended last: 1.5e6 histories took 0.454 ms, now 0.285; 4e6 0.701 ->
// 0.567 (head), 0.384 -> 0.362 (water); 1e7 1.350 -> 1.286; from some 2e7 nothing changes,
// where claims of 64 throughout would cost 2 to 5 %.  An eighth of a share,
// raised likewise, lost 4 to 8 % at 4e6 to 1e7 on heads, a thirtieth 2 to 3 % on water.  Beside other launches (streams of
// chains, overlapped batches, requests of one launch) the tails are filled anyway and
// smaller claims only cost: eight served requests of 4e6 histories a batch 108 -> 113 ms,
// overlapped batches of 2.5e6 water histories 0.97 -> 1.03.
constexpr int kClaimsPerWarp = 16;
static void set_claims(ctd::RequestDesc &q, uint64_t h0, uint64_t h1, int chunk, int warps, bool alone)
{
    const uint64_t larger = q.rem * (q.n_lo + 1);   // histories in the larger batches
    q.b0 = static_cast<int>(h0 < larger ? h0 / (q.n_lo + 1) : q.rem + (h0 - larger) / q.n_lo);
    q.h_begin = h0;
    q.h_end = h1;
    const uint64_t tail = 256 * static_cast<uint64_t>(std::max(warps, 1));
    q.h_big = h1 - h0 > tail ? h1 - tail : h0;
    const uint64_t share = (h1 - h0) / (kClaimsPerWarp * static_cast<uint64_t>(std::max(warps, 1)));
    q.big = alone ? static_cast<int>(std::min<uint64_t>((share / 32 + 1) * 32, chunk)) : chunk;
    q.small = std::min(32, chunk);
    q.h_hi = static_cast<uint32_t>(h0 >> 32);
    q.k0 = q.rk[0] ^ q.h_hi;
}

void set_range(ctd::RequestDesc &q, uint64_t n, int nb, uint64_t h0, uint64_t h1, double *tally, uint32_t stride,
               int chunk, int warps, bool alone)
{
    q.n_lo = n / nb;
    q.rem = n % nb;
    q.tally = tally;
    q.tally_stride = stride;
    set_claims(q, h0, h1, chunk, warps, alone);
}

int launch_single(const ctd_ctx *ctx, ctd::LaunchParams &L, const LaunchShape &shape, bool alone, cudaStream_t s,
                  const ctd::L2Window *win)
{
    ctd::RequestDesc &q = L.one;
    const uint64_t end = q.h_end;
    double *const tally = q.tally;
    const int b0 = q.b0, warps = shape.grid * (shape.block / 32);
    for (uint64_t h = q.h_begin; h < end; h = q.h_end) {
        const uint64_t last = h | 0xffffffffull;   // the last history with this upper word
        if (h != q.h_begin || last < end - 1) {
            if (h != q.h_begin && cudaMemsetAsync(q.work, 0, sizeof(unsigned long long), s) != cudaSuccess) return CTD_ECUDA;
            set_claims(q, h, last < end - 1 ? last + 1 : end, ctx->chunk, warps, alone);
            q.tally = tally + static_cast<size_t>(q.b0 - b0) * q.tally_stride;
        }
        const int rc = ctd::launch_transport(L, shape.grid, shape.block, shape.threads_per_sm, s, win);
        if (rc != CTD_OK) return rc;
    }
    return CTD_OK;
}

}  // namespace host
}  // namespace ctd
