// ctd_readback.cpp -- results from device arrays into the caller's host memory.
#include <cuda_runtime.h>

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <memory>
#include <thread>
#include <vector>

#include "ctd_host.h"

namespace ctd {
namespace host {

// Device arrays read back into host memory the caller has just allocated: its pages
// do not exist yet, and the copy itself (185 GB/s into existing pages) would wait for
// the kernel to make them one by one, 4 ms for 134 MB.  A few threads make them, a
// chunk at a time by writing one byte to each page of the destination (which the copy
// overwrites), while the copies follow chunk by chunk.  Outputs that are small, resident
// already (a reused buffer, by mincore) or in memory that CUDA knows (pinned, managed,
// or a device pointer given by mistake, which the copy refuses) are copied as they are:
// the host writes to nothing but plain memory.
namespace {

constexpr size_t kColdBytes = size_t(4) << 20, kReadChunk = size_t(8) << 20;

// whether most of the n bytes at p are pages without memory behind them
bool cold(const char *p, size_t n, size_t page)
{
    const uintptr_t a = reinterpret_cast<uintptr_t>(p) & ~(page - 1);
    const size_t pages = (reinterpret_cast<uintptr_t>(p) + n - a + page - 1) / page;
    std::vector<unsigned char> in(pages);
    if (mincore(reinterpret_cast<void *>(a), pages * page, in.data()) != 0) return false;
    size_t there = 0;
    for (unsigned char c : in) there += c & 1u;
    return 2 * there < pages;
}

// whether n bytes at p are memory of the process that CUDA knows nothing of
bool plain(const char *p, size_t n)
{
    for (const char *q : {p, p + n - 1}) {
        cudaPointerAttributes a;
        if (cudaPointerGetAttributes(&a, q) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (a.type != cudaMemoryTypeUnregistered) return false;
    }
    return true;
}

}  // namespace

int read_back(ctd_ctx *ctx, const ReadPart *parts, int n_parts)
{
    struct Chunk {
        char *dst;
        const char *src;
        size_t n;
        bool make;   // its pages are made before the copy
    };
    const size_t page = static_cast<size_t>(sysconf(_SC_PAGESIZE));
    size_t bytes = 0;
    for (int i = 0; i < n_parts; ++i) bytes += parts[i].bytes;
    std::vector<Chunk> chunks;
    std::vector<std::thread> makers;
    std::unique_ptr<std::atomic<int>[]> made;
    std::atomic<size_t> next{0};
    if (bytes >= kColdBytes) try {
            bool any = false;
            for (int i = 0; i < n_parts; ++i) {
                char *dst = static_cast<char *>(parts[i].dst);
                const size_t n = parts[i].bytes;
                const bool make = n >= page && cold(dst, n, page) && plain(dst, n);
                const size_t step = make ? kReadChunk : std::max<size_t>(n, 1);
                any = any || make;
                for (size_t o = 0; o < n; o += step)
                    chunks.push_back({dst + o, static_cast<const char *>(parts[i].src) + o, std::min(step, n - o), make});
            }
            if (any) {
                made.reset(new std::atomic<int>[chunks.size()]());
                const size_t hw = std::max(2u, std::thread::hardware_concurrency());
                const size_t n = std::min({size_t(6), hw / 2, chunks.size()});
                makers.reserve(n);
                for (size_t t = 0; t < n; ++t)
                    makers.emplace_back([&] {
                        for (size_t k; (k = next.fetch_add(1)) < chunks.size();) {
                            volatile char *p = chunks[k].dst;
                            if (chunks[k].make) {
                                for (size_t o = 0; o < chunks[k].n; o += page) p[o] = 0;
                                p[chunks[k].n - 1] = 0;
                            }
                            made[k].store(1, std::memory_order_release);
                        }
                    });
            }
        } catch (const std::exception &) {
            // no memory or no threads: what threads there are finish, the copies do not wait
        }
    cudaError_t e = cudaSuccess;
    if (makers.empty()) {
        for (int i = 0; i < n_parts && e == cudaSuccess; ++i)
            e = cudaMemcpyAsync(parts[i].dst, parts[i].src, parts[i].bytes, cudaMemcpyDeviceToHost, ctx->stream);
    } else {
        for (size_t k = 0; k < chunks.size(); ++k) {
            while (!made[k].load(std::memory_order_acquire)) std::this_thread::yield();
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(chunks[k].dst, chunks[k].src, chunks[k].n, cudaMemcpyDeviceToHost, ctx->stream);
        }
        for (std::thread &t : makers) t.join();
    }
    if (e != cudaSuccess) return fail(CTD_ECUDA, "cudaMemcpyAsync failed: %s", cudaGetErrorString(e));
    CK(cudaStreamSynchronize(ctx->stream));
    return CTD_OK;
}

}  // namespace host
}  // namespace ctd
