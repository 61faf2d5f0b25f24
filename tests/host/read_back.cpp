// The read-back (read_back) with destinations of every kind, over fakes of the CUDA calls:
// host memory new and in use, and memory that CUDA knows, which the host may not touch
// before the copy.  A "device" destination is address space without access, as a device
// allocation's is: a host thread that writes to it ends this process.
#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>

#include "ctd_host.h"

namespace {

struct Region {
    size_t n;
    cudaMemoryType type;
};
std::map<char *, Region> known;   // what cudaPointerGetAttributes knows
int touched;                      // copies into managed memory that found pages there already

const Region *region(const void *p)
{
    auto it = known.upper_bound(const_cast<char *>(static_cast<const char *>(p)));
    if (it == known.begin()) return nullptr;
    --it;
    return static_cast<const char *>(p) < it->first + it->second.n ? &it->second : nullptr;
}

}  // namespace

extern "C" {
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p)
{
    const Region *r = region(p);
    std::memset(a, 0, sizeof(*a));
    a->type = r ? r->type : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind, cudaStream_t)
{
    const Region *r = region(dst);
    if (r && r->type == cudaMemoryTypeDevice) return cudaErrorInvalidValue;
    if (r && r->type == cudaMemoryTypeManaged) {
        const size_t page = static_cast<size_t>(sysconf(_SC_PAGESIZE));
        unsigned char in = 0;
        char *p = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(dst) + n / 2) & ~(page - 1));
        mincore(p, page, &in);
        touched += in & 1;
    }
    std::memcpy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *) { return cudaSuccess; }
cudaError_t cudaMalloc(void **, size_t) { return cudaErrorMemoryAllocation; }
}

namespace ctd {
namespace host {
int fail(int code, const char *, ...) { return code; }
}  // namespace host
}  // namespace ctd

using namespace ctd::host;

static char *pages(size_t n, int prot)
{
    return static_cast<char *>(mmap(nullptr, n, prot, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0));
}

// kinds: one letter for each of the two outputs.  n new host memory, u host memory in use,
// m managed, d device, p pinned (in use)
int main(int argc, char **argv)
{
    const std::string kinds = argv[1];
    const size_t n = static_cast<size_t>(atoll(argv[2]));
    std::string src(n, 'x');
    for (size_t i = 0; i < n; ++i) src[i] = static_cast<char>(i * 7 + i / 4096);
    ctd_ctx ctx;
    ReadPart parts[2];
    char *dst[2];
    bool device = false;
    for (int i = 0; i < 2; ++i) {
        const char k = kinds[i];
        dst[i] = pages(n, k == 'd' ? PROT_NONE : PROT_READ | PROT_WRITE);
        if (k == 'u' || k == 'p') std::memset(dst[i], 1, n);
        if (k == 'm') known[dst[i]] = {n, cudaMemoryTypeManaged};
        if (k == 'd') known[dst[i]] = {n, cudaMemoryTypeDevice};
        if (k == 'p') known[dst[i]] = {n, cudaMemoryTypeHost};
        device = device || k == 'd';
        parts[i] = {dst[i], src.data(), n};
    }
    const int rc = read_back(&ctx, parts, 2);
    if (rc != (device ? CTD_ECUDA : CTD_OK)) return 10 + rc;
    if (touched) return 30;
    if (!device)
        for (int i = 0; i < 2; ++i)
            if (std::memcmp(dst[i], src.data(), n) != 0) return 40;
    std::puts("ok");
    return 0;
}
