// The library's device allocations over a fake device of a given size: what is idle in
// any context is given back when an allocation finds no memory, what is lent or in use is
// not, and two threads with a context each neither lose nor free a block twice.
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "ctd_host.h"

namespace {

std::mutex g_lock;
std::map<void *, std::pair<size_t, int>> g_blocks;
size_t g_used[2], g_size = 1000;
thread_local int g_device = 0;
int g_bad_frees = 0;

}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n)
{
    std::lock_guard<std::mutex> l(g_lock);
    if (g_used[g_device] + n > g_size) return cudaErrorMemoryAllocation;
    g_used[g_device] += n;
    *p = ::operator new(1);
    g_blocks[*p] = {n, g_device};
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    std::lock_guard<std::mutex> l(g_lock);
    auto it = g_blocks.find(p);
    if (it == g_blocks.end()) {
        ++g_bad_frees;
        return cudaErrorInvalidValue;
    }
    g_used[it->second.second] -= it->second.first;
    ::operator delete(p);
    g_blocks.erase(it);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = g_device;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
}

namespace ctd {
namespace host {
int fail(int code, const char *, ...) { return code; }
}  // namespace host
}  // namespace ctd

using namespace ctd::host;

#define EXPECT(x)                                              \
    do {                                                       \
        if (!(x)) {                                            \
            std::printf("line %d: %s\n", __LINE__, #x);        \
            return 1;                                          \
        }                                                      \
    } while (0)

// a released buffer of n bytes idle in c
static void release_into(BufferCache &c, size_t n)
{
    DevBuf<char> b;
    b.cache = &c;
    b.ensure(n);
}

// idle buffers and idle scratch, given back to an allocation of `who`: a buffer of the
// same context's (c), one without a context's cache (n), another context's (o)
static int given_back(char who)
{
    BufferCache a, other;
    a.attach(0);
    other.attach(0);
    release_into(a, 300);
    {
        Scratch s(a, nullptr);
        EXPECT(s.borrow(40));
        EXPECT(a.idle() == 300);
    }
    EXPECT(a.idle() == 620 && g_used[0] == 620);
    DevBuf<char> b;
    if (who == 'c') b.cache = &a;
    if (who == 'o') b.cache = &other;
    EXPECT(b.ensure(900) == CTD_OK);
    EXPECT(g_used[0] == 900 && a.idle() == 0);
    DevBuf<char> d;
    EXPECT(d.ensure(200) == CTD_ENOMEM && !d.p);
    return 0;
}

// lent scratch, buffers in use and other devices' idle memory stay
static int kept()
{
    BufferCache a, far;
    a.attach(0);
    far.attach(1);
    g_device = 1;
    release_into(far, 700);
    g_device = 0;
    Scratch s(a, nullptr);
    EXPECT(s.borrow(50));
    DevBuf<char> used;
    used.cache = &a;
    EXPECT(used.ensure(300) == CTD_OK);
    DevBuf<char> b;
    EXPECT(b.ensure(400) == CTD_ENOMEM);
    EXPECT(g_used[0] == 700 && g_used[1] == 700 && far.idle() == 700);
    Scratch second(a, nullptr);
    EXPECT(!second.borrow(1));
    return 0;
}

// buffers and scratch together stay within what a context may keep, the buffers first
static int bounded()
{
    const size_t G = size_t(1) << 30;
    g_size = 64 * G;
    EXPECT(BufferCache::kCap == 4 * G);
    BufferCache a;
    a.attach(0);
    auto lend = [&](size_t bytes) {
        Scratch s(a, nullptr);
        return s.borrow(bytes / 8);
    };
    EXPECT(lend(4 * G) && a.idle() == 4 * G);      // alone: kept
    release_into(a, G);                            // a released buffer takes its place
    EXPECT(a.idle() == G && g_used[0] == G);
    EXPECT(lend(3 * G) && a.idle() == 4 * G);      // just fits beside it
    EXPECT(lend(3 * G + 8) && a.idle() == G);      // does not: given back when the call ends
    {
        Scratch s(a, nullptr);
        EXPECT(s.borrow(2 * G / 8));
        release_into(a, 2 * G);                    // released while it is lent
        EXPECT(a.idle() == 3 * G && g_used[0] == 5 * G);
    }
    EXPECT(a.idle() == 3 * G && g_used[0] == 3 * G);
    release_into(a, 2 * G);                        // the cached one, taken and released again
    release_into(a, G + G / 2);                    // more than may be kept
    EXPECT(a.idle() == 3 * G && g_used[0] == 3 * G);
    return 0;
}

static int threads()
{
    bool ok[2] = {false, false};
    auto work = [&](int t) {
        BufferCache c;
        c.attach(0);
        ok[t] = true;
        for (int i = 0; i < 20000; ++i) {
            DevBuf<char> b, n;
            b.cache = &c;
            b.ensure(100 + 50 * (i % 7));
            n.ensure(200 + 100 * (i % 5));
            Scratch s(c, nullptr);
            if (s.borrow(1 + i % 60)) ok[t] = ok[t] && s.p;
        }
    };
    std::thread a(work, 0), b(work, 1);
    a.join();
    b.join();
    EXPECT(ok[0] && ok[1]);
    return 0;
}

int main(int, char **argv)
{
    const std::string what = argv[1];
    const int rc = what == "kept" ? kept() : what == "bounded" ? bounded() : what == "threads" ? threads() : given_back(what[0]);
    if (rc) return rc;
    EXPECT(g_bad_frees == 0 && g_used[0] == 0 && g_used[1] == 0);
    std::puts("ok");
    return 0;
}
