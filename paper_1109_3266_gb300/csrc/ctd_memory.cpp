// ctd_memory.cpp -- device memory of the contexts: released buffers kept for reuse, the
// scratch block a call borrows, and allocations that take idle memory back.
#include <cuda_runtime.h>

#include <algorithm>

#include "ctd_host.h"

namespace ctd {
namespace host {
namespace {

// The contexts' caches, so that one context's allocation can have what another keeps
// idle.  Locked before any cache's own lock; never destroyed (contexts may outlive it).
struct Registry {
    std::mutex lock;
    std::vector<BufferCache *> caches;
};

Registry &registry()
{
    static Registry *r = new Registry;
    return *r;
}

}  // namespace

void BufferCache::attach(int device)
{
    Registry &r = registry();
    std::lock_guard<std::mutex> l(r.lock);
    device_ = device;
    r.caches.push_back(this);
}

BufferCache::~BufferCache()
{
    {
        Registry &r = registry();
        std::lock_guard<std::mutex> l(r.lock);
        r.caches.erase(std::remove(r.caches.begin(), r.caches.end(), this), r.caches.end());
    }
    lent_ = false;
    drop();
}

void *BufferCache::take(size_t bytes)
{
    std::lock_guard<std::mutex> l(lock_);
    auto it = blocks_.find(bytes);
    if (it == blocks_.end()) return nullptr;
    void *p = it->second;
    blocks_.erase(it);
    cached_ -= bytes;
    return p;
}

bool BufferCache::give(void *p, size_t bytes)
{
    void *old = nullptr;
    {
        std::lock_guard<std::mutex> l(lock_);
        if (cached_ + bytes > kCap) return false;
        blocks_.emplace(bytes, p);
        cached_ += bytes;
        if (!lent_) old = excess_scratch();
    }
    if (old) cudaFree(old);
    return true;
}

// the scratch block, no longer the cache's, if it has no place beside the buffers
void *BufferCache::excess_scratch()
{
    if (cached_ + scratch_bytes_ <= kCap) return nullptr;
    void *p = scratch_;
    scratch_ = nullptr;
    scratch_bytes_ = 0;
    return p;
}

size_t BufferCache::idle() const
{
    std::lock_guard<std::mutex> l(lock_);
    return cached_ + (lent_ ? 0 : scratch_bytes_);
}

size_t BufferCache::drop()
{
    std::multimap<size_t, void *> blocks;
    {
        std::lock_guard<std::mutex> l(lock_);
        blocks.swap(blocks_);
        cached_ = 0;
        if (!lent_ && scratch_) {
            blocks.emplace(scratch_bytes_, scratch_);
            scratch_ = nullptr;
            scratch_bytes_ = 0;
        }
    }
    size_t n = 0;
    for (auto &b : blocks) {
        cudaFree(b.second);
        n += b.first;
    }
    return n;
}

void *BufferCache::borrow(size_t bytes)
{
    void *old;
    {
        std::lock_guard<std::mutex> l(lock_);
        if (lent_) return nullptr;
        lent_ = true;
        if (scratch_bytes_ >= bytes) return scratch_;
        old = scratch_;
        scratch_ = nullptr;
        scratch_bytes_ = 0;
    }
    if (old) cudaFree(old);
    void *p = device_allocate(bytes);
    std::lock_guard<std::mutex> l(lock_);
    scratch_ = p;
    scratch_bytes_ = p ? bytes : 0;
    lent_ = p != nullptr;
    return p;
}

void BufferCache::return_scratch()
{
    void *old;
    {
        std::lock_guard<std::mutex> l(lock_);
        lent_ = false;
        old = excess_scratch();
    }
    if (old) cudaFree(old);
}

void *device_allocate(size_t bytes)
{
    void *p = nullptr;
    if (cudaMalloc(&p, bytes) == cudaSuccess) return p;
    cudaGetLastError();
    int device = -1;
    cudaGetDevice(&device);
    size_t n = 0;
    {
        Registry &r = registry();
        std::lock_guard<std::mutex> l(r.lock);
        for (BufferCache *c : r.caches)
            if (c->device() == device) n += c->drop();
    }
    if (n && cudaMalloc(&p, bytes) == cudaSuccess) return p;
    cudaGetLastError();
    return nullptr;
}

}  // namespace host
}  // namespace ctd
