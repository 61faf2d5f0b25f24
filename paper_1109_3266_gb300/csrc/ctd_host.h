// ctd_host.h -- host-side state behind the C ABI of include/ctd.h, shared by
// ctd_capi.cu (contexts, phantoms, set-up, the plain form, results),
// ctd_forms.cu (the batched and served forms), ctd_tune.cu (launch-shape
// search, memory probes), ctd_claims.cpp (the histories of a launch),
// ctd_memory.cpp (device memory) and ctd_readback.cpp (results into host memory).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cstdint>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "ctd_internal.h"

namespace ctd {
namespace host {

// the calling thread's message for ctd_last_error(); fail() sets it and returns code
extern thread_local std::string g_error;
int fail(int code, const char *fmt, ...);

#define CK(call)                                                                                          \
    do {                                                                                                  \
        cudaError_t e_ = (call);                                                                          \
        if (e_ != cudaSuccess) return ::ctd::host::fail(CTD_ECUDA, "%s failed: %s", #call, cudaGetErrorString(e_));  \
    } while (0)

#define CKS(call)                                                                                         \
    do {                                                                                                  \
        int s_ = (call);                                                                                  \
        if (s_ != CTD_OK) {                                                                               \
            if (::ctd::host::g_error.empty()) ::ctd::host::fail(s_, "%s failed: %s", #call, cudaGetErrorString(cudaGetLastError())); \
            return s_;                                                                                    \
        }                                                                                                 \
    } while (0)

// Device buffers a context has released and may hand out again: the byte size of
// each, and one block of scratch memory that a call borrows while it runs; up to kCap
// bytes in all while no call runs, the released buffers before the scratch.  A phantom's buffers return here when it is destroyed (after its
// context's stream is idle), so a phantom of the same size created next takes them
// without cudaMalloc, and no cudaFree synchronises the device meanwhile.  The context
// frees what is left when it is destroyed; what is idle here is given back to the device
// when an allocation of this or another context of the process finds no memory
// (device_allocate), which may run in another thread.
class BufferCache {
public:
    static constexpr size_t kCap = size_t(4) << 30;
    BufferCache() = default;
    ~BufferCache();
    void attach(int device);   // once, before the context has any buffer
    int device() const { return device_; }
    void *take(size_t bytes);
    bool give(void *p, size_t bytes);
    // bytes that drop() would free
    size_t idle() const;
    // frees what is idle; the bytes freed
    size_t drop();
    // The scratch block, of at least `bytes` (it grows only); nullptr if it is lent
    // already or there is no memory.
    void *borrow(size_t bytes);
    void return_scratch();

private:
    void *excess_scratch();
    mutable std::mutex lock_;
    std::multimap<size_t, void *> blocks_;
    size_t cached_ = 0;
    void *scratch_ = nullptr;
    size_t scratch_bytes_ = 0;
    bool lent_ = false;
    int device_ = -1;
};

// cudaMalloc on the current device, once more after its contexts' idle memory is given
// back; nullptr if there is none
void *device_allocate(size_t bytes);

template <class T>
struct DevBuf {
    T *p = nullptr;
    size_t n = 0;
    BufferCache *cache = nullptr;   // where released buffers go (nullptr: cudaFree)
    ~DevBuf() { release(); }
    void release()
    {
        if (p && !(cache && cache->give(p, n * sizeof(T)))) cudaFree(p);
        p = nullptr;
        n = 0;
    }
    int ensure(size_t count)
    {
        if (count <= n && p) return CTD_OK;
        release();
        if (count == 0) count = 1;
        if (cache) p = static_cast<T *>(cache->take(count * sizeof(T)));
        if (!p) p = static_cast<T *>(device_allocate(count * sizeof(T)));
        if (!p) return fail(CTD_ENOMEM, "cudaMalloc of %zu bytes failed", count * sizeof(T));
        n = count;
        return CTD_OK;
    }
};

struct Phantom {
    int nx = 0, ny = 0, nz = 0;
    double dx = 0, dy = 0, dz = 0;
    size_t nvox = 0;
    std::vector<ctd_material> mats;
    std::vector<ctd::Elements> els;   // per material: independent-atom Rayleigh form factor (n = 0: none)
    std::vector<double> rho_max;
    std::vector<int> present;
    ctd_physics phys{};
    ctd_source src{};
    bool has_src = false;
    std::vector<double> e_lo, e_hi, w;
    bool has_spec = false;

    DevBuf<uint8_t> mat;
    DevBuf<float> rho;
    DevBuf<uint32_t> vox;      // material and density packed (what the transport reads)
    DevBuf<double> rinv;       // 1 / density per voxel, 0 where it is 0 (what the fold reads)
    // tables
    bool tables_ok = false;
    int n_e = 0;
    std::vector<float> h_tab, h_mm, h_cs, h_rs;
    DevBuf<float> tab, mm, cs, rs;
    // per-run state
    DevBuf<double> tally, sum_d, sum_d2, edep, dose, sd, partials;
    DevBuf<double> tally2;     // the second stream's batch tally of an overlapped plain run
    DevBuf<ctd::RunState> state;
    ctd::DeviceCounts *counts() const { return &state.p->c; }
    unsigned long long *work() const { return state.p->work; }
    double *result() const { return state.p->result; }
    DevBuf<uint64_t> pref;     // [2][nbins+1]: batch of n_lo+1, batch of n_lo
    DevBuf<float2> bins;       // [nbins]: lo, hi
    DevBuf<float4> proj;       // [n_proj]: cos, sin, height
    uint64_t alloc_n = ~0ull;
    int alloc_nb = -1;
    ctd_run_stats stats{};
    bool have_result = false;
    int64_t busy_req = 0;      // served request using this phantom, 0 if none
    // fluence map (Sec. 2.2.4): alias table over fl_nu x fl_nv beamlets (fl_nu = 0: none)
    int fl_nu = 0, fl_nv = 0;
    std::vector<uint32_t> h_thr;
    std::vector<int32_t> h_alias;
    DevBuf<uint2> fl;          // threshold, alias
    // a sharded run in progress (ctd_shard_*): its history count, batches and seed
    uint64_t shard_n = 0, shard_seed = 0;
    int shard_nb = 0;
    double shard_t0 = 0.0;
    // every device buffer of the phantom takes from and returns to cache c
    void use_cache(BufferCache *c)
    {
        for (DevBuf<float> *b : {&rho, &tab, &mm, &cs, &rs}) b->cache = c;
        bins.cache = c;
        proj.cache = c;
        fl.cache = c;
        for (DevBuf<double> *b : {&tally, &tally2, &sum_d, &sum_d2, &edep, &dose, &sd, &partials})
            b->cache = c;
        mat.cache = c;
        vox.cache = c;
        rinv.cache = c;
        state.cache = c;
        pref.cache = c;
    }
};

// The context's scratch block for the length of one call (on stream s, which is waited
// for if the call fails).
struct Scratch {
    BufferCache &cache;
    cudaStream_t stream;
    double *p = nullptr;
    bool idle = false;   // set once the call has waited for its work
    Scratch(BufferCache &c, cudaStream_t s) : cache(c), stream(s) {}
    ~Scratch()
    {
        if (!p) return;
        if (!idle) cudaStreamSynchronize(stream);
        cache.return_scratch();
    }
    bool borrow(size_t doubles) { return (p = static_cast<double *>(cache.borrow(doubles * sizeof(double)))) != nullptr; }
};

struct ServeReq {
    int64_t id = 0;
    int ph = 0;
    ctd_request req{};
    int state = CTD_REQ_QUEUED;
    int batches = 0;
    uint64_t histories = 0;
    double avg_rsd = 0.0, sigma_bar = 0.0;
    double t_submit = 0.0, t_start = 0.0, t_done = 0.0;
    bool cancel = false;
    // request chains (shared_launch = 0): the stream slot the request runs on; the
    // slices of its current batch done (`slice`); what it has on the GPU: the
    // batches those launches complete (`group`, the last followed by the stop
    // test's statistics when `checked`), the slice count after them, their
    // histories, and whether the lane's second event marks the end of all of them
    // but the last (`split`)
    int lane = -1;
    int slice = 0, group = 0, slice_after = 0;
    double flight_histories = 0.0;
    bool in_flight = false, checked = false, split = false;
};

// device memory that a plain run may borrow for the tallies of batches that share a
// launch, and a batched call for all its requests' (the context keeps it for the next
// call, BufferCache)
constexpr size_t kTallyBudget = size_t(1) << 30, kBatchTallyBudget = size_t(4) << 30;
constexpr int kMaxLanes = 64;     // streams for request chains
constexpr uint64_t kMaxTrace = 1ull << 26;   // histories of one trace call (16 B of device memory each)

}  // namespace host
}  // namespace ctd

struct ctd_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int num_sms = 0;
    int blocks_per_sm = 4;
    int multi_blocks_per_sm = 3;   // multi-request launches hold more state per lane
    int threads = 256;
    int chunk = 256;
    int flight_cap = 4;
    // released device buffers (declared before the phantoms: it outlives them)
    ctd::host::BufferCache buffers;
    std::map<int, std::unique_ptr<ctd::host::Phantom>> phantoms;
    int next_id = 1;
    std::vector<cudaEvent_t> events;
    // multi-request launches: request and fold descriptors, claim counters
    ctd::host::DevBuf<ctd::RequestDesc> u_reqs;
    ctd::host::DevBuf<uint64_t> u_tiles;
    ctd::host::DevBuf<ctd::FoldDesc> u_folds;
    ctd::host::DevBuf<unsigned long long> u_work;
    // served form: all requests by id, the admission queue and the running set
    std::map<int64_t, ctd::host::ServeReq> sreqs;
    std::vector<int64_t> pending, active;
    int64_t next_req = 1;
    int max_active = 64;
    double round_histories = 1e8;   // admission stops once a round would exceed this
    // batched form: the captured batch loop and what it was captured for
    cudaGraphExec_t batch_graph = nullptr;
    std::vector<unsigned char> batch_graph_key;
    cudaStream_t capture_stream = nullptr;
    double reserve_bytes = 1.0 * (1ull << 30);
    // batched and served forms: 0 runs each request as its own chain of
    // single-request launches on its own stream (the device overlaps the chains),
    // 1 shares one multi-request launch per batch among all requests
    int shared_launch = 0;
    int batch_lanes = 64;          // batched form: streams the request chains share
    // plain-form launches: an L2 access-policy window over the tally (1) or the
    // packed voxel words (2), with a persisting set-aside of its size (granted bytes; at
    // most the device's maximum), no larger than the device's window; the context's
    // persisting-L2 limit before, put back on destroy
    int l2_persist = 0;
    // overlapped plain runs: the second stream, the event that starts it, and one event
    // per stream marking its last fold (folds run in batch order)
    bool plain_overlap = false;
    cudaStream_t plain_aux = nullptr;
    cudaEvent_t plain_fork = nullptr, plain_fold[2] = {nullptr, nullptr};
    size_t l2_asked = 0, l2_setaside = 0, l2_persist_max = 0, l2_window_max = 0, l2_prev_limit = 0;
    ctd::RunState *staged = nullptr;      // pinned read-back of counts and results
    size_t staged_n = 0;
    // angular surfaces by (kind, q0, e_min, n_e, n_zeta[, the elements' (Z, count) pairs]):
    // they do not depend on the phantom
    std::map<std::vector<double>, std::vector<float>> surfaces;
    // node-table columns of a material by (Compton model, e_min, n_e, its parameters and
    // elements): the Waller-Hartree and independent-atom totals are numeric integrals
    std::map<std::vector<double>, std::vector<double>> columns;
    std::vector<cudaStream_t> lanes;
    std::vector<cudaEvent_t> lane_done;
    cudaEvent_t fork_event = nullptr;
    // served request chains: the request holding each lane (0: free), an event per lane
    // marking the end of its batch in flight, and pinned slots [lane][4] the batch's
    // avg RSD, sigma_bar and D_max come back to
    std::vector<int64_t> lane_owner;
    std::vector<cudaStream_t> serve_hi;   // per lane, a stream of the device's greatest priority
    std::vector<cudaEvent_t> serve_ev;
    std::vector<cudaEvent_t> serve_ev_pre;   // per lane: every batch in flight but the last done
    double *serve_res = nullptr;
    ctd::host::DevBuf<unsigned long long> serve_work;   // claim counter per lane
};

namespace ctd {
namespace host {

int use_device(ctd_ctx *ctx);
Phantom *find(ctd_ctx *ctx, ctd_phantom id);
// CTD_EBUSY while a served request holds the phantom
int busy(Phantom *P);
// Klein-Nishina C (kind 0), Rayleigh R (kind 1, form-factor width q0) or
// Waller-Hartree C (kind 2, scattering-function width q0) surface in binary32,
// built once per context and node grid
const std::vector<float> &angular_surface(ctd_ctx *ctx, int kind, double q0, const ctd::Elements *el, int e_min, int n_e,
                                         int n_zeta);
// attenuation tables, majorant and surfaces of the phantom's physics, uploaded
int build_tables(ctd_ctx *ctx, Phantom &P);
// bin starts of the stratified allocation for batches of n / nb (and one more)
int upload_allocation(ctd_ctx *ctx, Phantom &P, uint64_t n, int nb);
int ensure_run_buffers(Phantom &P);
int check_ready(Phantom &P);
int prepare_run(ctd_ctx *ctx, Phantom &P, uint64_t n, int nb);
// the per-request part of a transport launch; the shared part
void fill_request(Phantom &P, uint64_t seed, ctd::RequestDesc &q);
void fill_shared(Phantom &P, ctd::SharedTables &sh);
cudaEvent_t event_at(ctd_ctx *ctx, size_t i);
// streams for independent request chains: chain r runs on lane(ctx, r)
int ensure_lanes(ctd_ctx *ctx, int n);
int fork_lanes(ctd_ctx *ctx, cudaStream_t origin, int n);
int join_lanes(ctd_ctx *ctx, cudaStream_t origin, int n);
// the last fold's outputs for a run of nb batches of P
ctd::FoldLast last_of(Phantom &P, int nb, bool keep_sums);
// mean, standard error, avg RSD and deposited energy of nb folded batches
int finish_stats(Phantom &P, int nb, cudaStream_t s);
// grid, block and threads per SM of a single-request launch
struct LaunchShape {
    int grid, block, threads_per_sm;
};
LaunchShape launch_shape(const ctd_ctx *ctx, const ctd::SharedTables &sh, int mode, bool trace);
// one single-request launch of q on stream s
int launch_one(ctd_ctx *ctx, Phantom &P, const ctd::RequestDesc &q, const LaunchShape &shape, bool alone,
               cudaStream_t s);
// q covers histories [h0, h1) of the problem of n histories in nb batches, deposits of
// its first batch into tally and of each later one `stride` voxels further on, for a
// launch of `warps` warps (`alone`: no other launch fills the SMs that it leaves idle)
void set_range(ctd::RequestDesc &q, uint64_t n, int nb, uint64_t h0, uint64_t h1, double *tally, uint32_t stride,
               int chunk, int warps, bool alone);
// launches L (one request, its range set) on s, in pieces whose histories share the
// upper word of their index (`alone` as in set_range); the claim counter is at 0
int launch_single(const ctd_ctx *ctx, ctd::LaunchParams &L, const LaunchShape &shape, bool alone, cudaStream_t s,
                  const ctd::L2Window *win = nullptr);
// batch b of n histories in nb batches: its first history
inline uint64_t batch_start(uint64_t n, int nb, int b)
{
    const uint64_t n_lo = n / nb, rem = n % nb, ub = static_cast<uint64_t>(b);
    return ub * n_lo + (ub < rem ? ub : rem);
}
// how many of nb batches' tallies of nvox voxels fit side by side into budget bytes
// (one at least; voxel offsets are 32-bit on the device)
inline int tallies_within(size_t nvox, int nb, size_t budget)
{
    const size_t most = std::min(budget / (nvox * sizeof(double)), (static_cast<size_t>(1) << 32) / nvox);
    return static_cast<int>(std::min<size_t>(std::max<size_t>(most, 1), static_cast<size_t>(nb)));
}
// The request chains of a batched call, chain k of nvox[k] voxels (in the order of issue)
// on stream k mod lanes: how many of a request's batches share a launch, and the voxels
// of scratch that each stream's chains share for their tallies, `budget` bytes in all.
struct ChainPlan {
    int lanes;
    std::vector<int> group;
    std::vector<size_t> need;
};
// All of a request's batches share a launch, or as many as fit half the budget where they
// need more (a grid that large would not get them all on any number of streams).  As many
// streams as asked for are kept while the tallies of them all fit the budget, else fewer,
// two at least: 64 requests of 64^3 to 256^3 voxels, 1.28e10 histories, took 1196 ms on 64
// streams with most batches in launches of their own, 1056 ms on three with all of a
// request's in one, 1083 ms one ctd_run after another.  The sum is what has to fit: with an
// equal share for each stream one request of 256^3 voxels took 63 of 24^3 from 64 streams
// to 3, 5.5 instead of 4.1 ms on the GPU, and 24 of 64^3 in 20 batches from 25 to 2, 10.2
// instead of 8.0.
inline ChainPlan plan_chains(const std::vector<size_t> &nvox, int n_batches, int lanes, size_t budget)
{
    const int n = static_cast<int>(nvox.size());
    ChainPlan p{lanes, std::vector<int>(nvox.size()), {}};
    const size_t part = budget / static_cast<size_t>(std::min(lanes, 2));
    for (int k = 0; k < n; ++k) p.group[k] = tallies_within(nvox[k], n_batches, part);
    for (;; --p.lanes) {
        p.need.assign(p.lanes, 0);
        for (int k = 0; k < n; ++k)
            if (p.group[k] > 1) p.need[k % p.lanes] = std::max(p.need[k % p.lanes], nvox[k] * p.group[k]);
        size_t total = 0;
        for (size_t v : p.need) total += v;
        if (total <= budget / sizeof(double) || p.lanes <= 2) return p;
    }
}
// Whether a batch of a served request takes a third of the blocks per SM, so that three
// launches share every SM and one's tail, fold and stop test lie under the others'
// transport: batches that do not fill the GPU (`fill` histories), while three requests of
// such batches or more run (`running`: the batches of all that do, this one's among them).
// Eight requests of 4e6 histories a batch 107.1 -> 102.9 ms; arriving at 60 /s, p99 0.45 ->
// 0.33 s at the same p50.  (With the first in line on the whole GPU 104.0 ms; two requests
// at a third each would leave SMs idle.)  Beside requests that fill the GPU a small one
// keeps the whole grid, as the first in line should: a request of 24 batches of 4e6
// beside two and three such took 49.4 and 49.2 ms (on a third 50.7 and 52.4), one of 1e6 a
// batch 36.7 and 36.3 (38.4 and 37.4).
inline bool shares_sms(double batch, const std::vector<double> &running, double fill)
{
    return batch < fill && std::count_if(running.begin(), running.end(), [&](double b) { return b < fill; }) >= 3;
}
// fold of batches [b0, b0 + k) of the problem of n histories in nb batches from tally[k][nvox]
ctd::FoldBatches fold_of(const Phantom &P, uint64_t n, int nb, int b0, int k, double *tally, bool clear);
// one transport launch over histories [h0, h1) of n in nb batches (set_range), bracketed
// by timing events 2 ev_index and 2 ev_index + 1
// (trace: per-history records of histories trace_h0 .. trace_h0 + trace_n - 1, or nullptr)
// on stream s (null: the context's) with claim counter work (null: the phantom's first),
// cleared here unless it is 0 already
int transport(ctd_ctx *ctx, Phantom &P, ctd::RequestDesc &q, uint64_t n, int nb, uint64_t h0, uint64_t h1,
              double *tally, uint32_t stride, size_t ev_index, uint4 *trace = nullptr, uint64_t trace_h0 = 0,
              uint64_t trace_n = 0, cudaStream_t s = nullptr, unsigned long long *work = nullptr,
              bool clear_work = true);
// device arrays into host memory, waited for
struct ReadPart {
    void *dst;
    const void *src;
    size_t bytes;
};
int read_back(ctd_ctx *ctx, const ReadPart *parts, int n_parts);
double now_s();
int transport_time(ctd_ctx *ctx, size_t n_launch, double &t);
// counts and results of several phantoms read back through pinned staging
int collect_many(ctd_ctx *ctx, Phantom *const *ps, int n, size_t n_launch, double t0_wall,
                 const double *t0_each = nullptr, cudaStream_t stream = nullptr);
int collect(ctd_ctx *ctx, Phantom &P, size_t n_launch, double t0_wall);

}  // namespace host
}  // namespace ctd
