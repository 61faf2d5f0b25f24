// ctd_transport.cu -- photon transport kernel of the dose engine (sm_103a).
//
// Persistent grid.  Warps claim runs of consecutive histories from a global
// counter, so a warp works on one 1 keV spectrum interval at a time
// (Sec. 2.2.5).  Each warp keeps a queue of source photons in shared memory,
// filled 32 at a time by the whole warp (source sampling, Secs. 2.2.4-2.2.6);
// a lane whose history has ended takes the next photon from the queue.  A lane
// then runs up to flight_cap Woodcock flights against mu_max(E) (Sec. 2.1),
// stopping at a real interaction, which it carries out: photoelectric or
// Compton deposition into the FP64 tally as L2 reductions, polar angle from the
// C or R surface (Secs. 2.2.2-2.2.3), rotation and binary64 renormalisation.
// Per-step event counts live in registers, the rest of a lane's counts in its
// shared-memory slot.
//
// One kernel template, four forms: one request without a fluence map, one
// request with one (its source path compiled only there), both with the request
// in the kernel's parameter space; and many requests at once, without or with
// maps (warps walk through a request table, one request at a time, its
// descriptor in shared memory, its tables read through L1).
#include "ctd_device.cuh"

namespace ctd {
namespace {

using namespace dev;

struct Photon {
    float x, y, z;    // position in voxel units: (r - box origin) / voxel size per axis
    float ux, uy, uz, e;
    uint64_t h;       // its history, in launches of several requests, else the history's
    HistKey key;      // part of its random numbers
    uint32_t tally;   // first voxel of its batch's tally (single-request launches)
    uint32_t step;
    int j;            // energy node of e, its fraction and 1 / the majorant there;
    float te, imax;   // they change only with e
};

// Philox block of (history, step, stream) of request q
__device__ __forceinline__ U4 draw(const RequestDesc &q, uint64_t h, uint32_t step, uint32_t stream)
{
    return philox_rk(static_cast<uint32_t>(h), static_cast<uint32_t>(h >> 32), step, stream, q.rk);
}

// A transport block of a photon.  A single-request launch's histories share the upper
// word of their index (the host splits a launch where it changes), so the photon
// carries its history's part of the first two rounds: 18 products a block instead of
// 20.  CBCT water 14.94 -> 14.58 ms per 2e8 histories, head 24.25 -> 24.07.
template <bool kMulti>
__device__ __forceinline__ U4 draw_step(const RequestDesc &q, const Photon &ph)
{
    return kMulti ? draw(q, ph.h, ph.step, kStreamTransport) : philox_step(ph.key, ph.step, q.k0, q.rk);
}

// the photon's history (for the records of a trace launch)
template <bool kMulti>
__device__ __forceinline__ uint64_t history(const RequestDesc &q, const Photon &ph)
{
    return kMulti ? ph.h : (static_cast<uint64_t>(q.h_hi) << 32) | hist_of(ph.key, q.rk);
}

// energy node, fraction and inverse majorant of the photon's energy
__device__ __forceinline__ void set_energy(Photon &ph, const SharedTables &sh, const float *__restrict__ s_mm)
{
    ph.j = enode(ph.e, sh.e_min, sh.n_e, ph.te);
    const float m0 = s_mm[ph.j], m1 = s_mm[ph.j + 1];
    ph.imax = 1.0f / __fmaf_rn(ph.te, m1 - m0, m0);
}

// How a photon's flight through the phantom ends, as counted by a lane; misses are
// the source photons that end in none of these.
enum { kNotEnded = -1, kDonePe, kDoneCutoff, kDoneEscaped, kDoneTerminated, kDoneAborted, kDoneKinds };

// A lane's counts of ended histories, energy totals and the real interactions of
// its current photon, in shared memory: they change at most a few times per
// history, and registers are what bounds the kernel's residency.
struct LaneSlot {
    unsigned long long e_emitted, e_escaped;   // keV * 2^23
    uint32_t done[kDoneKinds];
    uint32_t nreal;                            // real interactions of the current photon
};
static_assert(sizeof(LaneSlot) == 40, "LaneSlot layout");

// Event counts of a lane: scatters and the Woodcock steps of ended histories in
// registers, the rest in the lane's slot.  Fictitious events are not counted: each
// step ends in exactly one of escape, fictitious, PE, Compton or Rayleigh.
struct LaneCounts {
    uint32_t steps, compton, rayleigh;
    LaneSlot *me;
    __device__ __forceinline__ void clear()
    {
        steps = compton = rayleigh = 0;
        me->e_emitted = 0;
        me->e_escaped = 0;
#pragma unroll
        for (int i = 0; i < kDoneKinds; ++i) me->done[i] = 0;
    }
    __device__ __forceinline__ void emitted(float e) { me->e_emitted += kev_fixed(e); }
    // the history ended after n steps with energy e left (counted as escaped unless
    // the last event deposited it)
    __device__ __forceinline__ void end(int how, uint32_t n, float e)
    {
        ++me->done[how];
        steps += n;
        if (how >= kDoneEscaped) me->e_escaped += kev_fixed(e);
    }
};

// Per-history records of a trace launch (kTrace instantiations only): each
// history writes its own record, so no two lanes write the same one.
struct Tracer {
    uint4 *rec;
    uint64_t h0, n;
    // the last real interaction: its type and voxel
    __device__ __forceinline__ void last(uint64_t h, int type, uint32_t idx) const
    {
        const uint64_t i = h - h0;
        if (i < n) {
            rec[i].x = (rec[i].x & 0xffu) | (static_cast<uint32_t>(type + 1) << 8);
            rec[i].z = idx;
        }
    }
    // how the history ended, its steps and the energy the ending event deposited
    __device__ __forceinline__ void end(uint64_t h, int code, uint32_t steps, float e) const
    {
        const uint64_t i = h - h0;
        if (i < n) {
            rec[i].x = (rec[i].x & 0xff00u) | static_cast<uint32_t>(code + 1);
            rec[i].y = steps;
            rec[i].w = __float_as_uint(e);
        }
    }
};

// A warp's counts added to a request's totals: warp sums, one atomic per
// counter (energies as 128-bit fixed-point totals).  `sourced` is the warp's number
// of source photons.  Leaves the counts cleared.
__device__ __forceinline__ void flush_warp(DeviceCounts *dst, LaneCounts &c, uint64_t sourced, int lane)
{
    __syncwarp();
    const LaneSlot &m = *c.me;
    unsigned long long v[kDoneKinds + 3] = {m.done[kDonePe],         m.done[kDoneCutoff],  m.done[kDoneEscaped],
                                            m.done[kDoneTerminated], m.done[kDoneAborted], c.steps,
                                            c.compton,               c.rayleigh};
    unsigned long long em = m.e_emitted, es = m.e_escaped;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int i = 0; i < kDoneKinds + 3; ++i) v[i] += __shfl_down_sync(kFull, v[i], o);
        em += __shfl_down_sync(kFull, em, o);
        es += __shfl_down_sync(kFull, es, o);
    }
    if (lane == 0 && sourced) {
        const unsigned long long steps = v[kDoneKinds], compton = v[kDoneKinds + 1], rayleigh = v[kDoneKinds + 2];
        const unsigned long long ended =
            v[kDonePe] + v[kDoneCutoff] + v[kDoneEscaped] + v[kDoneTerminated] + v[kDoneAborted];
        atomicAdd(&dst->n[kCntPe], v[kDonePe]);
        atomicAdd(&dst->n[kCntCompton], compton);
        atomicAdd(&dst->n[kCntRayleigh], rayleigh);
        atomicAdd(&dst->n[kCntFict], steps - v[kDonePe] - v[kDoneEscaped] - compton - rayleigh);
        atomicAdd(&dst->n[kCntEscaped], v[kDoneEscaped]);
        atomicAdd(&dst->n[kCntMissed], sourced - ended);
        atomicAdd(&dst->n[kCntCutoff], v[kDoneCutoff]);
        atomicAdd(&dst->n[kCntTerminated], v[kDoneTerminated]);
        atomicAdd(&dst->n[kCntAborted], v[kDoneAborted]);
        atomicAdd(&dst->n[kCntSteps], steps);
        const unsigned long long o1 = atomicAdd(&dst->e_fix[0], em);
        if (o1 + em < o1) atomicAdd(&dst->e_fix[1], 1ull);
        const unsigned long long o2 = atomicAdd(&dst->e_fix[2], es);
        if (o2 + es < o2) atomicAdd(&dst->e_fix[3], 1ull);
    }
    c.clear();
    __syncwarp();
}

__device__ __forceinline__ int bin_search(const uint64_t *pref, int nbins, uint64_t local)
{
    // largest bin j with pref[j] <= local
    int lo = 0, hi = nbins - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&pref[mid]) <= local) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Source photon of history h of request q, history `local` of its batch, whose bin
// starts are `pref`; `bin` is a lower bound of its 1 keV interval.  Returns true if
// the photon enters the phantom.
//
// A fifth of CBCT water's instructions.  Each lookup is one vector (an interval's
// bounds, a projection's angle and height, an alias column), three random lines a
// photon fewer, and a photon that misses is worked out to its end and dropped instead
// of leaving its warp early: CBCT water 14.60 -> 14.37 and 14.18 ms per 2e8 histories,
// head 24.11 -> 23.85 and 23.62, primary only 4.69 -> 4.62.
template <bool kFluence, bool kTrace>
__device__ __forceinline__ bool source(const RequestDesc &q, uint64_t h, const uint64_t *pref, uint64_t local, int bin,
                                       Photon &ph, LaneCounts &cnt, const Tracer &tr)
{
    while (bin < q.nbins - 1 && __ldg(&pref[bin + 1]) <= local) ++bin;
    const U4 b0 = draw(q, h, 0, kStreamSource);
    const float2 bounds = __ldg(&q.bins[bin]);
    const float e = __fmaf_rn(bounds.y - bounds.x, uni(b0.x), bounds.x);
    cnt.emitted(e);
    float cb = 1.0f, sb = 0.0f, zs = 0.0f;
    if (q.src_kind == CTD_SRC_ARC) {
        if (q.continuous) {
            // the angle in turns, reduced to [0, 1) (arcs may span several turns)
            const float turns = __fmaf_rn(q.awt, uni(b0.y), q.a0t);
            sincos_turns(turns - floorf(turns), cb, sb);
            zs = __fmaf_rn(q.hdz, uni(b0.y), q.hz0);
        } else {
            const uint32_t k =
                static_cast<uint32_t>((static_cast<uint64_t>(b0.y) * static_cast<uint64_t>(q.n_proj)) >> 32);
            const float4 pr = __ldg(&q.proj[k]);
            cb = pr.x;
            sb = pr.y;
            zs = pr.z;
        }
    }
    // uniform in solid angle over the field: uniform point, accepted with cos^3;
    // with a fluence map (Sec. 2.2.4): beamlet from the alias table, point uniform in it
    const float D = q.D, D2 = q.D2;
    bool accepted = false;
    float uu = 0.0f, vv = 0.0f, qq = 0.0f;
    if (kFluence && q.fl_n > 0) {
        const U4 b = draw(q, h, 1, kStreamSource);
        const uint32_t k =
            static_cast<uint32_t>((static_cast<uint64_t>(b.x) * static_cast<uint64_t>(static_cast<uint32_t>(q.fl_n))) >> 32);
        const uint2 col = __ldg(&q.fl[k]);
        const uint32_t beam = b.y < col.x ? k : col.y;
        const uint32_t iv = static_cast<uint32_t>((static_cast<uint64_t>(beam) * q.fl_magic) >> 40);
        const uint32_t iu = beam - iv * static_cast<uint32_t>(q.fl_nu);
        uu = __fmaf_rn(q.fl_du, static_cast<float>(iu) + uni(b.z), q.ulo);
        vv = __fmaf_rn(q.fl_dv, static_cast<float>(iv) + uni(b.w), q.vlo);
        qq = __fmaf_rn(vv, vv, __fmaf_rn(uu, uu, D2));
        accepted = true;
    }
    for (uint32_t t = 1; t <= kMaxTrials && !accepted; ++t) {
        const U4 b = draw(q, h, t, kStreamSource);
        uu = __fmaf_rn(q.uw, uni(b.x), q.ulo);
        vv = __fmaf_rn(q.vw, uni(b.y), q.vlo);
        qq = __fmaf_rn(vv, vv, __fmaf_rn(uu, uu, D2));
        const float c2 = D2 / qq;
        const float acc = c2 * sqrtf(c2);
        if (uni(b.z) < acc) {
            accepted = true;
            break;
        }
    }
    const float inv = 1.0f / sqrtf(qq);
    float ux, uy, uz, rx, ry, rz;
    if (q.src_kind == CTD_SRC_ARC) {
        ux = __fmaf_rn(uu, cb, -(D * sb)) * inv;
        uy = __fmaf_rn(-uu, sb, -(D * cb)) * inv;
        uz = vv * inv;
        rx = D * sb;
        ry = D * cb;
        rz = zs;
    } else {
        ux = uu * inv;
        uy = vv * inv;
        uz = D * inv;
        rx = 0.0f;
        ry = 0.0f;
        rz = -D;
    }
    // (the source direction is normalised in binary32; binary64 renormalisation
    // is for the directions made by scatters)
    // entry into the box (slab method, with the direction's reciprocals); outside is vacuum
    const float iux = 1.0f / ux, iuy = 1.0f / uy, iuz = 1.0f / uz;
    const float t0x = (q.bx0 - rx) * iux, t1x = (q.bx1 - rx) * iux;
    const float t0y = (q.by0 - ry) * iuy, t1y = (q.by1 - ry) * iuy;
    const float t0z = (q.bz0 - rz) * iuz, t1z = (q.bz1 - rz) * iuz;
    float tn = fmaxf(fmaxf(fminf(t0x, t1x), fminf(t0y, t1y)), fminf(t0z, t1z));
    const float tf = fminf(fminf(fmaxf(t0x, t1x), fmaxf(t0y, t1y)), fmaxf(t0z, t1z));
    const bool enters = accepted && tn < tf && tf > 0.0f;
    if (!enters) {
        if (accepted) cnt.me->e_escaped += kev_fixed(e);
        else cnt.end(kDoneAborted, 0, e);
        if (kTrace) tr.end(h, accepted ? kEndMissed : kEndAborted, 0, 0.0f);
    }
    tn = fmaxf(tn, 0.0f);
    // the entry point in voxel units, clamped into the box (it lies on the box's
    // surface; rounding can leave it just outside): [0, the number below n]
    ph.x = fminf(fmaxf((__fmaf_rn(tn, ux, rx) - q.bx0) * q.ix, 0.0f), __uint_as_float(__float_as_uint(q.fnx) - 1u));
    ph.y = fminf(fmaxf((__fmaf_rn(tn, uy, ry) - q.by0) * q.iy, 0.0f), __uint_as_float(__float_as_uint(q.fny) - 1u));
    ph.z = fminf(fmaxf((__fmaf_rn(tn, uz, rz) - q.bz0) * q.iz, 0.0f), __uint_as_float(__float_as_uint(q.fnz) - 1u));
    ph.ux = ux;
    ph.uy = uy;
    ph.uz = uz;
    ph.e = e;
    ph.h = h;
    return enters;
}

// Where a flight ended and the numbers its interaction needs
struct Site {
    bool inside, fictitious;
    uint32_t idx;     // voxel (phantoms hold fewer than 2^32 voxels; 0 outside the phantom)
    int m;            // material
    float y, sr;      // u1 and rho / mu_max
    uint32_t rz, rw;  // the step's random words for zeta and phi
};

// One Woodcock flight (Sec. 2.1): free path against mu_max(E), the move, the
// escape test, the voxel and whether its interaction is fictitious.  s_tab is the
// request's attenuation table.  The caller keeps ph.step below kMaxSteps (the
// history's step limit).
//
// A flight and an interaction are bound by the latency of their own instruction
// chains at eight warps per scheduler (ncu: issue active 75 %, of a warp's ten
// cycles per instruction 2.4 wait on the previous one, 0.6 on a branch), so each is
// one basic block: a photon that left the phantom looks voxel 0 up and discards
// it, all interaction types take the same path, and the compiler fills one
// chain's waits with another's instructions.  With a branch per outcome CBCT water
// took 16.70 ms of transport per 2e8 histories and the head 28.43; without,
// 15.31 and 25.03 ms (bit-identical).
template <bool kMulti, bool kWide>
__device__ __forceinline__ void flight(const SharedTables &sh, const RequestDesc &q, const float2 *__restrict__ s_tab,
                                       Photon &ph, Site &at)
{
    const U4 b = draw_step<kMulti>(q, ph);
    ph.step++;
    const float path = (-log32(uni(b.x))) * ph.imax;
    // the move in voxel units: each displacement s u_k times 1/d_k, added fused
    ph.x = __fmaf_rn(path * ph.ux, q.ix, ph.x);
    ph.y = __fmaf_rn(path * ph.uy, q.iy, ph.y);
    ph.z = __fmaf_rn(path * ph.uz, q.iz, ph.z);
    const float fx = ph.x, fy = ph.y, fz = ph.z;
    // 0 <= f < n on each axis, as one unsigned compare of the bit patterns: for
    // floats other than -0 it is the same test (negative floats and NaNs have the
    // sign bit or an all-ones exponent, so larger patterns than n), and a position
    // is never -0 (the entry point is clamped to +0 at least, and adding a nonzero
    // or +0 displacement to a value other than -0 never gives -0)
    at.inside = __float_as_uint(fx) < __float_as_uint(q.fnx) && __float_as_uint(fy) < __float_as_uint(q.fny) &&
                __float_as_uint(fz) < __float_as_uint(q.fnz);
    uint32_t idx;
    if (kWide) {
        idx = at.inside ? static_cast<uint32_t>(static_cast<int>(fx)) +
                              static_cast<uint32_t>(q.nx) *
                                  (static_cast<uint32_t>(static_cast<int>(fy)) +
                                   static_cast<uint32_t>(q.ny) * static_cast<uint32_t>(static_cast<int>(fz)))
                        : 0u;
    } else {
        // the integer parts from additions rounded toward zero; idx0 takes their
        // exponent bits off (all modulo 2^32)
        idx = __float_as_uint(trunc_up(fx)) + static_cast<uint32_t>(q.nx) * __float_as_uint(trunc_up(fy)) +
              q.nxy * __float_as_uint(trunc_up(fz)) + q.idx0;
        idx = at.inside ? idx : 0u;
    }
    // one gather: the material in the top 4 bits, the density's exponent rebased.  The
    // low 28 bits read as binary32 are the density times 2^-kRhoExpBias (0 for 0, else
    // normal), so one exact multiplication restores it.
    const uint32_t w = __ldg(&q.vox[idx]);
    at.idx = idx;
    at.m = static_cast<int>(w >> 28);
    const float rho = __uint_as_float(w & 0x0fffffffu) * kRhoScale;
    // interaction type with probabilities mu_i / mu_max: fictitious when u1 is at or
    // above the total share.  The table's first plane holds the total share and its
    // difference to the next node.
    const float2 T = s_tab[at.m * sh.n_e + ph.j];
    at.y = uni(b.y);
    at.sr = rho * ph.imax;
    at.fictitious = at.inside && !(at.y < at.sr * __fmaf_rn(ph.te, T.y, T.x));
    at.rz = b.z;
    at.rw = b.w;
}

// A real interaction: the type (the first cumulative share above u1, from c1 and c2
// of both nodes in the table's second plane), the C/R-surface polar angle, local
// deposition, rotation.  Returns how the history ended, or kNotEnded.  Straight-line
// code for all types (see flight): a Rayleigh event is a scatter with E' = E (which
// deposits 0 and leaves node and majorant as they were), and an absorbed photon's
// angle is discarded.  kAnyMode: the request may limit the real interactions
// (CTD_MODE_MAX_REAL), where most histories end here and skip the rest; full
// transport is compiled without that branch (with it 2 % slower on CBCT water, while
// a primary-only run without it was 4 % slower).
template <bool kMulti, bool kWide, bool kAnyMode, bool kTrace>
__device__ __forceinline__ int interact(const SharedTables &sh, const RequestDesc &q, const float2 *__restrict__ s_tab,
                                        const float *__restrict__ s_mm, Photon &ph, const Site &at, LaneCounts &cnt,
                                        const Tracer &tr)
{
    const float2 *t = s_tab + ((q.n_mat + at.m) * sh.n_e + ph.j);
    const float2 A = t[0], B = t[1];
    const float c1 = __fmaf_rn(ph.te, B.x - A.x, A.x);
    const float c2 = __fmaf_rn(ph.te, B.y - A.y, A.y);
    const bool pe = at.y < at.sr * c1;
    const bool compton = !pe && at.y < at.sr * c2;
    const bool rayleigh = !pe && !compton;
    const float *S = rayleigh ? q.rsurf : q.csurf;
    float mu;
    if (kWide) {
        const size_t cells = static_cast<size_t>(sh.n_e - 1) * (sh.n_zeta - 1);
        const size_t first = !rayleigh && q.cs_stride == 0 ? 0 : at.m * cells;
        mu = surface(S, first + static_cast<size_t>(ph.j) * (sh.n_zeta - 1), sh.n_zeta, ph.te, uni(at.rz));
    } else {
        const uint32_t stride = rayleigh ? sh.cells : static_cast<uint32_t>(q.cs_stride);
        mu = surface(S, static_cast<uint32_t>(at.m) * stride + static_cast<uint32_t>(ph.j) * (sh.n_zeta - 1), sh.n_zeta,
                     ph.te, uni(at.rz));
    }
    // Compton: E' = E / (1 + (E/mc^2)(1 - mu)), the electron gets E - E' (all of E
    // when E' is below the absorption energy); photoelectric absorption: all of E
    const float e = ph.e;
    const float k = e * static_cast<float>(1.0 / kMec2);
    const float ec = e / __fmaf_rn(k, 1.0f - mu, 1.0f);
    const bool cutoff = compton && ec < static_cast<float>(sh.e_min);
    const bool absorbed = pe || cutoff;
    ph.e = compton && !cutoff ? ec : e;
    const float dep = absorbed ? e : e - ph.e;
    deposit(q.tally, kMulti ? at.idx : at.idx + ph.tally, dep);
    cnt.compton += compton;
    cnt.rayleigh += rayleigh;
    int end = pe ? kDonePe : cutoff ? kDoneCutoff : kNotEnded;
    if (kAnyMode && q.mode == CTD_MODE_MAX_REAL && !absorbed && ++cnt.me->nreal >= static_cast<uint32_t>(q.max_real))
        end = kDoneTerminated;
    // (full transport takes no branch around a scatter's end: an absorbed photon's is
    // discarded)
    if (!kAnyMode || q.mode == CTD_MODE_FULL || end == kNotEnded) {
        set_energy(ph, sh, s_mm);
        rotate(ph.ux, ph.uy, ph.uz, mu, uni(at.rw));
    }
    if (kTrace) {
        const uint64_t h = history<kMulti>(q, ph);
        tr.last(h, pe ? 0 : compton ? 1 : 2, at.idx);
        if (end != kNotEnded)
            tr.end(h, pe ? kEndPe : cutoff ? kEndCutoff : kEndTerminated, ph.step, dep);
    }
    return end;
}

// Per-warp photon queue in shared memory: source photons are made 32 at a
// time by the whole warp and taken by lanes whose history has ended.
constexpr int kQueue = 48, kQueueLow = 16;
constexpr size_t kQueueBytes = 3 * kQueue * sizeof(float4);

// A warp's claim of histories [next, end) and what holds up to `lim`, the end of
// the claim or of the batch of `next`: the batch, its first history, its bin starts,
// the 1 keV interval of a history at or before `next` and the first voxel of its
// tally.  Kept in shared memory, read only when the queue is topped up.
struct WarpPool {
    uint64_t next, lim, end, first, sourced;   // sourced: histories the warp has claimed
    const uint64_t *pref;
    int batch, bin;
    uint32_t tally;
    int pad;
};

// Photons in vectors, so that one is stored or taken with three wide accesses; the
// inverse majorant is worked out by the whole warp that made the photon.  Topped up
// below 16 photons: 47 at most, and the tables, queues and slots of an SM's warps leave
// L1 more than 60 KB (with 28 KB, the largest shared-memory carve-out, CBCT water
// took 9 % longer: the gathers' lines in flight need it).
struct Queue {
    float4 *a;     // [kQueue] x, y, z (voxel units), ux
    float4 *b;     // [kQueue] uy, uz, e, 1 / mu_max(e)
    uint4 *c;      // [kQueue] the history's key and the first voxel of its batch's tally, or h (lo, hi)
    WarpPool *pool;
    template <bool kMulti>
    __device__ __forceinline__ void put(int slot, const Photon &ph) const
    {
        a[slot] = make_float4(ph.x, ph.y, ph.z, ph.ux);
        b[slot] = make_float4(ph.uy, ph.uz, ph.e, ph.imax);
        c[slot] = kMulti ? make_uint4(static_cast<uint32_t>(ph.h), static_cast<uint32_t>(ph.h >> 32), 0u, 0u)
                         : make_uint4(ph.key.a, ph.key.b, ph.key.c, ph.tally);
    }
    // all but the step; the node follows from e
    template <bool kMulti>
    __device__ __forceinline__ void get(int slot, Photon &ph, const SharedTables &sh) const
    {
        const float4 u = a[slot], v = b[slot];
        const uint4 w = c[slot];
        ph.x = u.x;
        ph.y = u.y;
        ph.z = u.z;
        ph.ux = u.w;
        ph.uy = v.x;
        ph.uz = v.y;
        ph.e = v.z;
        ph.imax = v.w;
        if (kMulti) {
            ph.h = w.x | (static_cast<uint64_t>(w.y) << 32);
        } else {
            ph.key = HistKey{w.x, w.y, w.z};
            ph.tally = w.w;
        }
        ph.j = enode(ph.e, sh.e_min, sh.n_e, ph.te);
    }
};

constexpr size_t kWarpBytes = kQueueBytes + sizeof(WarpPool) + 32 * sizeof(LaneSlot);
static_assert(kWarpBytes % 16 == 0, "a warp's shared-memory area must keep 16-byte alignment");

// All histories [q.h_begin, q.h_end) of one request, claimed by warps from q.work in
// runs of q.big, near the end of q.small.  A claim's photons carry their batch's
// tally with them, so a warp goes from one batch to the next without draining.
// Returns when the warp has no photon left.
//
// One launch per batch waited for each batch's last histories: some fifty to a
// hundred microseconds of a few deep histories and of warps with a claim of 256
// beside warps with none, which is nearly all of a small batch.  Transport of 1e5
// histories in 10 batches (32^3 water): 0.69 ms in 10 launches -> 0.071 in one; 1e6 in 7
// (51x51x32 head) 2.83 -> 0.43; 1e7 in 10 (48x48x40 head, helix) 4.31 -> 1.47; 2e8 in 2
// (CBCT water) 15.29 -> 15.00.  (With later steps and smaller claims 0.055, 0.23, 1.29 and
// 13.97.)
template <bool kMulti, bool kFluence, bool kWide, bool kAnyMode, bool kTrace>
__device__ __forceinline__ void run_request(const LaunchParams &P, const RequestDesc &q, const float2 *s_tab,
                                            const float *s_mm, const Queue &Q, int lane, LaneCounts &cnt)
{
    Tracer tr;
    tr.rec = P.trace;
    tr.h0 = P.trace_h0;
    tr.n = kTrace ? P.trace_n : 0;
    const unsigned lt_mask = (1u << lane) - 1u;
    Photon ph{};
    ph.e = static_cast<float>(P.sh.e_min);
    bool alive = false;
    bool drained = false;
    int qcount = 0;                         // photons waiting in the warp's queue
    if (lane == 0) {
        WarpPool w{};
        w.next = w.lim = w.end = q.h_begin;
        w.batch = q.b0;
        w.first = static_cast<uint64_t>(q.b0) * q.n_lo + (static_cast<uint64_t>(q.b0) < q.rem ? q.b0 : q.rem);
        *Q.pool = w;
    }
    __syncwarp();
    for (;;) {
        // top the queue up with one round of up to 32 source photons
        if (qcount < kQueueLow && !drained) {
            uint64_t next = Q.pool->next;
            if (next >= Q.pool->lim) {
                // the claim is used up, or goes on in the next batch
                uint64_t end = Q.pool->end, first = Q.pool->first;
                int batch = Q.pool->batch;
                if (next >= end) {
                    const unsigned size = end < q.h_big ? q.big : q.small;
                    unsigned long long base = 0;
                    if (lane == 0) base = atomicAdd(q.work, static_cast<unsigned long long>(size));
                    base = __shfl_sync(kFull, base, 0);
                    next = q.h_begin + base;
                    end = next + size < q.h_end ? next + size : q.h_end;
                    drained = next >= q.h_end;
                }
                if (!drained) {
                    uint64_t size = q.n_lo + (static_cast<uint64_t>(batch) < q.rem ? 1 : 0);
                    while (next - first >= size) {
                        first += size;
                        ++batch;
                        size = q.n_lo + (static_cast<uint64_t>(batch) < q.rem ? 1 : 0);
                    }
                    const uint64_t *pref = size > q.n_lo ? q.pref : q.pref + (q.nbins + 1);
                    const int bin = bin_search(pref, q.nbins, next - first);
                    __syncwarp();
                    if (lane == 0) {
                        Q.pool->sourced += next == Q.pool->next && Q.pool->end == end ? 0 : end - next;
                        Q.pool->next = next;
                        Q.pool->end = end;
                        Q.pool->lim = end < first + size ? end : first + size;
                        Q.pool->first = first;
                        Q.pool->pref = pref;
                        Q.pool->batch = batch;
                        Q.pool->bin = bin;
                        Q.pool->tally = static_cast<uint32_t>(batch - q.b0) * q.tally_stride;
                    }
                    __syncwarp();
                }
            }
            if (!drained) {
                const uint64_t avail = Q.pool->lim - next;
                const unsigned take = avail < 32 ? static_cast<unsigned>(avail) : 32u;
                // the lanes' own photons wait in the queue's free slots meanwhile, so that
                // source sampling has the registers to itself
                const int mine = qcount + lane;
                Q.put<kMulti>(mine, ph);
                __syncwarp();
                Photon np;
                bool ok = false;
                if (lane < take)
                    ok = source<kFluence, kTrace>(q, next + lane, Q.pool->pref, next - Q.pool->first + lane,
                                                         Q.pool->bin, np, cnt, tr);
                const unsigned okm = __ballot_sync(kFull, ok);
                Q.get<kMulti>(mine, ph, P.sh);
                __syncwarp();
                if (ok) {
                    set_energy(np, P.sh, s_mm);
                    if (!kMulti) {
                        np.key = hist_key(static_cast<uint32_t>(np.h), q.rk);
                        np.tally = Q.pool->tally;
                    }
                    Q.put<kMulti>(qcount + __popc(okm & lt_mask), np);
                }
                qcount += __popc(okm);
                if (lane == 0) Q.pool->next = next + take;
            }
            __syncwarp();
        }
        // lanes without a photon take one from the queue
        const unsigned need = __ballot_sync(kFull, !alive);
        const int npop = __popc(need) < qcount ? __popc(need) : qcount;
        if (!alive) {
            const int rank = __popc(need & lt_mask);
            if (rank < npop) {
                const int slot = qcount - 1 - rank;
                Q.get<kMulti>(slot, ph, P.sh);
                ph.step = 0;
                if (kAnyMode) cnt.me->nreal = 0;
                alive = true;
            }
        }
        qcount -= npop;
        __syncwarp();
        if (!__any_sync(kFull, alive)) {
            if (drained && qcount == 0) break;
            continue;
        }
        if (alive) {
            // flights until a real interaction, the escape or flight_cap flights; then the
            // interaction.  A run stops short of the history's step limit; a history that
            // has reached it is aborted when its next run would start.  The step count
            // itself ends the loop (a counter beside it took head 23.62 instead of 23.19 ms
            // per 2e8 histories, CBCT water 14.20 instead of 13.98), and the test for the
            // limit stays in front of the loop: without an if around it the compiler let
            // the lanes leave the loop one by one into the interaction (36.2 ms).
            int end = kNotEnded;
            const uint32_t capped = ph.step + static_cast<uint32_t>(P.flight_cap);
            const uint32_t stop = capped < kMaxSteps ? capped : kMaxSteps;
            if (ph.step >= kMaxSteps) {
                end = kDoneAborted;
                if (kTrace) tr.end(history<kMulti>(q, ph), kEndAborted, ph.step, 0.0f);
            } else {
                Site at;
                do {
                    flight<kMulti, kWide>(P.sh, q, s_tab, ph, at);
                } while (at.fictitious && ph.step < stop);
                if (!at.inside) {
                    end = kDoneEscaped;
                    if (kTrace) tr.end(history<kMulti>(q, ph), kEndEscaped, ph.step, 0.0f);
                } else if (!at.fictitious) {
                    end = interact<kMulti, kWide, kAnyMode, kTrace>(P.sh, q, s_tab, s_mm, ph, at, cnt, tr);
                }
            }
            // every way a history ends meets here, so that its lanes are counted together
            if (end != kNotEnded) {
                cnt.end(end, ph.step, ph.e);
                alive = false;
            }
        }
    }
}

// the two table planes are 16 n_mat n_e bytes in all
__device__ __forceinline__ void load_tables(const RequestDesc &q, int n_e, float4 *s_tab, float *s_mm)
{
    const int ntab = q.n_mat * n_e;
    for (int i = threadIdx.x; i < ntab; i += blockDim.x) s_tab[i] = reinterpret_cast<const float4 *>(q.tab)[i];
    for (int i = threadIdx.x; i < n_e; i += blockDim.x) s_mm[i] = q.mmax[i];
}

// Single request (kForm 0 or 1): the request lives in the kernel's parameter
// space, its attenuation table and majorant are copied into shared memory.
// Several requests: each warp works on one request at a time with a copy of its
// descriptor in shared memory and its tables read through L1, and when that
// request has no history left to claim the warp moves on to the next one by
// itself, so that one request's tail overlaps the next one's start without the
// block waiting for its slowest warp.
// kForm: 0 one request without a fluence map, 1 one request with a fluence map
// (the map's source path is compiled only into this form, so that it does not
// cost the open-field form registers), 2 several requests without maps, 3 several
// requests of which some have a map (checked per request).  The multi-request
// forms take each request's Philox round keys from its descriptor in shared
// memory.
// kTrace (single-request forms): also write each history's record to P.trace.
constexpr int kReqWords = sizeof(RequestDesc) / 16;

template <int kMaxThreads, int kMinBlocks, int kForm, bool kWide, bool kAnyMode, bool kTrace>
__global__ void __launch_bounds__(kMaxThreads, kMinBlocks) transport_kernel(const LaunchParams P)
{
    extern __shared__ float4 smem[];
    const int n_e = P.sh.n_e;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr bool kMulti = kForm >= 2;
    // single: the tables, then the warps' queues; several: per warp, a descriptor and
    // the queue
    float4 *s_tab = smem;
    float *s_mm = reinterpret_cast<float *>(smem + P.sh.max_n_mat * n_e);
    float4 *w_req4 = smem + warp * (kReqWords + kWarpBytes / 16);
    unsigned char *wbase = kMulti ? reinterpret_cast<unsigned char *>(w_req4 + kReqWords)
                                  : reinterpret_cast<unsigned char *>(smem + P.sh.max_n_mat * n_e + (n_e + 3) / 4) +
                                        warp * kWarpBytes;
    Queue Q;
    Q.a = reinterpret_cast<float4 *>(wbase);
    Q.b = Q.a + kQueue;
    Q.c = reinterpret_cast<uint4 *>(Q.b + kQueue);
    Q.pool = reinterpret_cast<WarpPool *>(wbase + kQueueBytes);
    LaneCounts cnt;
    cnt.me = reinterpret_cast<LaneSlot *>(wbase + kQueueBytes + sizeof(WarpPool)) + lane;
    cnt.clear();

    if (!kMulti) {
        load_tables(P.one, n_e, s_tab, s_mm);
        __syncthreads();
        run_request<false, kForm == 1, kWide, kAnyMode, kTrace>(P, P.one, reinterpret_cast<const float2 *>(s_tab), s_mm, Q, lane, cnt);
        flush_warp(P.one.counts, cnt, Q.pool->sourced, lane);
        return;
    }
    // every warp starts at the first request and walks forward to the next request
    // with histories left, so that the warps of an SM mostly work on one request
    // (its phantom and tally stay in L2) and a request's tail overlaps the next one's
    // start
    const RequestDesc &q = *reinterpret_cast<const RequestDesc *>(w_req4);
    int r = 0;
    for (;;) {
        int found = -1;
        if (lane == 0) {
            for (int rr = r; rr < P.n_req; ++rr) {
                const RequestDesc &c = P.reqs[rr];
                const unsigned long long claimed = *reinterpret_cast<volatile unsigned long long *>(c.work);
                if (c.h_begin + claimed < c.h_end) {
                    found = rr;
                    break;
                }
            }
        }
        found = __shfl_sync(kFull, found, 0);
        if (found < 0) break;
        const float4 *src = reinterpret_cast<const float4 *>(P.reqs + found);
        for (int i = lane; i < kReqWords; i += 32) w_req4[i] = src[i];
        __syncwarp();
        run_request<true, kForm == 3, kWide, true, false>(P, q, reinterpret_cast<const float2 *>(q.tab), q.mmax, Q, lane, cnt);
        flush_warp(q.counts, cnt, Q.pool->sourced, lane);
        __syncwarp();
        // the same request is exhausted now; continue the walk from it
        r = found;
    }
}

__global__ void sample_mu_kernel(const float *surf, int n_zeta, int n_e, int e_min, float e, uint64_t seed,
                                 uint64_t n, double *out)
{
    float te;
    const int j = enode(e, e_min, n_e, te);
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const U4 b = block(seed, i, 0, kStreamSampler);
        out[i] = static_cast<double>(surface(surf, static_cast<size_t>(j) * (n_zeta - 1), n_zeta, te, uni(b.x)));
    }
}

__global__ void eval_math_kernel(int fn, const float *x, float *out, size_t n)
{
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        if (fn == 0) {
            out[i] = log32(x[i]);
        } else if (fn == 2) {
            out[i] = uni(__float_as_uint(x[i]));
        } else {
            float c, s;
            sincos_turns(x[i], c, s);
            out[2 * i] = c;
            out[2 * i + 1] = s;
        }
    }
}

template <int kMaxThreads, int kMinBlocks, int kForm, bool kWide = false, bool kAnyMode = false, bool kTrace = false>
int launch_t(const LaunchParams &p, int grid, int block, size_t smem, cudaStream_t stream,
             const L2Window *win = nullptr)
{
    auto *k = transport_kernel<kMaxThreads, kMinBlocks, kForm, kWide, kAnyMode, kTrace>;
    if (smem > 48 * 1024) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
            return CTD_ECUDA;
    }
    if (!win) {
        k<<<grid, block, smem, stream>>>(p);
        return cudaGetLastError() == cudaSuccess ? CTD_OK : CTD_ECUDA;
    }
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeAccessPolicyWindow;
    attr.val.accessPolicyWindow.base_ptr = win->base;
    attr.val.accessPolicyWindow.num_bytes = win->bytes;
    attr.val.accessPolicyWindow.hitRatio = win->hit_ratio;
    attr.val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    attr.val.accessPolicyWindow.missProp = cudaAccessPropertyNormal;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, k, p) != cudaSuccess) return CTD_ECUDA;
    return cudaGetLastError() == cudaSuccess ? CTD_OK : CTD_ECUDA;
}

template <int kForm>
int launch_m(const LaunchParams &p, int grid, int block, int threads_per_sm, size_t smem, cudaStream_t s,
             const L2Window *win)
{
    // the register budget follows the residency asked for (65536 registers per SM)
    if constexpr (kForm < 2)
        if (block > 256) return launch_t<384, 3, kForm>(p, grid, block, smem, s, win);
    if (block <= 128 && threads_per_sm >= 896) return launch_t<128, 7, kForm>(p, grid, block, smem, s, win);
    if (threads_per_sm >= 1024) return launch_t<256, 4, kForm>(p, grid, block, smem, s, win);
    return launch_t<256, 3, kForm>(p, grid, block, smem, s, win);
}

}  // namespace

size_t transport_smem_bytes(const LaunchParams &p, int threads)
{
    // several requests: per warp, a descriptor and the queue
    if (p.n_req > 0) return static_cast<size_t>(threads / 32) * (kReqWords * sizeof(float4) + kWarpBytes);
    return (static_cast<size_t>(p.sh.max_n_mat) * p.sh.n_e + (p.sh.n_e + 3) / 4) * sizeof(float4) +
           static_cast<size_t>(threads / 32) * kWarpBytes;
}

// persistent grids: a few blocks per SM
constexpr int kMaxGrid = 1 << 16;

// Kernel variants by residency: 3 blocks of 384 threads per SM cap it at 56
// registers, 4 of 256 at 64, 7 blocks of 128 at 73, fewer at 85.  Blocks of more than
// 256 threads: full transport of one request, without records or wide indices.
int launch_transport(const LaunchParams &p, int grid, int block, int threads_per_sm, void *stream,
                     const L2Window *win)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool large = p.n_req == 0 && !p.trace && !p.sh.wide && p.one.mode == CTD_MODE_FULL;
    if (grid <= 0 || grid > kMaxGrid || block <= 0 || block > (large ? 384 : 256) || block % 32 != 0) {
        set_error("transport launch shape out of range");
        return CTD_EINVAL;
    }
    const size_t smem = transport_smem_bytes(p, block);
    if (p.trace) {
        // trace launches (validation): one instantiation per source form, at 64 registers
        if (p.n_req > 0) {
            set_error("trace launches take one request");
            return CTD_EINVAL;
        }
        if (p.sh.wide) return launch_t<256, 3, 1, true, true, true>(p, grid, block, smem, s);
        return p.one.fl_n > 0 ? launch_t<256, 4, 1, false, true, true>(p, grid, block, smem, s)
                              : launch_t<256, 4, 0, false, true, true>(p, grid, block, smem, s);
    }
    // general index arithmetic (wide_index): one instantiation per form, whatever the residency
    // (2e7 histories on an axis of 2^23 + 1 voxels 1.70 ms a call at 4 blocks of 256 threads
    // per SM, 1.74 at 7 of 128, 1.79 at 3 of 256; the branching kernel that every phantom
    // took before, compiled for each residency, 2.05, 2.11 and 2.15)
    if (p.sh.wide) return p.n_req > 0 ? launch_t<256, 3, 3, true, true>(p, grid, block, smem, s, win)
                                      : launch_t<256, 3, 1, true, true>(p, grid, block, smem, s, win);
    // a limit on real interactions: likewise (64 registers suit every residency; interact)
    if (p.n_req == 0 && p.one.mode != CTD_MODE_FULL)
        return p.one.fl_n > 0 ? launch_t<256, 4, 1, false, true>(p, grid, block, smem, s, win)
                              : launch_t<256, 4, 0, false, true>(p, grid, block, smem, s, win);
    if (p.n_req > 0) return p.any_fluence ? launch_m<3>(p, grid, block, threads_per_sm, smem, s, win)
                                           : launch_m<2>(p, grid, block, threads_per_sm, smem, s, win);
    return p.one.fl_n > 0 ? launch_m<1>(p, grid, block, threads_per_sm, smem, s, win)
                          : launch_m<0>(p, grid, block, threads_per_sm, smem, s, win);
}

int launch_sample_mu(const float *surf, int n_zeta, int n_e, int e_min, float e, uint64_t seed, uint64_t n,
                     double *out, void *stream)
{
    sample_mu_kernel<<<1024, 256, 0, static_cast<cudaStream_t>(stream)>>>(surf, n_zeta, n_e, e_min, e, seed, n, out);
    return cudaGetLastError() == cudaSuccess ? CTD_OK : CTD_ECUDA;
}

int launch_eval_math(int fn, const float *x, float *out, size_t n, void *stream)
{
    eval_math_kernel<<<1024, 256, 0, static_cast<cudaStream_t>(stream)>>>(fn, x, out, n);
    return cudaGetLastError() == cudaSuccess ? CTD_OK : CTD_ECUDA;
}

}  // namespace ctd
