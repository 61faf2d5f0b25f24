// ctd_device.cuh -- device arithmetic of the transport (sm_103a), shared by the
// transport kernels: Philox4x32-10, the uniform mapping, the logarithm and
// sincos, float/double bit conversions, the binary64 direction
// renormalisation, the rotation after a scatter, the 1 keV node lookup and the
// R/C-surface lookup.  The transport compiles with fast binary32 arithmetic
// (hardware reciprocal, square root, logarithm and sincos; multiply-adds
// contracted): the decisions it takes are checked history by history against
// binary64 with bounds on these errors.  Binary64 stays exact.
#pragma once

#include <cuda_runtime.h>

#include "ctd_internal.h"

namespace ctd {
namespace dev {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kStreamTransport = 0, kStreamSource = 1, kStreamSampler = 3;
constexpr uint32_t kMaxTrials = 1000;
constexpr uint32_t kMaxSteps = 100000000u;

// ---------------------------------------------------------------- Philox4x32-10
// Salmon, Moraes, Dror, Shaw (SC'11): ten rounds of two 32x32->64 products,
// xor with the round key, key bumped by the Weyl constants.
struct U4 {
    uint32_t x, y, z, w;
};

__device__ __forceinline__ U4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                     uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        const uint32_t n0 = hi1 ^ c1 ^ k0;
        const uint32_t n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return U4{c0, c1, c2, c3};
}

// Philox4x32-10 with the ten round keys given (rk[2r], rk[2r+1] = key + r * Weyl)
__device__ __forceinline__ U4 philox_rk(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const uint32_t *rk)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        const uint32_t n0 = hi1 ^ c1 ^ rk[2 * r];
        const uint32_t n2 = hi0 ^ c3 ^ rk[2 * r + 1];
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
    }
    return U4{c0, c1, c2, c3};
}

// Blocks (h, step, stream 0) of one history, for histories that share the upper word
// of h.  Of the first two rounds' four products only M1 step and M0 times a word made
// from it depend on the step; the others are the history's, kept as three words:
//   a = lo(M0 h) ^ k1', b = hi(M1 c2) ^ k0', c = lo(M1 c2) with c2 = hi(M0 h) ^ k1
// (k0, k1 the first round's keys, k0', k1' the second's).
struct HistKey {
    uint32_t a, b, c;
};

constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

// 1 / kPhiloxM0 modulo 2^32 (an odd number is its own inverse modulo 8; each step
// doubles the bits that are right)
constexpr uint32_t inverse32(uint32_t m)
{
    uint32_t x = m;
    for (int i = 0; i < 4; ++i) x *= 2u - m * x;
    return x;
}
constexpr uint32_t kPhiloxM0Inverse = inverse32(kPhiloxM0);
static_assert(kPhiloxM0 * kPhiloxM0Inverse == 1u, "inverse modulo 2^32");

__device__ __forceinline__ HistKey hist_key(uint32_t h, const uint32_t *rk)
{
    const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * h;
    const uint64_t p1 = static_cast<uint64_t>(kPhiloxM1) * (static_cast<uint32_t>(p0 >> 32) ^ rk[1]);
    return HistKey{static_cast<uint32_t>(p0) ^ rk[3], static_cast<uint32_t>(p1 >> 32) ^ rk[2], static_cast<uint32_t>(p1)};
}

// the lower word of the history a key was made from
__device__ __forceinline__ uint32_t hist_of(const HistKey &k, const uint32_t *rk)
{
    return (k.a ^ rk[3]) * kPhiloxM0Inverse;
}

// k0 is the first round's key ^ the upper word of h.  (The products are written as
// 64-bit ones: the compiler then takes the fewest instructions, 112 per history on the
// head against 117 with the high and low words apart.)
__device__ __forceinline__ U4 philox_step(const HistKey &k, uint32_t step, uint32_t k0, const uint32_t *rk)
{
    const uint64_t s0 = static_cast<uint64_t>(kPhiloxM1) * step;
    const uint64_t s1 = static_cast<uint64_t>(kPhiloxM0) * (static_cast<uint32_t>(s0 >> 32) ^ k0);
    uint32_t c0 = k.b ^ static_cast<uint32_t>(s0), c1 = k.c;
    uint32_t c2 = static_cast<uint32_t>(s1 >> 32) ^ k.a, c3 = static_cast<uint32_t>(s1);
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * c0, p1 = static_cast<uint64_t>(kPhiloxM1) * c2;
        c0 = static_cast<uint32_t>(p1 >> 32) ^ c1 ^ rk[2 * r];
        c2 = static_cast<uint32_t>(p0 >> 32) ^ c3 ^ rk[2 * r + 1];
        c1 = static_cast<uint32_t>(p1);
        c3 = static_cast<uint32_t>(p0);
    }
    return U4{c0, c1, c2, c3};
}

__device__ __forceinline__ U4 block(uint64_t seed, uint64_t h, uint32_t step, uint32_t stream)
{
    return philox(static_cast<uint32_t>(h), static_cast<uint32_t>(h >> 32), step, stream,
                  static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
}

// (2 (x >> 9) + 1) 2^-24: exact in binary32, never 0 or 1.  Built from bits:
// a = 1 + k 2^-23 (k = x >> 9 as the significand) minus (1 - 2^-24) is
// (2k + 1) 2^-24 exactly (2k + 1 < 2^24 fits the significand, so the one
// subtraction does not round): the same value without an integer conversion.
// One funnel shift of (127 : x) by 9 puts the exponent 127 above x >> 9.
__device__ __forceinline__ float uni(uint32_t x)
{
    return __uint_as_float(__funnelshift_r(x, 127u, 9)) - 0x1.fffffep-1f;
}

// trunc(f) + 2^23 for 0 <= f < 2^23, in one full-rate addition rounded toward
// zero (a conversion instruction runs at a quarter of the rate): its bit pattern
// is kTruncBits + trunc(f), and taking 2^23 off again is exact.
// Used for the voxel, the node and the surface cell, with the uniform and the density
// decoded in one instruction less each: CBCT water, 2e8 histories, transport 16.88 ->
// 16.70 ms; head 28.67 -> 28.43 ms; results bit-identical.
constexpr float kTrunc = 8388608.0f;
constexpr uint32_t kTruncBits = kTruncPattern;
__device__ __forceinline__ float trunc_up(float f) { return __fadd_rz(f, kTrunc); }

// 2^kRhoExpBias, which takes a packed density back to its value
constexpr float kRhoScale = 0x1p108f;
static_assert(kRhoExpBias == 108, "kRhoScale is 2^kRhoExpBias");

// ---------------------------------------------------------------- log and sincos
// The hardware approximations (the SFU's base-2 logarithm and sine/cosine).
// Measured against binary64 over every uniform the transport draws: ln u within
// 1.9e-6 absolutely (a free path -ln(u)/mu_max is then off by at most
// 1.9e-6/mu_max cm), cos and sin of 2 pi t within 3.4e-7.
__device__ __forceinline__ float log32(float x) { return __logf(x); }

// cos and sin of 2 pi t for t in [0, 1): of 2 pi (t - 1/2) in [-pi, pi), where
// the approximation holds its accuracy, negated
__device__ __forceinline__ void sincos_turns(float t, float &c, float &s)
{
    float sn, cs;
    __sincosf((t - 0.5f) * 6.2831853071795865f, &sn, &cs);
    c = -cs;
    s = -sn;
}

// |f| of a direction component (|f| < 2) widened to binary64 with three integer
// instructions and no branch (GB300's FP64 pipe is narrow; this keeps conversions
// off it): the exponent's top bit is clear, so rebiasing it by 896 = 0x380 sets
// bits that are free.  Exact for normal numbers; zeros and subnormals give some
// number below 2^-125, whose square leaves the sum below as it is.
__device__ __forceinline__ double widen_abs(float f)
{
    const uint32_t u = __float_as_uint(f);
    return __hiloint2double(static_cast<int>(((u >> 3) & 0x07ffffffu) | 0x38000000u), static_cast<int>(u << 29));
}

// binary64 of magnitude below 1 -> binary32 by truncating the significand to 23
// bits (round toward zero); magnitudes below 2^-126 give 0.  With the biased
// exponent at 897..1022 its low seven bits are the binary32 one's.
__device__ __forceinline__ float trunc32(double d)
{
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(d));
    const uint32_t lo = static_cast<uint32_t>(__double2loint(d));
    const uint32_t m = __funnelshift_l(lo, hi, 3);
    const uint32_t f = (m & 0x3fffffffu) | (hi & 0x80000000u);
    return __uint_as_float((hi & 0x7fffffffu) < (897u << 20) ? 0u : f);
}

// Back to unit length after a scatter: d = n2 - 1, the squared norm's excess,
// in binary64 with three fused multiply-adds, ((y^2 - 1) + x^2) + z^2, from the
// widened components (each square is exact in binary64); the correction
// e = -d/2 of one Newton step c = 1.5 - 0.5 n2 for 1/sqrt(n2) from 1 is d
// truncated to binary32 times -1/2, applied to each component with one fused
// multiply-add.
// Bound by issue slots and by the wait for the narrow FP64 pipe, not by its rate:
// the widening and truncation around the three multiply-adds were some forty
// instructions with branches, now fifteen without.  CBCT water, 2e8 histories:
// transport 18.44 -> 16.88 ms; head 30.12 -> 28.67 ms; results bit-identical.
__device__ __forceinline__ void renorm(float &ux, float &uy, float &uz)
{
    const double dx = widen_abs(ux), dy = widen_abs(uy), dz = widen_abs(uz);
    const double d = __fma_rn(dz, dz, __fma_rn(dx, dx, __fma_rn(dy, dy, -1.0)));
    const float ef = trunc32(d) * -0.5f;
    ux = __fmaf_rn(ux, ef, ux);
    uy = __fmaf_rn(uy, ef, uy);
    uz = __fmaf_rn(uz, ef, uz);
}

// E 2^23 as an integer: exact for 1 keV <= E < 2^40 keV (every photon energy of
// the transport is at least the node floor e_min >= 1 keV)
__device__ __forceinline__ unsigned long long kev_fixed(float e)
{
    const uint32_t u = __float_as_uint(e);
    const unsigned long long m = (u & 0x7fffffu) | 0x800000u;
    return m << ((u >> 23) - 127u);
}

// binary32 -> binary64 for positive normal numbers only: the exponent rebiased and
// the significand moved into place (the general widen() without its branches)
__device__ __forceinline__ double widen_normal(float f)
{
    const uint32_t u = __float_as_uint(f);
    const uint32_t hi = (((u >> 23) + 896u) << 20) | ((u & 0x7fffffu) >> 3);
    return __hiloint2double(static_cast<int>(hi), static_cast<int>(u << 29));
}

// Tally deposit of a non-negative binary32 energy into the binary64 grid, as a
// global reduction that returns nothing (a fire-and-forget L2 atomic), also
// when the grid's address was read from shared memory.  A positive deposit is a
// normal number: a photon energy (at least 1 keV) or the difference of two
// energies of at least 1 keV, which is a multiple of their binary32 ulp.
__device__ __forceinline__ void deposit(double *tally, size_t idx, float e)
{
    if (e > 0.0f)
        asm volatile("red.global.add.f64 [%0], %1;" ::"l"(__cvta_generic_to_global(tally + idx)),
                     "d"(widen_normal(e)));
}

// New direction after a scatter of polar cosine mu and azimuth 2 pi tphi.  Both
// cases are computed and one is selected: no branch interrupts the schedule.
__device__ __forceinline__ void rotate(float &ux, float &uy, float &uz, float mu, float tphi)
{
    const float st = sqrtf(fmaxf(__fmaf_rn(-mu, mu, 1.0f), 0.0f));
    float cp, sp;
    sincos_turns(tphi, cp, sp);
    const float a2 = __fmaf_rn(ux, ux, uy * uy);
    const bool axis = a2 < static_cast<float>(1e-12);   // along z: the general case divides by a
    const float a = sqrtf(a2);
    const float rr = st / a;
    const float nx = __fmaf_rn(rr, __fmaf_rn(ux * uz, cp, -(uy * sp)), ux * mu);
    const float ny = __fmaf_rn(rr, __fmaf_rn(uy * uz, cp, ux * sp), uy * mu);
    const float nz = __fmaf_rn(-(a * st), cp, uz * mu);
    const float zz = uz > 0.0f ? mu : -mu;
    ux = axis ? st * cp : nx;
    uy = axis ? st * sp : ny;
    uz = axis ? zz : nz;
    renorm(ux, uy, uz);
}

// energy node j and fraction te on the 1 keV grid (e >= e_min, n_e <= 10^5)
__device__ __forceinline__ int enode(float e, int e_min, int n_e, float &te)
{
    const float fe = e - static_cast<float>(e_min);
    const float t = fminf(trunc_up(fe), kTrunc + static_cast<float>(n_e - 2));
    te = fe - (t - kTrunc);
    return static_cast<int>(__float_as_uint(t) - kTruncBits);
}

// bilinear lookup of mu(zeta, E) (Sec. 2.2.2) on a surface whose row j of cells
// starts at S; a surface is held as cells of the four corners of a lookup,
// [n_e - 1][n_zeta - 1] float4, so one 16-byte read fetches them.  Cell is
// uint32_t where every cell index of the launch fits, else size_t.
template <class Cell>
__device__ __forceinline__ float surface(const float *__restrict__ S, Cell row, int n_zeta, float te, float z)
{
    const float zf = __fmul_rn(z, static_cast<float>(n_zeta - 1));   // rounded on its own, never fused
    const float t = fminf(trunc_up(zf), kTrunc + static_cast<float>(n_zeta - 2));
    const float a = zf - (t - kTrunc);
    const float4 c = __ldg(reinterpret_cast<const float4 *>(S) + (row + (__float_as_uint(t) - kTruncBits)));
    const float a0 = c.x, a1 = c.y, b0 = c.z, b1 = c.w;
    const float lo = __fmaf_rn(a, a1 - a0, a0);
    const float hi = __fmaf_rn(a, b1 - b0, b0);
    const float mu = __fmaf_rn(te, hi - lo, lo);
    return fminf(fmaxf(mu, -1.0f), 1.0f);
}

}  // namespace dev
}  // namespace ctd
