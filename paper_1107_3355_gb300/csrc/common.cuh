// Device-side building blocks of the GB300 gDPM engine: random numbers,
// geometry helpers and the data layouts shared by the transport kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "gdpm.h"

namespace gdpm {

constexpr int kMaxMat = GDPM_MAX_MATERIALS;
constexpr int kMaxBins = GDPM_MAX_BINS;
constexpr double kMC2 = 0.51099895;           // electron rest energy, MeV
constexpr float kMC2f = 0.51099895f;
constexpr float kTwoPi = 6.28318530717958647f;

// ---------------------------------------------------------------- status bits
enum : uint32_t {
    ST_QUEUE_OVERFLOW = 1u,
    ST_ITER_CAP = 2u,
    ST_PHASE_CAP = 4u,          // the device-driven phase loop reached its phase cap
    ST_BOUNDS = 8u,             // checked build: an index was out of range (class below)
    ST_B_VOXEL = 1u << 8,       //   phantom voxel
    ST_B_TALLY = 1u << 9,       //   tally cell
    ST_B_TABLE = 1u << 10,      //   material / beamlet table row
    ST_B_QUEUE = 1u << 11,      //   queue slot
    ST_B_RECORD = 1u << 12,     //   per-history record
};

// Checked build (compiled with GDPM_CHECKED=1): an index is tested against
// its range before use.  One out of range sets ST_BOUNDS and its class bit
// and is replaced by 0, so the access stays in bounds and the call returns
// GDPM_E_BOUNDS.  In the normal build the check and its range expression
// vanish.
#ifndef GDPM_CHECKED
#define GDPM_CHECKED 0
#endif
#if GDPM_CHECKED
__device__ __noinline__ inline void bounds_fail(uint32_t* status, uint32_t cls) {
    atomicOr(status, ST_BOUNDS | cls);
}
#define GDPM_IDX(status, i, n, cls) ((i) < (n) ? (i) : (bounds_fail((status), (cls)), decltype(i)(0)))
#else
#define GDPM_IDX(status, i, n, cls) (i)
#endif

// ---------------------------------------------------------------- counters
// Slots of the device counter array (uint64).  Names follow gdpm_stats.
enum {
    C_PRIMARY = 0, C_PH_CREATED, C_PH_TERMINATED, C_PH_FLIGHTS, C_PH_REAL, C_COMPTON,
    C_PHOTO, C_PAIR, C_EL_CREATED, C_EL_TERMINATED, C_EL_STEPS, C_MOLLER, C_BREMS,
    C_ANNIHIL, C_LOCAL_DEP, C_PUSH_PH, C_PUSH_EL, C_POP_PH, C_POP_EL, C_CROSS, C_NCOUNT
};
// Slots of the device FP64 ledger.
enum { L_SOURCE = 0, L_DEPOSITED, L_ESCAPED, L_DISCARDED, L_DMAX, L_SIGSUM, L_SIGCNT, L_NLEDGER };

// ---------------------------------------------------------------- Philox4x32-10
// Salmon et al., SC'11: ten rounds; each round multiplies words 0 and 2 by
// fixed 32-bit constants (64-bit products), mixes the halves with words 1
// and 3 and the round key, and bumps the key by two Weyl constants.
__host__ __device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = uint64_t(0xD2511F53u) * c.x, p1 = uint64_t(0xCD9E8D57u) * c.z;
        c = make_uint4(uint32_t(p1 >> 32) ^ c.y ^ k0, uint32_t(p1), uint32_t(p0 >> 32) ^ c.w ^ k1, uint32_t(p0));
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// The ten round keys of a key (k0, k1), and a block with round keys made
// before (they are the same for every block of a run).
struct RoundKeys {
    uint2 k[10];
};
__host__ __device__ __forceinline__ RoundKeys round_keys(uint32_t k0, uint32_t k1) {
    RoundKeys r;
    for (int i = 0; i < 10; ++i) {
        r.k[i] = make_uint2(k0, k1);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return r;
}
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const RoundKeys& K) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = uint64_t(0xD2511F53u) * c.x, p1 = uint64_t(0xCD9E8D57u) * c.z;
        c = make_uint4(uint32_t(p1 >> 32) ^ c.y ^ K.k[r].x, uint32_t(p1), uint32_t(p0 >> 32) ^ c.w ^ K.k[r].y,
                       uint32_t(p0));
    }
    return c;
}

// 23-bit uniform in the open interval (0,1): (floor(x/2^9) + 1/2) / 2^23,
// exactly representable in FP32, so it never rounds to 0 or 1.  The top 23
// bits become the mantissa of a float in [1, 2) (one funnel shift), and
// subtracting 1 - 2^-24 is exact.
__device__ __forceinline__ float u01(uint32_t x) {
    return __uint_as_float(__funnelshift_r(x, 0x7Fu, 9)) - 0.999999940395355224609375f;
}

// Id of the k-th banked secondary: the SplitMix64 output function
// (Steele, Lea, Flood 2014) applied to parent ^ (k+1)*golden.
__host__ __device__ __forceinline__ uint64_t child_id(uint64_t parent, uint32_t k) {
    const uint64_t golden = 0x9E3779B97F4A7C15ull;
    uint64_t z = (parent ^ (uint64_t(k + 1) * golden)) + golden;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// ---------------------------------------------------------------- particle state
// Register copy of one particle (flags as above).
struct Part {
    float x, y, z, u, v, w, E;
    int ix, iy, iz;
    uint32_t hist, pidlo, pidhi, ctr, flags;
};
constexpr uint32_t kPositron = 0x80000000u;
// flags: bits 0..15 count the secondaries a particle has banked (the child
// index of the next one), bits 16..30 its tally slot (the batch of its
// history when batches run side by side; beamlet x batch in a dose-matrix
// run), bit 31 marks a positron.
constexpr uint32_t kChildMask = 0xFFFFu;
constexpr uint32_t kBatchShift = 16, kBatchMask = 0x7FFF0000u;
constexpr int kMaxConcurrentBatches = 128;
constexpr int kMaxSlots = 32767;

// One Philox block for the transport kernels.  Out of line (it has no
// warp-synchronous operations), so its ten unrolled rounds exist once in
// the kernel instead of at every draw site.
static __device__ __noinline__ uint4 philox_block(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                           uint32_t k0, uint32_t k1) {
    return philox4x32_10(make_uint4(c0, c1, c2, c3), k0, k1);
}

__device__ __forceinline__ float4 draw(Part& p, uint32_t k0, uint32_t k1) {
    const uint4 r = philox_block(p.hist, p.pidlo, p.pidhi, p.ctr, k0, k1);
    ++p.ctr;
    return make_float4(u01(r.x), u01(r.y), u01(r.z), u01(r.w));
}

// Particle queue: a record of three (a banked particle) or two (a primary)
// 16-byte words per slot, read and written with 16-byte accesses.
//   banked:  x y z E | u v w voxel | history, particle id lo, hi, flags
//   primary: x y z E | u v w flags
// A banked particle has made no draw yet (draw counter 0).  A primary's
// history is its phase's first plus its slot, its particle id 1, its draw
// counter 1 and its voxel follows from its position.  E < 0 marks an empty
// slot.  bank() writes the banked ones.  A record is written once and read once, with streaming accesses: the
// L2 is for the phantom and the tallies (CT plan photon phase -3 %).
// One address and three loads per refill, where 13 arrays of one word
// took 13 of each: CT plan, photon phase 23.9 -> 22.5 ms, electron phase
// 31.7 -> 30.1 ms (1e8 histories).
struct Queue {
    uint4* rec;
    uint32_t capacity;
};
constexpr int kQueueWords = 12;
constexpr int kSourceWords = 8;

__device__ __forceinline__ uint4 pack4(float a, float b, float c, uint32_t d) {
    return make_uint4(__float_as_uint(a), __float_as_uint(b), __float_as_uint(c), d);
}
__device__ __forceinline__ void queue_mark_empty(const Queue& q, uint32_t s) {
    q.rec[size_t(s) * (kQueueWords / 4)].w = __float_as_uint(-1.f);
}
__device__ __forceinline__ void queue_load(const Queue& q, uint32_t s, Part& p) {
    const uint4* r = q.rec + size_t(s) * (kQueueWords / 4);
    const uint4 a = __ldcs(r), b = __ldcs(r + 1), c = __ldcs(r + 2);
    p.x = __uint_as_float(a.x); p.y = __uint_as_float(a.y); p.z = __uint_as_float(a.z);
    p.E = __uint_as_float(a.w);
    p.u = __uint_as_float(b.x); p.v = __uint_as_float(b.y); p.w = __uint_as_float(b.z);
    p.ix = int(b.w & 1023u); p.iy = int((b.w >> 10) & 1023u); p.iz = int(b.w >> 20);
    p.hist = c.x; p.pidlo = c.y; p.pidhi = c.z; p.flags = c.w;
    p.ctr = 0u;
}
__device__ __forceinline__ void source_store(const Queue& q, uint32_t s, const Part& p) {
    uint4* r = q.rec + size_t(s) * (kSourceWords / 4);
    __stcs(&r[0], pack4(p.x, p.y, p.z, __float_as_uint(p.E)));
    __stcs(&r[1], pack4(p.u, p.v, p.w, p.flags));
}
__device__ __forceinline__ void source_mark_empty(const Queue& q, uint32_t s) {
    q.rec[size_t(s) * (kSourceWords / 4)].w = __float_as_uint(-1.f);
}
__device__ __forceinline__ void source_load(const Queue& q, uint32_t s, Part& p) {
    const uint4* r = q.rec + size_t(s) * (kSourceWords / 4);
    const uint4 a = __ldcs(r), b = __ldcs(r + 1);
    p.x = __uint_as_float(a.x); p.y = __uint_as_float(a.y); p.z = __uint_as_float(a.z);
    p.E = __uint_as_float(a.w);
    p.u = __uint_as_float(b.x); p.v = __uint_as_float(b.y); p.w = __uint_as_float(b.z);
    p.flags = b.w;
    p.pidlo = 1u; p.pidhi = 0u; p.ctr = 1u;
}

// ---------------------------------------------------------------- Metropolis chains
// Most steps a chain takes when C chains share n consecutive histories, and
// the tiles of `tile` steps they fill.  Quotients first: n may reach 2^32 - 1
// and C 2^24, so rounding up by adding to n would wrap.
__host__ __device__ __forceinline__ uint32_t chain_steps(uint32_t n, uint32_t C) { return n / C + (n % C != 0u); }
__host__ __device__ __forceinline__ uint32_t chain_tiles(uint32_t n, uint32_t C, uint32_t tile) {
    const uint32_t most = chain_steps(n, C);
    return most / tile + (most % tile != 0u);
}

// ---------------------------------------------------------------- geometry
// Rotate (u,v,w) by polar cosine `cost` and azimuth phi given as (cp, sp).
// Azimuth reference: e1 = (u w, v w, -(1-w^2))/s, e2 = (-v, u, 0)/s with
// s = sqrt(1-w^2); for s^2 < 1e-10 the x and y axes.  The result is
// renormalised.  Which products are fused is spelled out, here and wherever a
// sum of two products decides a history: left to the compiler it changes
// with the surrounding code, and a history's result with it.  TURNED: the
// Moller primary, whose (cp, sp) are the delta ray's negated, fuses the
// other product of each pair.
template <bool TURNED = false>
__device__ __forceinline__ void rotate(float& u, float& v, float& w, float cost, float cp, float sp) {
    const float sint = sqrtf(fmaxf(0.f, fmaf(-cost, cost, 1.f)));
    const float s2 = fmaf(-w, w, 1.f);
    float un, vn, wn;
    if (s2 < 1e-10f) {
        un = cost * u + sint * cp;
        vn = cost * v + sint * sp;
        wn = cost * w;
    } else {
        const float s = sqrtf(s2);
        const float is = 1.f / s;
        const float cu = __fmul_rn(cp, u), cv = __fmul_rn(cp, v);
        // a = cp u w - sp v, b = cp v w + sp u
        const float a = TURNED ? fmaf(cu, w, -__fmul_rn(sp, v)) : fmaf(-sp, v, __fmul_rn(cu, w));
        const float b = TURNED ? fmaf(sp, u, __fmul_rn(cv, w)) : fmaf(cv, w, __fmul_rn(sp, u));
        un = fmaf(cost, u, __fmul_rn(__fmul_rn(sint, a), is));
        vn = fmaf(cost, v, __fmul_rn(__fmul_rn(sint, b), is));
        wn = fmaf(cost, w, -__fmul_rn(__fmul_rn(sint, cp), s));
    }
    const float n = rsqrtf(fmaf(wn, wn, fmaf(un, un, __fmul_rn(vn, vn))));
    u = __fmul_rn(un, n); v = __fmul_rn(vn, n); w = __fmul_rn(wn, n);
}

// cos and sin of 2*pi*r for r in (0,1): evaluated at the angle 2*pi*r - pi in
// [-pi, pi] where the hardware approximations are accurate, then negated.
__device__ __forceinline__ void cossin_2pi(float r, float& c, float& s) {
    float sn, cs;
    __sincosf(kTwoPi * r - 3.14159265358979f, &sn, &cs);
    c = -cs;
    s = -sn;
}

// ---------------------------------------------------------------- device tables
struct DevTables {
    int n_mat, n_e, n_r, n_a;
    float l2min, inv_dl2;                // energy grid: u = (log2 E - l2min) * inv_dl2
    const float* ph_tot;                 // [m][i] total attenuation per unit density
    const float2* ph_cum;                // [m][i] {mu_c, mu_c + mu_pe}
    const float4* el;                    // [m][i] {R, x_ms, Sigma_moller, Sigma_brems}
    const float* rinv;                   // [m][j] T(r_j), r_j = rlo_m + j/rinv_idr_m
    const float* atab;                   // [k] ln A at ln G1 = a_l1lo + k/a_idl
    float a_l1lo, a_idl, a_g1hi;
    float x0[kMaxMat], inv_x0[kMaxMat], sigmax[kMaxMat], inv_sigmax[kMaxMat];
    float r_eabs[kMaxMat], rinv_lo[kMaxMat], rinv_idr[kMaxMat];
    float eabs_ph, eabs_el, ms_keep;      // ms_keep = 1 - ms_loss
    int flags;
};

// Energy -> table cell (i, f), linear interpolation in ln E (Sec. 2.2.2).
__device__ __forceinline__ void grid_pos(const DevTables& T, float E, int& i, float& f) {
    const float uu = (__log2f(E) - T.l2min) * T.inv_dl2;
    const float fl = floorf(uu);
    i = min(max(int(fl), 0), T.n_e - 2);
    f = fminf(fmaxf(uu - float(i), 0.f), 1.f);
}
__device__ __forceinline__ float lerpf(float a, float b, float f) { return fmaf(f, b - a, a); }

// ---------------------------------------------------------------- warp helpers
__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }
__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

}  // namespace gdpm
