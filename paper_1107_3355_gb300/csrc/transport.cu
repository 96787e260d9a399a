// Transport kernels of the gDPM method on sm_103a.
//
// Photon and electron transport run in separate phases (Sec. 2.2.1: only
// one particle type is in flight at a time; secondaries go to per-type
// stacks).  Each phase is one persistent launch.  A warp works in rounds:
//   flight / step round: every lane advances its own particle, a photon by
//             one Woodcock flight against the majorant, an electron by a
//             condensed-history step (CSDA loss over the step, random hinge
//             multiple scattering, voxel walk depositing along the path) or a
//             part of its walk (Sec. 2.1);
//   event round: what the particles of a step round ran into (Compton,
//             photoelectric and pair events; hard-event candidates, Moller
//             trials, bremsstrahlung, annihilation) happens to few of a
//             warp's lanes at a time, so those particles wait in the warp's
//             stack in shared memory and are taken 32 at a time, one draw
//             each; their secondaries are banked with full-warp ballots.
// A lane whose particle waits or has ended takes another from the stack, which
// is refilled from the phase's input (freshly generated primaries, then the
// queue of banked particles), so warps stay full until the input is drained.
// Tables live in shared memory (but the electrons' largest where it would
// crowd out warps, kFarWarps) and are read by linear interpolation (Sec.
// 2.2.2); random numbers come from Philox4x32-10 keyed per history and
// particle, so results do not depend on scheduling.
#include <algorithm>
#include <cfloat>

#include "internal.h"

namespace gdpm {
namespace {

constexpr float kInf = FLT_MAX;
constexpr float kEs = 21.2f;            // Rossi-Greisen scattering energy, MeV
constexpr uint32_t kFull = 0xffffffffu;

// CTA shape each phase kernel is compiled for: threads per CTA and the
// resident CTAs per SM that fix its register budget.  A warp's stack takes
// 4.6 KB (photons) or 7.0 KB (electrons) of shared memory, so one CTA stages
// the tables once and leaves the L1 what it can.  Photons: 896 threads and 72
// registers, which wide phases fill (kNarrowThreads for the others); 1e8 CT
// histories take 16.8 ms of photon phases instead of 17.9 at 768 and 17.1 at
// 1024 (64 registers), the lung slab's 2.5e8 25.2 instead of 27.0 and 24.8.
// Electrons at 896 lose 5-8 %, at 640 4 %.
#ifndef GDPM_THREADS_PHOTON
#define GDPM_THREADS_PHOTON 896
#endif
#ifndef GDPM_MIN_CTAS_PHOTON
#define GDPM_MIN_CTAS_PHOTON 1
#endif
#ifndef GDPM_THREADS_ELECTRON
#define GDPM_THREADS_ELECTRON 768
#endif
#ifndef GDPM_MIN_CTAS_ELECTRON
#define GDPM_MIN_CTAS_ELECTRON 1
#endif
template <int PT>
struct PhaseShape {
    static constexpr int threads = PT == 0 ? GDPM_THREADS_PHOTON : GDPM_THREADS_ELECTRON;
    static constexpr int ctas = PT == 0 ? GDPM_MIN_CTAS_PHOTON : GDPM_MIN_CTAS_ELECTRON;
};

// ---------------------------------------------------------------- ledger/tally
struct Acc {
    double src, esc;
};

// Secondaries created by one step: n of them (0..2) at the particle's
// current position; the second is a positron (pair) or, for photons, the
// back-to-back partner (annihilation).
struct Sec {
    int n;
    bool photon, pos2;
    float E1, E2, dx, dy, dz;
};

// Forms of the phase kernels: FP64 tally or FP32 pair tally, without
// per-history records, and the general form, which looks at both at every
// deposit and event.
constexpr int kPlain = 0, kPair = 1, kGeneral = 2;

// Deposit e MeV in voxel vox of the tally of the batch in `flags`.
// FP32 pair: hi accumulates, lo collects the exact rounding error of each
// addition (TwoSum on the value the atomic returned); the second half
// (tally_end) can come after other work, which then hides the atomic's return
// trip.
struct Deposit {
    size_t vox;
    float e, old;
};
template <int GEN>
__device__ __forceinline__ Deposit tally_begin(const SimParams& P, uint32_t flags, uint32_t vox0, float e) {
    size_t vox = uint64_t((flags & kBatchMask) >> kBatchShift) * P.batch_stride + vox0;
#if GDPM_CHECKED
    if (vox < P.tally_lo || vox >= P.tally_hi) {
        bounds_fail(P.status, ST_B_TALLY);
        vox = P.tally_lo;
    }
#endif
    Deposit d{vox, e, 0.f};
    if (GEN == kPlain || (GEN == kGeneral && P.tally_mode == 0)) atomicAdd(&P.edep[vox], double(e));
    else d.old = atomicAdd(&P.edep_hi[vox], e);
    return d;
}
template <int GEN>
__device__ __forceinline__ void tally_end(const SimParams& P, const Deposit& d) {
    if (GEN == kPlain || (GEN == kGeneral && P.tally_mode == 0)) return;
    const float s = d.old + d.e;
    const float bb = s - d.old;
    const float err = (d.old - (s - bb)) + (d.e - bb);
    if (err != 0.f) atomicAdd(&P.edep_lo[d.vox], err);
}
template <int GEN>
__device__ __forceinline__ void tally(const SimParams& P, uint32_t flags, uint32_t vox0, float e) {
    tally_end<GEN>(P, tally_begin<GEN>(P, flags, vox0, e));
}

__device__ __forceinline__ uint32_t vox_of(const SimParams& P, int ix, int iy, int iz) {
    return uint32_t(ix) + uint32_t(P.nx) * (uint32_t(iy) + uint32_t(P.ny) * uint32_t(iz));
}

template <int GEN>
__device__ __forceinline__ void hist_count(const SimParams& P, uint32_t hist, int k) {
    if (GEN == kGeneral && P.hrec) atomicAdd(&P.hrec[size_t(GDPM_IDX(P.status, hist, P.n_records, ST_B_RECORD)) * 4 + k], 1);
}
template <int GEN>
__device__ __forceinline__ void hist_add(const SimParams& P, uint32_t hist, int k, double v) {
    if (GEN == kGeneral && P.hrec) atomicAdd(&P.hrecd[size_t(GDPM_IDX(P.status, hist, P.n_records, ST_B_RECORD)) * 2 + k], v);
}
#if GDPM_CHECKED
__device__ __forceinline__ uint32_t n_voxels(const SimParams& P) {
    return uint32_t(P.nx) * uint32_t(P.ny) * uint32_t(P.nz);
}
#endif

// ---------------------------------------------------------------- samplers
// Klein-Nishina in eps = E'/E by the two-branch mixture method: with weight
// ln(1/eps0) sample from 1/eps, with weight (1-eps0^2)/2 from eps, accept
// with 1 - eps sin^2(theta)/(1+eps^2).  Draws: (branch, eps, accept, phi).
__device__ __forceinline__ bool kn_trial(uint4 r, float E, float& eps, float& cost, float& rphi) {
    const float k = E * (1.f / kMC2f);
    const float e0 = 1.f / fmaf(2.f, k, 1.f);
    const float a1 = -__logf(e0), a2 = 0.5f * (1.f - e0 * e0);
    const float4 c = make_float4(u01(r.x), u01(r.y), u01(r.z), u01(r.w));
    if (c.x * (a1 + a2) < a1) eps = __expf(-a1 * c.y);
    else eps = sqrtf(fmaf(1.f - e0 * e0, c.y, e0 * e0));
    const float t = (1.f - eps) / (k * eps);
    const float g = 1.f - eps * t * (2.f - t) / fmaf(eps, eps, 1.f);
    rphi = c.w;
    cost = 1.f - t;
    return c.z <= g;
}
// A whole Klein-Nishina event (checks of the sampler).
__device__ __forceinline__ void sample_kn(Part& p, const SimParams& P, float E, float& eps,
                                          float& cost, float& rphi) {
    for (int it = 0; it < 4096; ++it)
        if (kn_trial(philox_block(p.hist, p.pidlo, p.pidhi, p.ctr++, P.key0, P.key1), E, eps, cost, rphi))
            break;
}

// Moller: eps = W/T on [W_cc/T, 1/2] from the 1/eps^2 proposal, accepted with
// eps^2 f(eps) / (2 + c1/4).  Draws: (eps, accept, phi, -).
__device__ __forceinline__ bool moller_trial(uint4 x, float T, float wcc, float& eps, float& rphi) {
    const float tau = T * (1.f / kMC2f);
    const float g = tau / (tau + 1.f);
    const float c1 = g * g, c2 = (2.f * tau + 1.f) / ((tau + 1.f) * (tau + 1.f));
    const float ec = wcc / T;
    const float bound = 2.f + 0.25f * c1;
    const float4 w = make_float4(u01(x.x), u01(x.y), u01(x.z), u01(x.w));
    eps = ec / (1.f - w.x * (1.f - 2.f * ec));
    const float y = eps / (1.f - eps);
    const float gg = 1.f + y * y + c1 * eps * eps - c2 * y;
    rphi = w.z;
    return w.y * bound <= gg;
}
// A whole Moller event (checks of the sampler).
__device__ __forceinline__ void sample_moller(Part& p, const SimParams& P, float T, float wcc, float& eps,
                                              float& rphi) {
    for (int it = 0; it < 4096; ++it)
        if (moller_trial(philox_block(p.hist, p.pidlo, p.pidhi, p.ctr++, P.key0, P.key1), T, wcc, eps, rphi))
            break;
}

// Sauter's K-shell photoelectron distribution (physics variant) in
// mu = cos(theta), for kinetic energy T: p(mu) ~ (1-mu^2)/(1-beta mu)^4
// [1 + b (1 - beta mu)], b = gamma(gamma-1)(gamma-2)/2.  Proposal
// q(mu) ~ 1/(1 - beta mu)^2 by inversion, 1/(1 - beta mu) = 1/(1+beta) +
// xi 2beta/(1-beta^2); accepted with (1-mu^2)(1-beta^2)/(1-beta mu)^2 times
// g/g_max.  Draws per trial: (proposal, accept, phi, -).
__device__ __forceinline__ void sample_sauter(Part& p, const SimParams& P, float T, float& mu,
                                              float& rphi) {
    const float g = 1.f + T * (1.f / kMC2f);
    const float beta = sqrtf(fmaxf(0.f, 1.f - 1.f / (g * g)));
    const float b = 0.5f * g * (g - 1.f) * (g - 2.f);
    const float gmax = b >= 0.f ? 1.f + b * (1.f + beta) : 1.f + b * (1.f - beta);
    const float ib = 1.f / (1.f + beta), sc = 2.f * beta / (1.f - beta * beta);
    mu = 0.f;
    rphi = 0.f;
    for (int it = 0; it < 4096; ++it) {
        const float4 c = draw(p, P.key0, P.key1);
        const float x = ib + c.x * sc;
        const float m = fminf(fmaxf((1.f - 1.f / x) / beta, -1.f), 1.f);
        const float d = 1.f - beta * m;
        const float w = (1.f - m * m) * (1.f - beta * beta) / (d * d) * (1.f + b * d) / gmax;
        mu = m;
        rphi = c.z;
        if (c.y < w) break;
    }
}

// Screening parameter A for first moment G1 (table in ln G1; asymptote
// 1/A = 3d(1 + 3d/2), d = 1 - G1, near isotropy).
__device__ __forceinline__ float screening_A(const DevTables& T, const float* atab, float G1) {
    if (G1 > T.a_g1hi) {
        const float d = 1.f - G1;
        return 1.f / (3.f * d * (1.f + 1.5f * d));
    }
    float kk = (__logf(G1) - T.a_l1lo) * T.a_idl;
    kk = fmaxf(kk, 0.f);
    const int k = min(int(kk), T.n_a - 2);
    const float f = fminf(kk - float(k), 1.f);
    return __expf(lerpf(atab[k], atab[k + 1], f));
}

// ---------------------------------------------------------------- geometry
__device__ __forceinline__ bool inside(const SimParams& P, float x, float y, float z) {
    return x >= 0.f && x <= P.Lx && y >= 0.f && y <= P.Ly && z >= 0.f && z <= P.Lz;
}

__device__ __forceinline__ void voxel_of(const SimParams& P, Part& p) {
    p.ix = min(int(p.x * P.inv_dx), P.nx - 1);
    p.iy = min(int(p.y * P.inv_dy), P.ny - 1);
    p.iz = min(int(p.z * P.inv_dz), P.nz - 1);
}

// Move a primary from outside onto the phantom surface (ray-box slabs); the
// entry coordinate is set exactly on the face.  False if the ray misses.
__device__ __forceinline__ bool enter_box(const SimParams& P, Part& p) {
    if (inside(P, p.x, p.y, p.z)) return true;
    const float o[3] = {p.x, p.y, p.z}, d[3] = {p.u, p.v, p.w}, L[3] = {P.Lx, P.Ly, P.Lz};
    float tmin = -kInf, tmax = kInf;
    int amin = -1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (d[a] == 0.f) {
            if (o[a] < 0.f || o[a] > L[a]) return false;
            continue;
        }
        const float t1 = (0.f - o[a]) / d[a], t2 = (L[a] - o[a]) / d[a];
        const float lo = fminf(t1, t2), hi = fmaxf(t1, t2);
        if (lo > tmin) { tmin = lo; amin = a; }
        if (hi < tmax) tmax = hi;
    }
    if (amin < 0 || tmax <= tmin || tmax <= 0.f) return false;
    float q[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        q[a] = fminf(fmaxf(fmaf(tmin, d[a], o[a]), 0.f), L[a]);
        if (a == amin) q[a] = d[a] > 0.f ? 0.f : L[a];   // by value: an index would put the arrays in local memory
    }
    p.x = q[0]; p.y = q[1]; p.z = q[2];
    return true;
}

// Beamlet of history h as its position in the list of positive-weight
// beamlets (Sec. 2.3.1).  Metropolis picks were made by k_metropolis before
// the phase; the alias method reads the Philox block at (h, 0, 0, 0); the
// cumulative search uses the primary's own uniform rw.
__device__ __forceinline__ int pick_beamlet(const DevSource& S, const PhaseArgs& A, uint32_t idx,
                                            uint32_t h, float rw, uint32_t k0, uint32_t k1,
                                            const float* cdf) {
    if (S.sampler == GDPM_SAMPLE_METROPOLIS) return int(A.bl_pick[idx]);
    if (S.sampler == GDPM_SAMPLE_ALIAS) {
        const uint4 w = philox_block(h, 0u, 0u, 0u, k0, k1);
        const int J = int(__umulhi(w.x, uint32_t(S.n_beamlets)));
        return uint64_t(w.y) < S.al_cut[J] ? J : S.al_alias[J];   // u = (w.y + 1/2) 2^-32 < cut
    }
    // the I with P(I) <= r < P(I+1) (rounded-up FP32 table: the same decisions
    // as comparing double(r) with the FP64 cumulative weights)
    int l = 0, hi = S.n_beamlets - 1;
    while (l < hi) {
        const int mid = (l + hi) >> 1;
        if (rw < cdf[mid]) hi = mid; else l = mid + 1;
    }
    return l;
}

// Primary number `idx` of this phase (Sec. 2.3): energy from the batch's
// spectrum interval allotment (uniform inside the interval), position and
// direction from the source geometry.  Draw 0 of the primary's stream:
// (u-position, v-position, energy, beamlet).
// prefix_tab / cdf_tab: copies of A.bin_prefix and S.bl_cdf (e.g. in shared
// memory), or null to read the originals.
__device__ bool make_primary(const SimParams& P, const PhaseArgs& A, uint32_t idx, Part& p,
                             Acc& acc, uint32_t inv_big, uint32_t inv_small,
                             const uint32_t* prefix_tab = nullptr, const float* cdf_tab = nullptr) {
    const DevSource& S = P.S;
    const uint32_t h = A.src_first + idx;
    // a dose-matrix run: sub-problem k holds histories [sub_first[k],
    // sub_first[k+1]); its batches are slots k*nb .. k*nb+nb-1
    uint32_t k = 0u, h0 = 0u, nb_small = A.nb_small, nb_rem = A.nb_rem;
    if (A.n_sub) {
        uint32_t lo = 0u, hi = A.n_sub;
        while (hi - lo > 1u) {
            const uint32_t mid = (lo + hi) >> 1;
            if (A.sub_first[mid] <= h) lo = mid; else hi = mid;
        }
        k = lo;
        h0 = A.sub_first[k];
        const uint32_t nk = A.sub_first[k + 1] - h0;
        nb_small = nk / A.sub_batches;
        nb_rem = nk % A.sub_batches;
    }
    // batch b of history h and h's index within it (batches are contiguous;
    // the first nb_rem hold nb_small + 1 histories)
    const uint32_t hl = h - h0;
    const uint32_t big = nb_small + 1u, split = nb_rem * big;
    // hl < split: histories of the long batches.  The quotient by the batch
    // size from its reciprocal, floor((2^32 - 1) / size), is one too small at
    // most
    const bool first = hl < split;
    const uint32_t size = first ? big : nb_small, at = first ? hl : hl - split;
    const uint32_t inv = A.n_sub ? 0xffffffffu / size : first ? inv_big : inv_small;
    uint32_t b = __umulhi(at, inv), local = at - b * size;
    if (local >= size) {
        ++b;
        local -= size;
    }
    if (!first) b += nb_rem;
    const uint32_t slot = A.n_sub ? k * A.sub_batches + b : b;
    const uint32_t* prefix = (prefix_tab ? prefix_tab : A.bin_prefix) + size_t(slot) * (S.n_bins + 1);
    p.hist = h;
    p.pidlo = 1u; p.pidhi = 0u; p.ctr = 0u;
    p.flags = (slot << kBatchShift) & kBatchMask;
    const uint4 rx = philox4x32_10(make_uint4(h, 1u, 0u, 0u), P.keys);
    ++p.ctr;
    const float4 r = make_float4(u01(rx.x), u01(rx.y), u01(rx.z), u01(rx.w));
    int lo = 0, hi = S.n_bins;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= local) lo = mid; else hi = mid;
    }
    p.E = fmaf(S.edges[lo + 1] - S.edges[lo], r.z, S.edges[lo]);
    if (S.geometry == GDPM_GEO_PENCIL) {
        p.x = S.origin[0]; p.y = S.origin[1]; p.z = S.origin[2];
        p.u = S.direction[0]; p.v = S.direction[1]; p.w = S.direction[2];
    } else {
        float src[3], cen[3], au[3], av[3];
        float a0, a1, b0, b1;
        if (S.geometry == GDPM_GEO_POINT_FIELD) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                src[a] = S.origin[a]; cen[a] = S.center[a]; au[a] = S.axis_u[a]; av[a] = S.axis_v[a];
            }
            a0 = -S.half_u; a1 = S.half_u; b0 = -S.half_v; b1 = S.half_v;
        } else {
            // a dose-matrix sub-problem is its own beamlet; otherwise sample one
            const int kb = A.n_sub ? int(k)
                                   : pick_beamlet(S, A, idx, h, r.w, P.key0, P.key1, cdf_tab ? cdf_tab : S.bl_cdf);
            // a row is 16 floats, 64 bytes from a 16-byte aligned base: four vector loads
            const float4* row = reinterpret_cast<const float4*>(S.beamlets) +
                                size_t(GDPM_IDX(P.status, kb, S.n_beamlets, ST_B_TABLE)) * 4;
            const float4 q0 = __ldg(row), q1 = __ldg(row + 1), q2 = __ldg(row + 2), q3 = __ldg(row + 3);
            src[0] = q0.x; src[1] = q0.y; src[2] = q0.z;
            cen[0] = q0.w; cen[1] = q1.x; cen[2] = q1.y;
            au[0] = q1.z; au[1] = q1.w; au[2] = q2.x;
            av[0] = q2.y; av[1] = q2.z; av[2] = q2.w;
            a0 = q3.x; a1 = q3.y; b0 = q3.z; b1 = q3.w;
        }
        const float su = fmaf(a1 - a0, r.x, a0), sv = fmaf(b1 - b0, r.y, b0);
        const float ax = fmaf(sv, av[0], fmaf(su, au[0], cen[0]));
        const float ay = fmaf(sv, av[1], fmaf(su, au[1], cen[1]));
        const float az = fmaf(sv, av[2], fmaf(su, au[2], cen[2]));
        p.x = src[0]; p.y = src[1]; p.z = src[2];
        const float dx = ax - p.x, dy = ay - p.y, dz = az - p.z;
        const float n = rsqrtf(fmaf(dz, dz, fmaf(dx, dx, __fmul_rn(dy, dy))));
        p.u = __fmul_rn(dx, n); p.v = __fmul_rn(dy, n); p.w = __fmul_rn(dz, n);
    }
    acc.src += p.E;
    if (!enter_box(P, p)) {
        acc.esc += p.E;
        hist_add<kGeneral>(P, p.hist, 0, p.E);
        return false;
    }
    voxel_of(P, p);
    return true;
}

// ---------------------------------------------------------------- photon step
struct PhSmem {
    const float* maj;
    const float* tot;
    const float2* cum;
};

// Outcome of a flight: the photon makes a virtual (delta) collision and flies
// on, leaves the phantom, or waits for its event.
enum class Flight { fly, gone, wait };

// What a waiting photon waits for is kept in its state: a photoelectric event
// sets kAbsorbed in its flags (no photon uses the positron bit), a pair has
// the sign of its energy set, a Compton event neither.
constexpr uint32_t kAbsorbed = 0x80000000u;

// One Woodcock flight against the majorant (Sec. 2.1) with the draw x.
template <int GEN>
__device__ __forceinline__ Flight photon_flight(const SimParams& P, const PhSmem& S, Part& p, uint4 x,
                                                double& esc) {
    const DevTables& T = P.T;
    int i;
    float f;
    grid_pos(T, p.E, i, f);
    const float mm = lerpf(S.maj[i], S.maj[i + 1], f);
    const float inv_mm = 1.f / mm;
    const float s = -__logf(u01(x.x)) * inv_mm;
    p.x = fmaf(s, p.u, p.x);
    p.y = fmaf(s, p.v, p.y);
    p.z = fmaf(s, p.w, p.z);
    if (!inside(P, p.x, p.y, p.z)) {
        esc += p.E;
        hist_add<GEN>(P, p.hist, 0, p.E);
        return Flight::gone;
    }
    voxel_of(P, p);
    const uint32_t vox = GDPM_IDX(P.status, vox_of(P, p.ix, p.iy, p.iz), n_voxels(P), ST_B_VOXEL);
    const int m = GDPM_IDX(P.status, int(__ldg(&P.mat[vox])), T.n_mat, ST_B_TABLE);
    const float rho = __ldg(&P.rho[vox]);
    const int mi = m * T.n_e + i;
    const float mt = lerpf(S.tot[mi], S.tot[mi + 1], f);
    if (!(u01(x.y) * mm < mt * rho)) return Flight::fly;
    hist_count<GEN>(P, p.hist, 0);
    const float2 c0 = S.cum[mi], c1 = S.cum[mi + 1];
    const float rr = u01(x.z) * mt;
    if (!(rr < lerpf(c0.x, c1.x, f))) {
        if (rr < lerpf(c0.y, c1.y, f)) {
            p.flags |= kAbsorbed;
        } else {
            p.E = -p.E;
            --p.ctr;        // the event shares the energy with this draw's last uniform
        }
    }
    return Flight::wait;
}

// The event a photon waits for, with the draw x at its counter: pair
// production (the electron takes the flight's last uniform of the kinetic
// energy, the positron the rest), photoelectric absorption (photoelectron
// along the photon, or at Sauter's angle to it, physics variant), or one
// trial of a Compton event (`force` accepts any).  After a Compton event the
// photon has turned and lost energy, with a recoil electron along
// E u - E' u', and `goes_on` says whether it stays above its absorption
// energy (below it, it is deposited here).
enum class PhEvent { none, compton, photo, pair };
template <int GEN>
__device__ __forceinline__ PhEvent photon_event(const SimParams& P, Part& p, uint4 x, bool force, bool& goes_on,
                                                Sec& sec) {
    const float E = p.E;
    sec.dx = p.u; sec.dy = p.v; sec.dz = p.w;
    sec.photon = sec.pos2 = false;
    if (E < 0.f) {
        const float tav = -E - 2.f * kMC2f;
        sec.E1 = u01(x.w) * tav;
        sec.E2 = tav - sec.E1;
        sec.n = 2;
        sec.pos2 = true;
        return PhEvent::pair;
    }
    if (p.flags & kAbsorbed) {
        p.flags &= ~kAbsorbed;
        sec.n = 1;
        sec.E1 = E;
        if (P.T.flags & GDPM_FLAG_SAUTER) {
            float mu, rphi, cp, sp;
            sample_sauter(p, P, E, mu, rphi);
            cossin_2pi(rphi, cp, sp);
            rotate(sec.dx, sec.dy, sec.dz, mu, cp, sp);
        }
        return PhEvent::photo;
    }
    ++p.ctr;
    float eps, cost, rphi;
    if (!kn_trial(x, E, eps, cost, rphi) && !force) return PhEvent::none;
    sec.n = 1;
    float cp, sp;
    cossin_2pi(rphi, cp, sp);
    rotate(p.u, p.v, p.w, cost, cp, sp);
    const float Ep = __fmul_rn(eps, E);
    sec.E1 = __fsub_rn(E, Ep);
    const float dx = fmaf(E, sec.dx, -__fmul_rn(Ep, p.u)), dy = fmaf(E, sec.dy, -__fmul_rn(Ep, p.v)),
                dz = fmaf(E, sec.dz, -__fmul_rn(Ep, p.w));
    const float en = rsqrtf(fmaf(dz, dz, fmaf(dx, dx, __fmul_rn(dy, dy))));
    sec.dx = dx * en; sec.dy = dy * en; sec.dz = dz * en;
    goes_on = !(Ep < P.T.eabs_ph);
    if (goes_on) p.E = Ep;
    else tally<GEN>(P, p.flags, vox_of(P, p.ix, p.iy, p.iz), Ep);
    return PhEvent::compton;
}

// ---------------------------------------------------------------- electron step
struct __align__(16) ElMat {      // a material's constants of a step (shared memory)
    float r_eabs, inv_sigmax, rinv_lo, rinv_idr, inv_x0, sigmax, pad[2];
};
struct ElSmem {
    const float4* el;       // in shared memory, or in global memory (FAR)
    const float* rinv;
    const float* atab;
    const ElMat* mat;
};
// Entry i of the step and event table.
template <bool FAR>
__device__ __forceinline__ float4 el_entry(const ElSmem& S, int i) {
    return FAR ? __ldg(S.el + i) : S.el[i];
}

// An electron or positron in a lane: its voxel is packed (10 bits an axis),
// pend is energy it owes to that voxel and has not tallied yet.
struct Electron {
    float x, y, z, u, v, w, E, pend;
    uint32_t vox, hist, pidlo, pidhi, ctr, flags;
};

// The condensed-history step in progress (Sec. 2.1): set up once (limits, end
// energy, hinge deflection), then its straight legs are walked through the
// voxels over one or more rounds of the phase loop.  What leg 2 needs is in
// the lane's ElStack::hinge.
struct ElStep {
    float left;        // mass thickness left in the current leg (g/cm2)
    float dpm;         // energy loss per unit mass thickness along the step
    float Tend;        // energy at the end of the step
    float dep;         // energy of the step tallied or owed to a voxel so far
    float rho;         // density of the particle's current voxel
    uint32_t what;     // bits 0-1: 0 no step in progress, 1 or 2 walking that leg; bits 2-3: what
                       // ends the step (0 reach E_abs, 1 hard candidate, 2 MS step); bits 4+: start material
};

// Outcome of a lane's round: the particle stays in its lane, its track has
// ended, or it waits for an event.
enum class Round { go, ended, wait };
// Events a waiting particle waits for.
constexpr uint32_t kCandidate = 0u, kMoller = 1u, kAnnihilation = 2u;

__device__ __forceinline__ uint32_t vox_packed(int ix, int iy, int iz) {
    return uint32_t(ix) | (uint32_t(iy) << 10) | (uint32_t(iz) << 20);
}
__device__ __forceinline__ uint32_t vox_linear(const SimParams& P, uint32_t v) {
    return (v & 1023u) + uint32_t(P.nx) * (((v >> 10) & 1023u) + uint32_t(P.ny) * (v >> 20));
}

// End of track: residual energy deposited in the voxel; a positron then waits
// to annihilate, or its rest energy is discarded (Sec. 2.1, Sec. 4).
template <int GEN>
__device__ __forceinline__ Round absorb(const SimParams& P, Electron& p, uint32_t& kind) {
    tally<GEN>(P, p.flags, vox_linear(P, p.vox), p.E + p.pend);
    p.pend = 0.f;
    if (!(p.flags & kPositron)) return Round::ended;
    if (!P.S.annihilation) {
        atomicAdd(&P.ledger[L_DISCARDED], 2.0 * kMC2);
        return Round::ended;
    }
    kind = kAnnihilation;
    return Round::wait;
}

// Set up a step with the draw x: step limits as mass thickness in the start
// voxel's material (`mat`), energy at its end, deflection at the random hinge.
template <int GEN, bool FAR>
__device__ __forceinline__ void electron_setup(const SimParams& P, const ElSmem& S, const Electron& p, uint4 x,
                                               int mat, ElStep& st, float4& hinge) {
    const DevTables& T = P.T;
    const float4 r = make_float4(u01(x.x), u01(x.y), u01(x.z), u01(x.w));
    hist_count<GEN>(P, p.hist, 1);
    const int m = GDPM_IDX(P.status, mat, T.n_mat, ST_B_TABLE);
    int i;
    float f;
    grid_pos(T, p.E, i, f);
    const int mi = m * T.n_e + i;
    const float4 a0 = el_entry<FAR>(S, mi), a1 = el_entry<FAR>(S, mi + 1);
    const float R0 = lerpf(a0.x, a1.x, f);
    const float xms = lerpf(a0.y, a1.y, f);
    const ElMat M = S.mat[m];
    const float xcut = R0 - M.r_eabs;
    const float xhard = (T.flags & GDPM_FLAG_NO_HARD) ? kInf : -__logf(r.x) * M.inv_sigmax;
    uint32_t lim;
    float xs;
    if (xcut <= xms && xcut <= xhard) { lim = 0u; xs = xcut; }
    else if (xhard <= xms) { lim = 1u; xs = xhard; }
    else { lim = 2u; xs = xms; }
    xs = fmaxf(xs, 0.f);
    float Tend;
    if (lim == 0u) {
        Tend = T.eabs_el;
    } else {
        const float rr = (R0 - xs - M.rinv_lo) * M.rinv_idr;
        const int j = min(max(int(floorf(rr)), 0), T.n_r - 2);
        const float g = fminf(fmaxf(rr - float(j), 0.f), 1.f);
        const float* ri = S.rinv + m * T.n_r;
        Tend = fminf(lerpf(ri[j], ri[j + 1], g), p.E);
    }
    const float Tk = p.E;
    const float dT = Tk - Tend;
    hist_add<GEN>(P, p.hist, 1, double(xs));
    // multiple scattering at the mid-step energy
    const float Tm = 0.5f * (Tk + Tend);
    const float pbc = Tm * (Tm + 2.f * kMC2f) / (Tm + kMC2f);
    const float q = kEs / pbc;
    const float G1 = xs * q * q * 0.5f * M.inv_x0;
    float mu;
    if (G1 >= 1.f) {
        mu = 2.f * r.z - 1.f;
    } else {
        const float Asc = screening_A(T, S.atab, G1);
        mu = 1.f - 2.f * Asc * r.z / (1.f - r.z + Asc);
    }
    float cp, sp;
    cossin_2pi(r.w, cp, sp);
    // leg 1 keeps the step's start direction, so the deflection is applied to
    // it here, with all lanes that start a step together
    float u1 = p.u, v1 = p.v, w1 = p.w;
    rotate(u1, v1, w1, mu, cp, sp);
    st.dpm = xs > 0.f ? dT / xs : 0.f;
    st.dep = 0.f;
    st.Tend = Tend;
    // random hinge: zeta x_s straight, deflect, (1 - zeta) x_s straight
    st.left = r.y * xs;
    hinge = make_float4(u1, v1, w1, (1.f - r.y) * xs);
    st.what = 1u | (lim << 2) | (uint32_t(m) << 4);
}

// Voxel walk (3-D DDA) of the step in progress, depositing dpm MeV per g/cm2
// in each voxel: along leg 1 (zeta x_s), turn to the deflected direction at
// the hinge, along leg 2 ((1 - zeta) x_s).  A track tallies once per voxel it
// visits, on leaving it (pend); the last piece of leg 2 is left to the
// caller.
struct Walk {
    float iu, iv, iw;      // 1 / direction (0 for a zero component)
    float ou, ov, ow;      // added to the distance: kInf for a zero component
    float fx, fy, fz;      // voxel indices
    uint32_t lin;          // linear voxel index
    float tb;              // distance to the exit face
    int axis;              // of the exit face
};
__device__ __forceinline__ void walk_aim(const Electron& p, Walk& k) {
    k.iu = p.u != 0.f ? 1.f / p.u : 0.f; k.ou = p.u != 0.f ? 0.f : kInf;
    k.iv = p.v != 0.f ? 1.f / p.v : 0.f; k.ov = p.v != 0.f ? 0.f : kInf;
    k.iw = p.w != 0.f ? 1.f / p.w : 0.f; k.ow = p.w != 0.f ? 0.f : kInf;
}
// Move to the end of the leg (true) or to the exit face of the voxel.
__device__ __forceinline__ bool walk_move(const SimParams& P, Electron& p, const ElStep& s, Walk& k) {
    const float tx = fmaf(fmaf(k.fx + (p.u > 0.f ? 1.f : 0.f), P.dx, -p.x), k.iu, k.ou);
    const float ty = fmaf(fmaf(k.fy + (p.v > 0.f ? 1.f : 0.f), P.dy, -p.y), k.iv, k.ov);
    const float tz = fmaf(fmaf(k.fz + (p.w > 0.f ? 1.f : 0.f), P.dz, -p.z), k.iw, k.ow);
    const bool cx = tx <= ty && tx <= tz, cy = ty <= tz;
    k.axis = cx ? 0 : cy ? 1 : 2;
    k.tb = fmaxf(cx ? tx : cy ? ty : tz, 0.f);
    const bool ends = __fmul_rn(s.rho, k.tb) >= s.left;
    const float t = ends ? s.left / s.rho : k.tb;
    p.x = fmaf(t, p.u, p.x);
    p.y = fmaf(t, p.v, p.y);
    p.z = fmaf(t, p.w, p.z);
    return ends;
}
// Cross the exit face; false when the particle leaves the phantom.
template <int GEN>
__device__ __forceinline__ bool walk_cross(const SimParams& P, Electron& p, ElStep& s, Walk& k,
                                           uint32_t& crossings) {
    const float piece = __fmul_rn(s.rho, k.tb);
    const float owed = fmaf(s.dpm, piece, p.pend);
    Deposit dep{0, 0.f, 0.f};
    if (owed > 0.f) dep = tally_begin<GEN>(P, p.flags, k.lin, owed);
    s.dep = fmaf(s.dpm, piece, s.dep);
    p.pend = 0.f;
    s.left = __fsub_rn(s.left, piece);
    ++crossings;
    const bool up = (k.axis == 0 ? p.u : k.axis == 1 ? p.v : p.w) > 0.f;
    const uint32_t n = k.axis == 0 ? P.nx : k.axis == 1 ? P.ny : P.nz;
    const uint32_t d = k.axis == 0 ? 1u : k.axis == 1 ? uint32_t(P.nx) : uint32_t(P.nx) * uint32_t(P.ny);
    const uint32_t shift = 10u * uint32_t(k.axis);
    const uint32_t at = ((p.vox >> shift) & 1023u) + (up ? 1u : ~0u);       // wraps below zero
    if (at >= n) {
        tally_end<GEN>(P, dep);
        return false;
    }
    p.vox = up ? p.vox + (1u << shift) : p.vox - (1u << shift);
    const float f = float(at);
    if (k.axis == 0) k.fx = f;
    else if (k.axis == 1) k.fy = f;
    else k.fz = f;
    k.lin = up ? k.lin + d : k.lin - d;
    k.lin = GDPM_IDX(P.status, k.lin, n_voxels(P), ST_B_VOXEL);
    s.rho = __ldg(&P.rho[k.lin]);
    tally_end<GEN>(P, dep);
    return true;
}
// One stretch of the walk: to the end of leg 1, the turn at the hinge and the
// end of leg 2, or to the next crossing on the way, so that the lanes that
// end a leg do it together and those that cross a face do that together.
// Returns 0 when the step goes on, 1 at the end of leg 2, 2 when the particle
// left the phantom.
template <int GEN>
__device__ __forceinline__ int walk_stretch(const SimParams& P, Electron& p, ElStep& s, Walk& k,
                                            const float4& hinge, uint32_t& crossings) {
    bool ends = walk_move(P, p, s, k);
    if (ends && (s.what & 3u) == 1u) {
        // the hinge: the rest of leg 1 stays owed to the current voxel
        p.pend = fmaf(s.dpm, s.left, p.pend);
        s.dep = fmaf(s.dpm, s.left, s.dep);
        const float4 h = hinge;
        p.u = h.x; p.v = h.y; p.w = h.z;
        s.what ^= 3u;                         // leg 1 -> leg 2
        s.left = h.w;
        walk_aim(p, k);
        ends = walk_move(P, p, s, k);
    }
    if (ends) return 1;
    return walk_cross<GEN>(P, p, s, k, crossings) ? 0 : 2;
}

// Stretches per round once the phase's input is drained: a lane whose step
// ends has nothing to take over, so the lanes with many crossings (air) need
// not give up the warp.
constexpr int kDrainedStretches = 16;

// A lane's round: set up a step when none is in progress (with the draw x in
// the start voxel's material `mat`), walk, and at the step's end escape, be absorbed, or wait for the
// hard-event candidate.
template <int GEN, bool FAR>
__device__ __forceinline__ Round electron_round(const SimParams& P, const ElSmem& S, Electron& p, ElStep& st,
                                                uint4 x, int mat, float4& hinge, int stretches, double& esc,
                                                uint32_t& crossings, uint32_t& kind) {
    if ((st.what & 3u) == 0u) {
        electron_setup<GEN, FAR>(P, S, p, x, mat, st, hinge);
    }
    Walk k;
    k.lin = vox_linear(P, p.vox);
    k.fx = float(p.vox & 1023u); k.fy = float((p.vox >> 10) & 1023u); k.fz = float(p.vox >> 20);
    walk_aim(p, k);
    int res = walk_stretch<GEN>(P, p, st, k, hinge, crossings);
#pragma unroll 1
    for (int n = 1; res == 0 && n < stretches; ++n) res = walk_stretch<GEN>(P, p, st, k, hinge, crossings);
    if (res == 0) return Round::go;
    st.what &= ~3u;
    if (res == 2) {
        double e = p.E - st.dep;
        if (p.flags & kPositron) {
            if (P.S.annihilation) e += 2.0 * kMC2;
            else atomicAdd(&P.ledger[L_DISCARDED], 2.0 * kMC2);
        }
        esc += e;
        hist_add<GEN>(P, p.hist, 0, e);
        return Round::ended;
    }
    // the step's remainder stays owed to the voxel the step ends in
    p.pend += (p.E - st.Tend) - st.dep;
    p.E = st.Tend;
    const uint32_t lim = (st.what >> 2) & 3u;
    if (lim == 1u) {
        kind = kCandidate | ((st.what >> 4) << 2);
        return Round::wait;
    }
    if (lim == 0u || p.E < P.T.eabs_el) return absorb<GEN>(P, p, kind);
    return Round::go;
}

// One draw of the event a particle waits for.  A hard-event candidate is
// accepted with Sigma_h(T)/Sigma_max of the step's start material, as
// bremsstrahlung (done with this draw) or as a Moller event, which then takes
// one rejection trial per draw (`force` accepts any); a positron at rest
// annihilates.  Returns go when the particle takes its next step, wait when
// it needs another draw, ended at the end of its track.
template <int GEN, bool FAR>
__device__ __forceinline__ Round electron_event(const SimParams& P, const ElSmem& S, Electron& p, uint32_t& kind,
                                                uint4 x, bool force, Sec& sec) {
    const DevTables& T = P.T;
    ++p.ctr;
    sec.dx = p.u; sec.dy = p.v; sec.dz = p.w;
    sec.photon = sec.pos2 = false;
    const uint32_t what = kind & 3u;
    if (what == kCandidate) {
        const int m = int(kind >> 2);
        const float Tn = p.E, wcc = T.eabs_el, wcb = T.eabs_ph;
        float sm = 0.f, sb = 0.f;
        if (Tn > wcb || Tn > 2.f * wcc) {
            int i;
            float f;
            grid_pos(T, Tn, i, f);
            const int mj = m * T.n_e + i;
            const float4 a0 = el_entry<FAR>(S, mj), a1 = el_entry<FAR>(S, mj + 1);
            if (Tn > 2.f * wcc) sm = lerpf(a0.z, a1.z, f);
            if (Tn > wcb) sb = lerpf(a0.w, a1.w, f);
        }
        const float sh = sm + sb;
        if (u01(x.x) * S.mat[m].sigmax < sh) {
            hist_count<GEN>(P, p.hist, 2);
            if (u01(x.y) * sh < sm) {
                kind = kMoller;
                return Round::wait;
            }
            const float k = wcb * exp2f(u01(x.z) * __log2f(Tn / wcb));
            sec.n = 1;
            sec.photon = true;
            sec.E1 = k;
            p.E = Tn - k;
        }
    } else if (what == kMoller) {
        const float Tn = p.E;
        float eps, rphi;
        if (!moller_trial(x, Tn, T.eabs_el, eps, rphi) && !force) return Round::wait;
        float c, sn;
        cossin_2pi(rphi, c, sn);
        const float W = eps * Tn, Tp = Tn - W;
        const float cd = sqrtf(W * (Tn + 2.f * kMC2f) / (Tn * (W + 2.f * kMC2f)));
        const float cpr = sqrtf(Tp * (Tn + 2.f * kMC2f) / (Tn * (Tp + 2.f * kMC2f)));
        rotate(sec.dx, sec.dy, sec.dz, cd, c, sn);
        sec.n = 1;
        sec.E1 = W;
        rotate<true>(p.u, p.v, p.w, cpr, -c, -sn);
        p.E = Tp;
    } else {
        // two back-to-back 0.511 MeV photons (isotropic)
        const float cost = 2.f * u01(x.x) - 1.f;
        const float sint = sqrtf(fmaxf(0.f, 1.f - cost * cost));
        float cp, sp;
        cossin_2pi(u01(x.y), cp, sp);
        sec.n = 2;
        sec.photon = true;
        sec.E1 = sec.E2 = kMC2f;
        sec.dx = sint * cp; sec.dy = sint * sp; sec.dz = cost;
        return Round::ended;
    }
    return p.E < T.eabs_el ? absorb<GEN>(P, p, kind) : Round::go;
}

// ---------------------------------------------------------------- warp-uniform parts
// Add n to counter k of the CTA (call with the whole warp).
__device__ __forceinline__ void count(uint32_t* s_cnt, int k, uint32_t n) {
    if (lane_id() == 0) atomicAdd(&s_cnt[k], n);
}

// Queue slots a warp holds: [base, base + left) reserved but not yet written.
struct Slots {
    uint32_t base, left;
};

// `c` consecutive slots for the warp's pushes to one queue: from the
// reservation first, then a new reservation of PhaseArgs::bank_block slots
// (one atomic; fewer in a phase of few particles).  Returns the slot of the
// push of rank r.
__device__ __forceinline__ uint32_t reserve(Slots& sl, uint32_t c, uint32_t r, uint32_t* counter,
                                            const PhaseArgs& A, uint32_t total) {
    const uint32_t base = sl.base, left = sl.left;
    if (c <= left) {
        sl.base += c;
        sl.left -= c;
        return base + r;
    }
    // beyond 32 slots at most an eighth of the warp's even share of the phase's
    // items, so that a small phase leaves its queue dense
    const uint32_t share = total >> A.share_shift;
    const uint32_t miss = c - left;
    const uint32_t want = max(miss, min(A.bank_block, max(min(share, 32u), share >> 2)));
    uint32_t nb = 0;
    if (lane_id() == 0) nb = atomicAdd(counter, want);
    nb = __shfl_sync(kFull, nb, 0);
    sl.base = nb + miss;
    sl.left = want - miss;
    return r < left ? base + r : nb + (r - left);
}

// Bank the secondaries of a round of events (call with the whole warp):
// below-cutoff electrons and photons deposit on the spot, the rest get slots
// in the warp's reservations and counter-derived ids.  vox: the parents'
// packed voxels; pushes: the warp's pushes to the electron queue (0) and the
// photon queue (1).  PT 0: photons create electrons only.
template <int PT, int GEN, class Parent>
__device__ __forceinline__ void bank(const SimParams& P, const PhaseArgs& A, uint32_t total, Parent& p,
                                     uint32_t vox, const Sec& sec, Slots (&sl)[PT + 1],
                                     uint32_t (&pushes)[PT + 1]) {
    const bool photon = PT != 0 && sec.photon;
    for (int k = 0; k < 2; ++k) {
        const bool want = k < sec.n;
        if (!__any_sync(kFull, want)) return;
        const bool pos = k == 1 && sec.pos2;
        const float E = k ? sec.E2 : sec.E1;
        const float sg = (k == 1 && photon) ? -1.f : 1.f;
        const bool push = want && (pos || E >= (photon ? P.T.eabs_ph : P.T.eabs_el));
        if (want && !push) tally<GEN>(P, p.flags, vox_linear(P, vox), E);
#pragma unroll
        for (int q = 0; q < (PT == 0 ? 1 : 2); ++q) {   // q = 0 electron queue, 1 photon queue
            const bool mine = push && (photon == (q == 1));
            const uint32_t m = __ballot_sync(kFull, mine);
            if (!m) continue;
            const uint32_t c = __popc(m), r = __popc(m & lanemask_lt());
            const uint32_t slot = reserve(sl[q], c, r, q ? A.out_ph_count : A.out_el_count, A, total);
            if (mine) {
                const uint64_t id = child_id(uint64_t(p.pidlo) | (uint64_t(p.pidhi) << 32), p.flags & kChildMask);
                // the child index cannot wrap into the slot bits (no particle
                // comes near 65535 secondaries; flag it if one ever did)
                if ((p.flags & kChildMask) == kChildMask) atomicOr(P.status, ST_QUEUE_OVERFLOW);
                const uint32_t flags = (p.flags & kBatchMask) | (pos ? kPositron : 0u);
                ++p.flags;
                const Queue& Q = q ? A.out_ph : A.out_el;
                if (slot < Q.capacity) {
                    uint4* rec = Q.rec + size_t(slot) * (kQueueWords / 4);
                    __stcs(&rec[0], pack4(p.x, p.y, p.z, __float_as_uint(E)));
                    __stcs(&rec[1], pack4(sg * sec.dx, sg * sec.dy, sg * sec.dz, vox));
                    __stcs(&rec[2], make_uint4(p.hist, uint32_t(id), uint32_t(id >> 32), flags));
                } else {
                    atomicOr(P.status, ST_QUEUE_OVERFLOW);
                }
                hist_count<GEN>(P, p.hist, 3);
            }
            pushes[q] += c;
        }
    }
}

// ---------------------------------------------------------------- phase kernel
__device__ __forceinline__ void copy_to_smem(void* dst, const void* src, size_t bytes) {
    const float4* s = static_cast<const float4*>(src);
    float4* d = static_cast<float4*>(dst);
    const size_t n4 = bytes / 16;
    for (size_t k = threadIdx.x; k < n4; k += blockDim.x) d[k] = __ldg(&s[k]);
    const size_t rem = bytes - n4 * 16;
    const unsigned char* sb = static_cast<const unsigned char*>(src) + n4 * 16;
    unsigned char* db = static_cast<unsigned char*>(dst) + n4 * 16;
    for (size_t k = threadIdx.x; k < rem; k += blockDim.x) db[k] = sb[k];
}

__host__ __device__ inline size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

// Indices of this phase's work a warp takes at a time (primaries first,
// then queued particles): one atomic per block instead of one per refill.
// Every block boundary costs the warp a round trip to the shared counter,
// so blocks are several refills deep (128: measured best against 32, 64
// and 256).  A block is at most half the warp's even share of the work left
// (PhaseArgs::share_shift), so blocks shrink towards the end of a phase, down
// to exactly what the warp needs, and no warp sits on spare work.
constexpr uint32_t kGrab = 128u;

// Lanes of a warp that take particles.  A phase with less than one particle
// per lane (a small calculation, the last phases of any) is bound by the
// latency of a warp's loop, which grows with the lanes that diverge in it:
// its particles are spread over all resident warps.  Measured: 1e4 histories of
// a pencil in water 0.29 -> 0.20 ms a call, one CT beamlet of 1e5 1.09 -> 0.94,
// 1e6 20 MeV electrons on the 128^3 slab 6.0 -> 5.5 ms.
__device__ __forceinline__ uint32_t phase_lanes(uint32_t total) {
    return min((total - 1u) / (gridDim.x * (blockDim.x >> 5)) + 1u, 32u);
}

// What a warp leaves behind at the end of its phase: empty marks on the queue
// slots it reserved but never wrote, its share of the ledger; then the CTA's
// counters (Compton events are the other real collisions; a photoelectric
// event ends its photon without a deposit; a push creates a particle).
template <int PT>
__device__ __forceinline__ void phase_end(const SimParams& P, const PhaseArgs& A, double esc,
                                          const Slots (&sl)[PT + 1], uint32_t* s_cnt) {
    const uint32_t lane = lane_id();
#pragma unroll
    for (int q = 0; q < PT + 1; ++q) {
        const Queue& Q = q ? A.out_ph : A.out_el;
        const Slots h = sl[q];
        for (uint32_t i = lane; i < h.left; i += 32u)
            if (h.base + i < Q.capacity) queue_mark_empty(Q, h.base + i);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) esc += __shfl_down_sync(kFull, esc, o);
    if (lane == 0 && esc != 0.0) atomicAdd(&P.ledger[L_ESCAPED], esc);
    __syncthreads();
    for (int k = threadIdx.x; k < C_NCOUNT; k += blockDim.x) {
        const uint32_t n = k == C_COMPTON      ? s_cnt[C_PH_REAL] - s_cnt[C_PHOTO] - s_cnt[C_PAIR]
                           : k == C_LOCAL_DEP  ? s_cnt[C_LOCAL_DEP] - s_cnt[C_PHOTO]
                           : k == C_EL_CREATED ? s_cnt[C_PUSH_EL]
                           : k == C_PH_CREATED ? s_cnt[C_PUSH_PH]
                                               : s_cnt[k];
        if (n) atomicAdd(&P.counters[k], (unsigned long long)n);
    }
}

// Particle idx of the phase's input (its primaries first, then the queue)
// into p; false for an empty slot (a primary that missed the phantom, which
// k_sources accounts, or a reserved slot that was never written).
__device__ __forceinline__ bool load_input(const SimParams& P, const PhaseArgs& A, uint32_t idx, Part& p,
                                           bool& from_queue) {
    if (idx < A.n_src) {
        source_load(A.src, GDPM_IDX(P.status, idx, A.src.capacity, ST_B_QUEUE), p);
        p.hist = A.src_first + idx;
        return p.E >= 0.f;
    }
    queue_load(A.in, GDPM_IDX(P.status, idx - A.n_src, A.in.capacity, ST_B_QUEUE), p);
    from_queue = p.E >= 0.f;
    return from_queue;
}

// ---------------------------------------------------------------- photon phase
// A warp's photons that are not in a lane: a stack in shared memory that
// holds the ones ready to fly (from the bottom) and the ones waiting for a
// Compton event (from the top).
struct PhRec {
    uint4 a, b, c;      // x y z E | u v w flags | history, particle id lo, hi, draw counter
};
constexpr uint32_t kPhReady = 32, kPhStack = kPhReady + 64;

__device__ __forceinline__ void rec_store(PhRec& r, const Part& p) {
    r.a = pack4(p.x, p.y, p.z, __float_as_uint(p.E));
    r.b = pack4(p.u, p.v, p.w, p.flags);
    r.c = make_uint4(p.hist, p.pidlo, p.pidhi, p.ctr);
}
__device__ __forceinline__ void rec_load(const PhRec& r, Part& p) {
    const uint4 a = r.a, b = r.b, c = r.c;
    p.x = __uint_as_float(a.x); p.y = __uint_as_float(a.y); p.z = __uint_as_float(a.z);
    p.E = __uint_as_float(a.w);
    p.u = __uint_as_float(b.x); p.v = __uint_as_float(b.y); p.w = __uint_as_float(b.z);
    p.flags = b.w;
    p.hist = c.x; p.pidlo = c.y; p.pidhi = c.z; p.ctr = c.w;
}

// A phase kernel may start while the phase before it ends: CTAs that find room
// stage the tables, which no kernel of a calculation writes, and then wait for
// that phase to complete before they read anything it left (launch_phase).
// Both are without effect in a kernel launched to start after its predecessor.
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The photon phase.  Every lane of a warp takes one Woodcock flight per round.
// A photon that collides is set aside in shared memory and its lane takes
// another photon; once 32 wait, a round runs one Klein-Nishina trial (or the
// photoelectric absorption) of each, all lanes at work, and the accepted ones
// go back to fly.  Flights, rejection trials and recoil banking in one lane's
// own loop, as each lane reached them, kept 14 of 32 lanes active; now 27 are.
// Measured (1e8 histories of the CT plan / 2.5e8 of the paper's lung slab):
// 22.5 -> 20.6 ms / 36.0 -> 28.1 ms; 160 instead of 225 warp instructions a
// history; with sparser queue reservations, streamed queues and 28 warps (see
// bank_block, PhaseShape) 142 and 16.8 / 25.2 ms.  Issue slots are then 72 %
// taken; what a warp waits for is the latency of the voxel loads, two a flight
// at random voxels, of which 5 % hit the L1 and 75 % the L2.  New photons come kPhReady at a time into the stack, not one by one as lanes
// fall free.  Both kinds of round start with one draw, at one place in the
// code: a single inlined copy of the generator, which leaves the loop without
// calls and its constants in uniform registers.
// Stack bounds: photons enter the warp (and free lanes take one) only while
// at most 31 wait, and only up to kPhReady ready; 32 more are in the lanes.
template <int GEN>
__device__ __forceinline__ void photon_run(const SimParams& P, const PhaseArgs& A) {
    extern __shared__ __align__(16) unsigned char smem[];
    next_may_start();
    const DevTables& T = P.T;
    const size_t ne = size_t(T.n_mat) * T.n_e;
    float2* cum = reinterpret_cast<float2*>(smem);
    float* tot = reinterpret_cast<float*>(smem + align16(ne * 8));
    float* maj = reinterpret_cast<float*>(smem + align16(ne * 8) + align16(ne * 4));
    unsigned char* after = smem + align16(ne * 8) + align16(ne * 4) + align16(size_t(T.n_e) * 4);
    uint32_t* s_cnt = reinterpret_cast<uint32_t*>(after);
    PhRec* stack = reinterpret_cast<PhRec*>(after + align16(C_NCOUNT * 4)) + (threadIdx.x >> 5) * kPhStack;
    copy_to_smem(cum, T.ph_cum, ne * 8);
    copy_to_smem(tot, T.ph_tot, ne * 4);
    const PhSmem ps{maj, tot, cum};
    for (int k = threadIdx.x; k < C_NCOUNT; k += blockDim.x) s_cnt[k] = 0u;
    wait_for_previous();
    copy_to_smem(maj, P.maj, size_t(T.n_e) * 4);
    __syncthreads();
    const uint32_t n_in = A.in_count ? min(*A.in_count, A.in.capacity) : 0u;
    const uint32_t total = A.n_src + n_in;
    if (blockIdx.x >= total) return;
    const uint32_t lanes = phase_lanes(total), full = kFull >> (32u - lanes);
    double esc = 0.0;
    Part p{};
    const uint32_t lane = lane_id(), lt = lanemask_lt();
    bool active = false;
    uint32_t alive = 0u;                         // ballot of `active`
    uint32_t n_flights = 0u;                     // the lane's, inside the phantom
    uint32_t n_in_warp = 0u, n_done = 0u, n_on = 0u;   // the warp's: photons taken in, events, photons that went on
    Slots sl[1] = {{0u, 0u}};
    uint32_t pushes[1] = {0u};
    uint32_t n_ready = 0u, n_wait = 0u;          // the stack: [0, n_ready) and [kPhStack - n_wait, kPhStack)
    uint32_t st_base = 0u, st_left = 0u;         // the warp's block of work indices
    bool drained = false;                        // no input left
    for (uint32_t it = 0, trials = 0;; ++it) {
        while (n_wait < 32u && alive != full) {
            const uint32_t nm = full & ~alive, need = __popc(nm);
            // ---- input into the stack, up to kPhReady ready
            if (n_ready < min(need, kPhReady) && !drained) {
                if (st_left == 0u) {
                    const uint32_t block = max(need, min((total - min(total, st_base)) >> A.share_shift, kGrab));
                    uint32_t nb = 0u;
                    if (lane == 0) nb = atomicAdd(A.head, block);
                    nb = __shfl_sync(kFull, nb, 0);
                    st_base = nb;
                    st_left = nb < total ? min(block, total - nb) : 0u;
                    drained = st_left == 0u;
                }
                const uint32_t k = min(kPhReady - n_ready, st_left);
                Part q;
                bool from_queue = false, have = false;
                if (lane < k) have = load_input(P, A, st_base + lane, q, from_queue);
                st_base += k;
                st_left -= k;
                count(s_cnt, C_POP_PH, __popc(__ballot_sync(kFull, from_queue)));
                const bool low = have && q.E < T.eabs_ph;   // only a source photon
                if (__any_sync(kFull, low)) {
                    if (low) {
                        voxel_of(P, q);
                        tally<GEN>(P, q.flags, vox_of(P, q.ix, q.iy, q.iz), q.E);
                        have = false;
                    }
                    count(s_cnt, C_PH_TERMINATED, __popc(__ballot_sync(kFull, low)));
                }
                const uint32_t m = __ballot_sync(kFull, have);
                if (have) rec_store(stack[n_ready + __popc(m & lt)], q);
                n_ready += __popc(m);
                n_in_warp += __popc(m);
                __syncwarp();
            }
            // ---- free lanes take ready photons
            const uint32_t r = __popc(nm & lt);
            if (!active && r < n_ready && lane < lanes) {
                rec_load(stack[n_ready - 1u - r], p);
                active = true;
            }
            n_ready -= min(need, n_ready);
            __syncwarp();
            alive = __ballot_sync(kFull, active);
            if (drained) break;
        }
        // ---- which round: events once 32 photons wait, or, when the input is
        // drained, once no fewer wait than fly
        const uint32_t fly = __popc(alive) + n_ready;
        const bool events = n_wait >= 32u || (drained && n_wait >= fly);
        if (fly + n_wait == 0u) break;
        if (it >= P.max_iters) {
            if (lane == 0) atomicOr(P.status, ST_ITER_CAP);
            break;
        }
        const uint32_t k = min(n_wait, 32u);
        const PhRec* const rec = stack + (kPhStack - n_wait) + (lane < k ? lane : 0u);   // the k last set aside
        uint4 c = make_uint4(p.hist, p.pidlo, p.pidhi, p.ctr);
        if (events) c = rec->c;
        const uint4 x = philox4x32_10(c, P.keys);
        if (!events) {
            trials = 0u;
            Flight what = Flight::fly;
            if (active) {
                ++p.ctr;
                what = photon_flight<GEN>(P, ps, p, x, esc);
                active = what == Flight::fly;
                n_flights += what != Flight::gone;
            }
            const uint32_t m = __ballot_sync(kFull, what == Flight::wait);
            alive = __ballot_sync(kFull, active);
            if (what == Flight::wait) rec_store(stack[kPhStack - 1u - n_wait - __popc(m & lt)], p);
            n_wait += __popc(m);
            __syncwarp();
        } else {
            ++trials;
            Part q{};
            Sec sec{};
            bool goes_on = false;
            PhEvent what = PhEvent::none;
            if (lane < k) {
                rec_load(*rec, q);
                voxel_of(P, q);
                what = photon_event<GEN>(P, q, x, trials > 4096u, goes_on, sec);
            }
            n_wait -= k;
            bank<0, GEN>(P, A, total, q, vox_packed(q.ix, q.iy, q.iz), sec, sl, pushes);
            __syncwarp();
            const uint32_t gm = __ballot_sync(kFull, goes_on);
            const uint32_t wm = __ballot_sync(kFull, lane < k && what == PhEvent::none);
            if (lane < k && (goes_on || what == PhEvent::none))
                rec_store(stack[goes_on ? n_ready + __popc(gm & lt) : kPhStack - 1u - n_wait - __popc(wm & lt)], q);
            if (__any_sync(kFull, what > PhEvent::compton)) {
                count(s_cnt, C_PHOTO, __popc(__ballot_sync(kFull, what == PhEvent::photo)));
                count(s_cnt, C_PAIR, __popc(__ballot_sync(kFull, what == PhEvent::pair)));
            }
            n_done += k - __popc(wm);
            n_on += __popc(gm);
            n_ready += __popc(gm);
            n_wait += __popc(wm);
            __syncwarp();
        }
    }
    // every photon taken in escaped or ended in an event; a Compton event that
    // ends its photon deposits it (a photoelectric one does not, see
    // phase_end), and every event has one secondary (a pair two), banked or
    // deposited
    n_flights = __reduce_add_sync(kFull, n_flights);
    count(s_cnt, C_PH_FLIGHTS, n_flights);
    count(s_cnt, C_PH_TERMINATED, n_in_warp);
    count(s_cnt, C_PH_REAL, n_done);
    count(s_cnt, C_LOCAL_DEP, 2u * n_done - n_on - pushes[0]);
    count(s_cnt, C_PUSH_EL, pushes[0]);
    phase_end<0>(P, A, esc, sl, s_cnt);
}

// ---------------------------------------------------------------- electron phase
// A warp's electrons that are not in a lane: a stack in shared memory like
// the photons', in planes of 16 bytes (a 64-byte record would put every
// second lane on the same banks).
constexpr uint32_t kElReady = 32, kElWait = 32, kElStack = kElReady + kElWait + 32;
struct ElStack {
    uint4 a[kElStack], b[kElStack], c[kElStack], d[kElStack];
    Slots held[2];      // the warp's queue reservations, used only by event rounds
    // What a lane needs once a round or a step, kept out of its registers (no
    // spills instead of 72 bytes): history, id and draw counter of its
    // electron; direction after the hinge and mass thickness of leg 2.  1e8 CT
    // histories: electron phases 24.0 -> 23.3 ms, lung slab 47.1 -> 46.2.  The
    // KB a warp leaves room for 24 warps beside 58 KB of tables (4 materials
    // of 512 energies take 53); beside more see kFarWarps.
    uint4 ids[32];
    float4 hinge[32];
};

__device__ __forceinline__ void el_store(ElStack& s, uint32_t i, const Electron& p, uint32_t kind) {
    s.a[i] = pack4(p.x, p.y, p.z, __float_as_uint(p.E));
    s.b[i] = pack4(p.u, p.v, p.w, p.vox);
    s.c[i] = make_uint4(p.hist, p.pidlo, p.pidhi, p.ctr);
    s.d[i] = make_uint4(__float_as_uint(p.pend), p.flags, kind, 0u);
}
__device__ __forceinline__ uint32_t el_load(const ElStack& s, uint32_t i, Electron& p) {
    const uint4 a = s.a[i], b = s.b[i], c = s.c[i], d = s.d[i];
    p.x = __uint_as_float(a.x); p.y = __uint_as_float(a.y); p.z = __uint_as_float(a.z);
    p.E = __uint_as_float(a.w);
    p.u = __uint_as_float(b.x); p.v = __uint_as_float(b.y); p.w = __uint_as_float(b.z);
    p.vox = b.w;
    p.hist = c.x; p.pidlo = c.y; p.pidhi = c.z; p.ctr = c.w;
    p.pend = __uint_as_float(d.x);
    p.flags = d.y;
    return d.z;
}

// The electron phase, in rounds like the photon phase.  In a step round every
// lane sets up a step (unless one is in progress) and walks it.  A step that
// ends in a hard-event candidate, and a positron at rest, waits in shared
// memory; once kElWait wait, an event round gives each of 32 its next draw.
// In one lane's own loop, as each lane reached them, the draw, walk, candidate
// and Moller code ran with 14.8 of 32 lanes active and 271 warp instructions
// a history; now 20 and 214.  Measured against that (1e8 histories of the CT
// plan; 2.5e8 of the paper's lung slab; 2.5e6 20 MeV electrons on its bone
// slab): electron phase 29.6 -> 25.7, 54.8 -> 50.0, 7.0 -> 5.6 ms; with the
// constants, ids and hinge directions in shared memory 23.3, 46.2, 5.2 ms.
// Bound by its instructions (75 % of the issue slots taken).  On the CT plan 27
// lanes set up a step in a round and 31 start its walk; the hinge runs twice
// with 14, a crossing twice with 7 and the second stretch once with 10, and 6
// lanes are refilled.  Running the second stretch only for 6 to 12 lanes or
// more, or the refill for 2 to 12, was slower by 1 to 10 %.
template <int GEN, bool FAR>
__device__ __forceinline__ void electron_run(const SimParams& P, const PhaseArgs& A) {
    extern __shared__ __align__(16) unsigned char smem[];
    next_may_start();
    const DevTables& T = P.T;
    const size_t ne = size_t(T.n_mat) * T.n_e;
    float4* el = reinterpret_cast<float4*>(smem);
    const size_t el_bytes = FAR ? 0 : ne * 16;
    float* rinv = reinterpret_cast<float*>(smem + el_bytes);
    const size_t nr = size_t(T.n_mat) * T.n_r;
    float* atab = reinterpret_cast<float*>(smem + el_bytes + align16(nr * 4));
    unsigned char* after = smem + el_bytes + align16(nr * 4) + align16(size_t(T.n_a) * 4);
    uint32_t* s_cnt = reinterpret_cast<uint32_t*>(after);
    ElMat* mats = reinterpret_cast<ElMat*>(after + align16(C_NCOUNT * 4));
    ElStack& stack = reinterpret_cast<ElStack*>(mats + kMaxMat)[threadIdx.x >> 5];
    if (threadIdx.x < uint32_t(T.n_mat)) {
        const int m = int(threadIdx.x);
        mats[m] = ElMat{T.r_eabs[m], T.inv_sigmax[m], T.rinv_lo[m], T.rinv_idr[m], T.inv_x0[m], T.sigmax[m]};
    }
    if (lane_id() < 4u) (&stack.held[0].base)[lane_id()] = 0u;
    if (!FAR) copy_to_smem(el, T.el, ne * 16);
    copy_to_smem(rinv, T.rinv, nr * 4);
    copy_to_smem(atab, T.atab, size_t(T.n_a) * 4);
    const ElSmem es{FAR ? T.el : el, rinv, atab, mats};
    for (int k = threadIdx.x; k < C_NCOUNT; k += blockDim.x) s_cnt[k] = 0u;
    wait_for_previous();
    __syncthreads();
    const uint32_t n_in = A.in_count ? min(*A.in_count, A.in.capacity) : 0u;
    const uint32_t total = A.n_src + n_in;
    if (blockIdx.x >= total) return;
    const uint32_t lanes = phase_lanes(total), full = kFull >> (32u - lanes);
    double esc = 0.0;
    Electron p{};
    ElStep st{};
    const uint32_t lane = lane_id(), lt = lanemask_lt();
    bool active = false;
    uint32_t alive = 0u;                         // ballot of `active`
    uint32_t n_steps = 0u, n_ended = 0u;         // the warp's
    uint32_t crossings = 0u;                     // the lane's
    uint32_t n_ready = 0u, n_wait = 0u;          // the stack: [0, n_ready) and [kElStack - n_wait, kElStack)
    uint32_t st_base = 0u, st_left = 0u;         // the warp's block of work indices
    bool drained = false;                        // no input left
    for (uint32_t it = 0, draws = 0;; ++it) {
        while (n_wait < kElWait && alive != full) {
            const uint32_t nm = full & ~alive, need = __popc(nm);
            // ---- input into the stack, up to kElReady ready
            if (n_ready < min(need, kElReady) && !drained) {
                if (st_left == 0u) {
                    const uint32_t block = max(need, min((total - min(total, st_base)) >> A.share_shift, kGrab));
                    uint32_t nb = 0u;
                    if (lane == 0) nb = atomicAdd(A.head, block);
                    nb = __shfl_sync(kFull, nb, 0);
                    st_base = nb;
                    st_left = nb < total ? min(block, total - nb) : 0u;
                    drained = st_left == 0u;
                }
                const uint32_t k = min(kElReady - n_ready, st_left);
                Part q;
                Electron e{};
                bool from_queue = false, have = false;
                if (lane < k) {
                    have = load_input(P, A, st_base + lane, q, from_queue);
                    if (have && !from_queue) voxel_of(P, q);
                    e = Electron{q.x, q.y, q.z, q.u, q.v, q.w, q.E, 0.f, vox_packed(q.ix, q.iy, q.iz),
                                 q.hist, q.pidlo, q.pidhi, q.ctr, q.flags};
                }
                st_base += k;
                st_left -= k;
                count(s_cnt, C_POP_EL, __popc(__ballot_sync(kFull, from_queue)));
                // below the cutoff: a source electron, or a positron, which
                // annihilates
                const bool low = have && e.E < T.eabs_el;
                if (__any_sync(kFull, low)) {
                    uint32_t kind = 0u;
                    const bool wait = low && absorb<GEN>(P, e, kind) == Round::wait;
                    const uint32_t wm = __ballot_sync(kFull, wait);
                    if (wait) el_store(stack, kElStack - 1u - n_wait - __popc(wm & lt), e, kind);
                    n_wait += __popc(wm);
                    n_ended += __popc(__ballot_sync(kFull, low)) - __popc(wm);
                    have = have && !low;
                }
                const uint32_t m = __ballot_sync(kFull, have);
                if (have) el_store(stack, n_ready + __popc(m & lt), e, 0u);
                n_ready += __popc(m);
                __syncwarp();
            }
            // ---- free lanes take ready electrons
            const uint32_t r = __popc(nm & lt);
            if (!active && r < n_ready && lane < lanes) {
                el_load(stack, n_ready - 1u - r, p);
                stack.ids[lane] = make_uint4(p.hist, p.pidlo, p.pidhi, p.ctr);
                active = true;
                st.what = 0u;
            }
            n_ready -= min(need, n_ready);
            __syncwarp();
            alive = __ballot_sync(kFull, active);
            if (drained) break;
        }
        // ---- which round: events once kElWait electrons wait, or, when the
        // input is drained, once no fewer wait than walk
        const uint32_t walking = __popc(alive) + n_ready;
        const bool events = n_wait >= kElWait || (drained && n_wait >= walking);
        if (walking + n_wait == 0u) break;
        if (it >= P.max_iters) {
            if (lane == 0) atomicOr(P.status, ST_ITER_CAP);
            break;
        }
        const uint32_t k = min(n_wait, 32u);
        const uint32_t top = kElStack - n_wait + (lane < k ? lane : 0u);     // the k last set aside
        uint4 c = stack.ids[lane];
        // material and density of the voxel a step starts in: the loads run
        // while the draw is made
        int mat = 0;
        if (events) {
            c = stack.c[top];
        } else if (active && (st.what & 3u) == 0u) {
            const uint32_t vox0 = GDPM_IDX(P.status, vox_linear(P, p.vox), n_voxels(P), ST_B_VOXEL);
            mat = int(__ldg(&P.mat[vox0]));
            st.rho = __ldg(&P.rho[vox0]);
        }
        const uint4 x = philox4x32_10(c, P.keys);
        if (!events) {
            draws = 0u;
            uint32_t kind = 0u;
            Round what = Round::go;
            n_steps += __popc(__ballot_sync(kFull, active && (st.what & 3u) == 0u));
            if (active) {
                if ((st.what & 3u) == 0u) stack.ids[lane].w = c.w + 1u;
                p.hist = c.x;
                what = electron_round<GEN, FAR>(P, es, p, st, x, mat, stack.hinge[lane],
                                           drained ? max(P.walk_trips, kDrainedStretches) : P.walk_trips, esc,
                                           crossings, kind);
                active = what == Round::go;
            }
            const uint32_t m = __ballot_sync(kFull, what == Round::wait);
            n_ended += __popc(alive);
            alive = __ballot_sync(kFull, active);
            n_ended -= __popc(m) + __popc(alive);
            if (what == Round::wait) {
                const uint4 id = stack.ids[lane];
                p.hist = id.x; p.pidlo = id.y; p.pidhi = id.z; p.ctr = id.w;
                el_store(stack, kElStack - 1u - n_wait - __popc(m & lt), p, kind);
            }
            n_wait += __popc(m);
            __syncwarp();
        } else {
            ++draws;
            Electron q{};
            Sec sec{};
            uint32_t kind = 0u, was = 0u;
            Round what = Round::ended;
            if (lane < k) {
                was = kind = el_load(stack, top, q);
                what = electron_event<GEN, FAR>(P, es, q, kind, x, draws > 4096u, sec);
            }
            n_wait -= k;
            if (__any_sync(kFull, sec.n > 0)) {
                Slots sl[2] = {stack.held[0], stack.held[1]};
                uint32_t pushes[2] = {0u, 0u};
                bank<1, GEN>(P, A, total, q, q.vox, sec, sl, pushes);
                const uint32_t mol = __popc(__ballot_sync(kFull, sec.n > 0 && (was & 3u) == kMoller));
                const uint32_t brems = __popc(__ballot_sync(kFull, sec.n > 0 && (was & 3u) == kCandidate));
                const uint32_t annihil = __popc(__ballot_sync(kFull, sec.n > 1));
                if (lane == 0) {
                    stack.held[0] = sl[0];
                    stack.held[1] = sl[1];
                }
                // one shared-memory atomic for the six counters
                const uint32_t n = lane == 0 ? mol : lane == 1 ? brems : lane == 2 ? annihil
                                   : lane == 3 ? pushes[0] : lane == 4 ? pushes[1]
                                               : mol + brems + 2u * annihil - pushes[0] - pushes[1];
                const int slot = lane == 0 ? C_MOLLER : lane == 1 ? C_BREMS : lane == 2 ? C_ANNIHIL
                                 : lane == 3 ? C_PUSH_EL : lane == 4 ? C_PUSH_PH : C_LOCAL_DEP;
                if (lane < 6u) atomicAdd(&s_cnt[slot], n);
            }
            __syncwarp();
            const uint32_t gm = __ballot_sync(kFull, lane < k && what == Round::go);
            const uint32_t wm = __ballot_sync(kFull, lane < k && what == Round::wait);
            if (lane < k && what != Round::ended)
                el_store(stack, what == Round::go ? n_ready + __popc(gm & lt)
                                                  : kElStack - 1u - n_wait - __popc(wm & lt), q, kind);
            n_ended += k - __popc(gm) - __popc(wm);
            n_ready += __popc(gm);
            n_wait += __popc(wm);
            __syncwarp();
        }
    }
    // only a phase stopped by its iteration cap leaves a track unfinished
    if (active && p.pend != 0.f) tally<GEN>(P, p.flags, vox_linear(P, p.vox), p.pend);
    count(s_cnt, C_EL_STEPS, n_steps);
    count(s_cnt, C_EL_TERMINATED, n_ended);
    count(s_cnt, C_CROSS, __reduce_add_sync(kFull, crossings));
    const Slots sl[2] = {stack.held[0], stack.held[1]};
    phase_end<1>(P, A, esc, sl, s_cnt);
}

// One transport phase (Sec. 2.2.1 Step 3), a persistent loop per warp.  PT: 0
// photons, 1 electrons, 2 electrons beside large tables (kFarWarps).
template <int PT, int GEN>
__device__ __forceinline__ void phase_run(const SimParams& P, const PhaseArgs& A) {
    if constexpr (PT == 0) photon_run<GEN>(P, A);
    else electron_run<GEN, PT == 2>(P, A);
}

template <int PT, int GEN>
__global__ void __launch_bounds__(PhaseShape<PT>::threads, PhaseShape<PT>::ctas)
k_phase(const SimParams P, const PhaseArgs A) {
    phase_run<PT, GEN>(P, A);
}


// ---------------------------------------------------------------- sources
// Source CTAs: one of 1024 threads per SM for phases that fill them, which
// stages its tables once and leaves the L1 to the beamlets' rows (eight of
// 256, of which six are resident, take 7 % longer); CTAs of 256 below.
constexpr int kSourceThreads = 1024;
// The primaries of one source phase (Sec. 2.3), made with every lane busy
// before the phase runs: primary idx goes to slot idx of A.src.  One that
// misses the phantom leaves its slot empty (E < 0) and is accounted here:
// source and escaped energy, a created and a terminated particle.
// The spectrum prefix counts of the batches and the cumulative beamlet
// weights are searched for every primary: a CTA copies them to shared
// memory when they fit (n_prefix, n_cdf of them; see sources_smem).
// Bound by its instructions and the latency of its searches, not by the 32
// bytes a primary it writes.  1e8 primaries of the CT plan 2.21 -> 1.79 ms,
// 2.5e8 of the lung slab's field 3.32 -> 2.93 ms: the box entry without arrays
// in local memory, the batch index without two divisions and the draw's round
// keys took 0.30 and 0.19 of that, the CTA shape 0.13 and 0.20.
template <int PT>
__device__ __forceinline__ void make_sources(const SimParams& P, const PhaseArgs& A, uint32_t n_prefix,
                                             uint32_t n_cdf) {
    extern __shared__ __align__(16) unsigned char smem[];
    next_may_start();
    float* s_cdf = reinterpret_cast<float*>(smem);
    uint32_t* s_prefix = reinterpret_cast<uint32_t*>(smem + size_t(n_cdf) * 4);
    for (uint32_t i = threadIdx.x; i < n_cdf; i += blockDim.x) s_cdf[i] = P.S.bl_cdf[i];
    for (uint32_t i = threadIdx.x; i < n_prefix; i += blockDim.x) s_prefix[i] = A.bin_prefix[i];
    __syncthreads();
    const uint32_t* ptab = n_prefix ? s_prefix : nullptr;
    const float* ctab = n_cdf ? s_cdf : nullptr;
    Acc acc{0.0, 0.0};
    const uint32_t inv_big = 0xffffffffu / (A.nb_small + 1u), inv_small = 0xffffffffu / max(A.nb_small, 1u);
    uint32_t made = 0u, missed = 0u;
    for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < A.n_src;
         idx += gridDim.x * blockDim.x) {
        Part p{};
        if (make_primary(P, A, idx, p, acc, inv_big, inv_small, ptab, ctab)) {
            source_store(A.src, GDPM_IDX(P.status, idx, A.src.capacity, ST_B_QUEUE), p);
        } else {
            source_mark_empty(A.src, GDPM_IDX(P.status, idx, A.src.capacity, ST_B_QUEUE));
            ++missed;
        }
        ++made;
    }
    made = __reduce_add_sync(kFull, made);
    missed = __reduce_add_sync(kFull, missed);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc.src += __shfl_down_sync(kFull, acc.src, o);
        acc.esc += __shfl_down_sync(kFull, acc.esc, o);
    }
    if (lane_id() == 0) {
        if (acc.src != 0.0) atomicAdd(&P.ledger[L_SOURCE], acc.src);
        if (acc.esc != 0.0) atomicAdd(&P.ledger[L_ESCAPED], acc.esc);
        if (made) {
            atomicAdd(&P.counters[C_PRIMARY], (unsigned long long)made);
            atomicAdd(&P.counters[PT == 0 ? C_PH_CREATED : C_EL_CREATED], (unsigned long long)made);
        }
        if (missed) atomicAdd(&P.counters[PT == 0 ? C_PH_TERMINATED : C_EL_TERMINATED], (unsigned long long)missed);
    }
}

template <int PT>
__global__ void __launch_bounds__(kSourceThreads) k_sources(const SimParams P, const PhaseArgs A, uint32_t n_prefix,
                                                 uint32_t n_cdf) {
    make_sources<PT>(P, A, n_prefix, n_cdf);
}

// Cumulative-weight entries the sources search (the cumulative sampler of a
// sampled fluence map; none otherwise).
inline uint32_t cdf_entries(const SimParams& P, const PhaseArgs& A) {
    return (P.S.geometry == GDPM_GEO_BEAMLETS && P.S.sampler == GDPM_SAMPLE_CDF && A.n_sub == 0)
               ? uint32_t(P.S.n_beamlets) : 0u;
}

// Entries of the prefix and cumulative-weight tables a source CTA stages in
// shared memory (0: read from global memory), within a 40 KB budget: below the
// 48 KB any launch may ask for, so no launch sets a limit that another host
// thread's launch of the same kernel would run into.
__host__ __device__ inline void sources_smem(uint32_t prefix_entries, uint32_t cdf_entries,
                                             uint32_t& n_prefix, uint32_t& n_cdf) {
    const size_t budget = 40u << 10;
    n_cdf = size_t(cdf_entries) * 4 <= budget ? cdf_entries : 0u;
    n_prefix = size_t(n_cdf) * 4 + size_t(prefix_entries) * 4 <= budget ? prefix_entries : 0u;
}

// ---------------------------------------------------------------- Metropolis chains
// Advance the chains through the histories of [first, first+n) that belong to
// them (h = c, c + C, c + 2C, ...), in order: propose J uniform, accept when
// u f_I < f_J (u < f_J / f_I without the division), record the state as the
// beamlet of history h (Algorithm A1).  A chain's steps are sequential, but
// only the acceptance is: the proposals are draws of their own.  A CTA takes
// 32 chains; its first warp walks them, one lane a chain, through a tile of
// proposals that the other warps have made (draw, beamlet, weight), while
// they make the next tile.  The acceptance is decided in FP32 unless the two
// sides agree to 1e-6 (their rounding is below 3e-7) or leave FP32's range,
// and then in FP64.  One thread a chain doing all of it took a draw, a load
// and two FP64 operations behind one another per step: 390 ns, 1.9 ms for 2e7
// histories and 4096 chains; now 0.3 ms.
constexpr int kMetroChains = 32, kMetroThreads = 256, kMetroTile = 56;
// The acceptance in FP64; out of line, or its loads and FP64 operations run
// ahead of the test that seldom needs them (1.03 instead of 0.3 ms).
__device__ __noinline__ bool metropolis_exact(const double* f, uint32_t I, uint32_t J, uint32_t w) {
    return (double(w) + 0.5) * 0x1p-32 * f[I] < f[J];
}
__device__ __forceinline__ void metropolis_run(const SimParams& P, uint32_t first, uint32_t n, uint32_t* chains,
                                               uint32_t* pick) {
    __shared__ uint32_t s_J[2][kMetroTile][kMetroChains], s_w[2][kMetroTile][kMetroChains];
    __shared__ float s_f[2][kMetroTile][kMetroChains];
    const uint32_t C = P.S.n_chains, nf = uint32_t(P.S.n_beamlets);
    const double* f = P.S.bl_f;
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5, c = blockIdx.x * kMetroChains + lane;
    const uint64_t end = uint64_t(first) + n;
    // the chain's first history of the range, and how many it has there
    const uint64_t h0 = uint64_t(first) + (uint64_t(c) + C - first % C) % C;
    const uint32_t steps = c < C && h0 < end ? uint32_t((end - 1u - h0) / C) + 1u : 0u;
    const uint32_t tiles = chain_tiles(n, C, kMetroTile);
    auto propose = [&](uint32_t t) {
        for (uint32_t j = warp - 1u; j < uint32_t(kMetroTile); j += kMetroThreads / 32 - 1) {
            const uint32_t step = t * kMetroTile + j;
            if (step < steps) {
                const uint64_t h = h0 + uint64_t(step) * C;
                const uint4 w = philox4x32_10(make_uint4(uint32_t(h), 0u, 0u, 0u), P.key0, P.key1);
                const uint32_t J = __umulhi(w.x, nf);
                s_J[t & 1u][j][lane] = J;
                s_w[t & 1u][j][lane] = w.y;
                s_f[t & 1u][j][lane] = float(f[J]);
            }
        }
    };
    uint32_t I = 0u;
    float fI = 0.f;
    if (warp == 0u) {
        if (c < C) {
            I = chains[c];
            fI = float(f[I]);
        }
    } else {
        propose(0u);
    }
    uint64_t at = h0 - first;
    for (uint32_t t = 0; t < tiles; ++t) {
        __syncthreads();
        if (warp != 0u) {
            if (t + 1u < tiles) propose(t + 1u);
            continue;
        }
        const uint32_t here = steps > t * kMetroTile ? min(steps - t * kMetroTile, uint32_t(kMetroTile)) : 0u;
#pragma unroll 4
        for (uint32_t j = 0; j < here; ++j) {
            const uint32_t J = s_J[t & 1u][j][lane], w = s_w[t & 1u][j][lane];
            const float fJ = s_f[t & 1u][j][lane];
            const float lhs = (float(w) + 0.5f) * 0x1p-32f * fI, d = fJ - lhs;
            bool accept = d > 0.f;
            if (!(fabsf(d) > 1e-6f * (fJ + lhs))) accept = metropolis_exact(f, I, J, w);
            if (accept) {
                I = J;
                fI = fJ;
            }
            pick[at] = I;
            at += C;
        }
    }
    if (warp == 0u && c < C) chains[c] = I;
}

// ---------------------------------------------------------------- device-driven phase loop
// Phase k's arguments from k alone, as the host loop sets them: photon
// phase k (even) reads photons P[k] and banks electrons into E[k+1];
// electron phase k (odd) reads E[k] and banks photons into P[k+1] and
// electrons into E[k+2].  Row k of ctl holds (pop head, P[k] count, E[k]
// count, -).  The source particle's j-th phase takes primaries
// [first + j*chunk, first + min((j+1)*chunk, n_src)).
__device__ __forceinline__ PhaseArgs phase_args(const LoopArgs& L, uint32_t k) {
    PhaseArgs A{};
    A.nb_small = L.nb_small;
    A.nb_rem = L.nb_rem;
    A.bin_prefix = L.bin_prefix;
    A.prefix_n = L.prefix_n;
    A.n_sub = L.n_sub;
    A.sub_batches = L.sub_batches;
    A.sub_first = L.sub_first;
    A.bank_block = L.bank_block;
    A.src = L.qsrc;
    const bool ph = (k % 2u) == 0u;
    A.share_shift = L.share_shift[ph ? 0 : 1];
    const bool src_phase = ph == (L.src_particle == GDPM_PHOTON);
    if (src_phase) {
        const uint32_t j = L.src_particle == GDPM_PHOTON ? k / 2u : (k - 1u) / 2u;
        const uint64_t off = uint64_t(j) * L.chunk;
        if (off < L.n_src) {
            A.n_src = uint32_t(min(uint64_t(L.chunk), uint64_t(L.n_src) - off));
            A.src_first = L.first + uint32_t(off);
            A.bl_pick = L.pick;
        }
    }
    uint32_t* ctl = L.ctl;
    A.head = ctl + size_t(k) * 4;
    if (ph) {
        A.in = L.qph;
        A.in_count = k >= 1u ? ctl + size_t(k) * 4 + 1 : nullptr;
        A.out_el = ((k + 1u) / 2u) % 2u ? L.qe1 : L.qe0;
        A.out_el_count = ctl + size_t(k + 1) * 4 + 2;
        A.out_ph = L.qph;
        A.out_ph_count = ctl + size_t(k + 2) * 4 + 1;
    } else {
        A.in = (k / 2u) % 2u ? L.qe1 : L.qe0;
        A.in_count = ctl + size_t(k) * 4 + 2;
        A.out_ph = L.qph;
        A.out_ph_count = ctl + size_t(k + 1) * 4 + 1;
        A.out_el = ((k + 2u) / 2u) % 2u ? L.qe1 : L.qe0;
        A.out_el_count = ctl + size_t(k + 2) * 4 + 2;
    }
    return A;
}

// One pass of the device-driven loop runs photon phase k and electron
// phase k+1, k = *L.k (even); PT selects which of the two this launch is
// (0 the photon phase, 1 the electron phase).
// The phase's arguments are derived in shared memory from k.  (A kernel of
// its own: the host loop's k_phase takes them as kernel parameters, which
// keeps more registers for the transport loop.)
template <int PT>
__global__ void __launch_bounds__(PhaseShape<PT>::threads, PhaseShape<PT>::ctas)
k_phase_loop(const SimParams P, const LoopArgs L) {
    __shared__ PhaseArgs sA;
    if (threadIdx.x == 0) sA = phase_args(L, *L.k + (PT == 0 ? 0u : 1u));
    __syncthreads();
    phase_run<PT, kGeneral>(P, sA);
}

// Primaries of this pass's source phase (before it runs).
template <int PT>
__global__ void __launch_bounds__(kSourceThreads) k_sources_loop(const SimParams P, const LoopArgs L, uint32_t n_prefix,
                                                      uint32_t n_cdf) {
    const PhaseArgs A = phase_args(L, *L.k + uint32_t(PT));
    if (A.n_src) make_sources<PT>(P, A, n_prefix, n_cdf);
}

// Metropolis picks for this pass's source phase (before it runs).
__global__ void __launch_bounds__(kMetroThreads) k_metropolis_loop(const SimParams P, const LoopArgs L) {
    const uint32_t k = *L.k + (L.src_particle == GDPM_PHOTON ? 0u : 1u);
    const PhaseArgs A = phase_args(L, k);
    if (A.n_src) metropolis_run(P, A.src_first, A.n_src, L.chains, L.pick);
}

// After a pass: go on while primaries remain or the pass left particles for
// the next one (photons P[k+2], electrons E[k+3]); stop at the phase cap
// with a status bit.  One thread.
__global__ void k_loop_ctl(const LoopArgs L, cudaGraphConditionalHandle h) {
    const uint32_t k = *L.k, k2 = k + 2u;
    const uint32_t j_next = k2 / 2u;        // index of the next pass's source phase
    const bool src_left = uint64_t(j_next) * L.chunk < uint64_t(L.n_src);
    const uint32_t pending = L.ctl[size_t(k2) * 4 + 1] + L.ctl[size_t(k2 + 1) * 4 + 2];
    bool more = src_left || pending > 0u;
    if (more && int(k2) + 3 >= L.max_phases) {
        atomicOr(L.status, ST_PHASE_CAP);
        more = false;
    }
    *L.k = k2;
    cudaGraphSetConditional(h, more ? 1u : 0u);
}

// ---------------------------------------------------------------- checks
__global__ void k_debug_philox(const uint32_t* ctr, uint32_t k0, uint32_t k1, uint32_t* out,
                               uint64_t n) {
    for (uint64_t s = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; s < n;
         s += uint64_t(gridDim.x) * blockDim.x) {
        const uint4 c = make_uint4(ctr[4 * s], ctr[4 * s + 1], ctr[4 * s + 2], ctr[4 * s + 3]);
        const uint4 o = philox4x32_10(c, k0, k1);
        out[4 * s] = o.x; out[4 * s + 1] = o.y; out[4 * s + 2] = o.z; out[4 * s + 3] = o.w;
    }
}

__global__ void k_debug_sample(int kind, float a, float b, uint64_t n, uint32_t k0, uint32_t k1,
                               double* out1, double* out2) {
    SimParams P{};
    P.key0 = k0;
    P.key1 = k1;
    for (uint64_t s = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; s < n;
         s += uint64_t(gridDim.x) * blockDim.x) {
        Part p{};
        p.hist = uint32_t(s);
        p.pidlo = 1u;
        double o1 = 0, o2 = 0;
        if (kind == 0) {
            float eps, cost, rphi;
            sample_kn(p, P, a, eps, cost, rphi);
            o1 = eps; o2 = cost;
        } else if (kind == 1) {
            float eps, rphi;
            sample_moller(p, P, a, b, eps, rphi);
            const float W = eps * a;
            o1 = eps;
            o2 = sqrtf(W * (a + 2.f * kMC2f) / (a * (W + 2.f * kMC2f)));
        } else if (kind == 2) {
            const float4 v = draw(p, k0, k1);
            o1 = b * exp2f(v.z * __log2f(a / b));
        } else if (kind == 3) {
            const float4 r = draw(p, k0, k1);
            o1 = 1.f - 2.f * a * r.z / (1.f - r.z + a);
        } else if (kind == 5) {
            float mu, rphi;
            sample_sauter(p, P, a, mu, rphi);
            o1 = mu;
            o2 = kTwoPi * rphi;
        } else {
            const float4 r = draw(p, k0, k1);
            o1 = 2.f * r.x - 1.f;
            o2 = kTwoPi * r.y;
        }
        out1[s] = o1;
        if (out2) out2[s] = o2;
    }
}

// Metropolis chains of Algorithm A1, one thread per chain c.  Chain c starts
// at a uniform beamlet from the Philox block at (c, 0, 1, 0).
__global__ void k_metropolis_init(const SimParams P, uint32_t* chains) {
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= P.S.n_chains) return;
    const uint4 w = philox_block(c, 0u, 1u, 0u, P.key0, P.key1);
    chains[c] = __umulhi(w.x, uint32_t(P.S.n_beamlets));
}

__global__ void __launch_bounds__(kMetroThreads) k_metropolis(const SimParams P, uint32_t first, uint32_t n,
                                                              uint32_t* chains, uint32_t* pick) {
    metropolis_run(P, first, n, chains, pick);
}

// Beamlet rows of histories [first, first+n) (checks of the samplers).
__global__ void k_debug_beamlets(const SimParams P, uint32_t first, uint64_t n,
                                 const uint32_t* pick, int32_t* out) {
    for (uint64_t s = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; s < n; s += uint64_t(gridDim.x) * blockDim.x) {
        Part p{};
        p.hist = first + uint32_t(s);
        p.pidlo = 1u;
        const float4 r = draw(p, P.key0, P.key1);
        PhaseArgs A{};
        A.bl_pick = pick;
        out[s] = P.S.bl_row[pick_beamlet(P.S, A, uint32_t(s), first + uint32_t(s), r.w, P.key0, P.key1, P.S.bl_cdf)];
    }
}

__global__ void k_debug_sources(const SimParams P, const PhaseArgs A, uint64_t n, double* out) {
    for (uint64_t s = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; s < n;
         s += uint64_t(gridDim.x) * blockDim.x) {
        Part p{};
        Acc acc{0, 0};
        const bool in = make_primary(P, A, uint32_t(s), p, acc, 0xffffffffu / (A.nb_small + 1u),
                                     0xffffffffu / max(A.nb_small, 1u));
        double* o = out + 8 * s;
        o[0] = p.x; o[1] = p.y; o[2] = p.z; o[3] = p.u; o[4] = p.v; o[5] = p.w; o[6] = p.E;
        o[7] = in ? 1.0 : 0.0;
    }
}

}  // namespace

// Shared memory of the staged tables and the CTA's counters, which bounds the
// tables a context accepts, and with the electrons' per-material constants.
static size_t tables_smem(const DevTables& T, int particle) {
    const size_t ne = size_t(T.n_mat) * T.n_e;
    const size_t cnt = align16(C_NCOUNT * 4);
    if (particle == GDPM_PHOTON)
        return align16(ne * 8) + align16(ne * 4) + align16(size_t(T.n_e) * 4) + cnt;
    return ne * 16 + align16(size_t(T.n_mat) * T.n_r * 4) + align16(size_t(T.n_a) * 4) + cnt;
}
// pt: 0 photons, 1 electrons, 2 electrons with the step and event table left
// in global memory.
static size_t smem_of(const DevTables& T, int pt) {
    if (pt == 0) return tables_smem(T, GDPM_PHOTON);
    const size_t el = pt == 2 ? size_t(T.n_mat) * T.n_e * 16 : 0;
    return tables_smem(T, GDPM_ELECTRON) + kMaxMat * sizeof(ElMat) - el;
}

// log2 of at least twice the warps of a phase: items >> shift is at most half
// a warp's even share of them.
static uint32_t share_shift(uint32_t warps) {
    uint32_t s = 1u;
    while ((1ull << s) < 2ull * warps) ++s;
    return s;
}

// Queue slots a warp reserves at a time: up to 32, while all warps' spare
// slots stay below an eighth of the queue, and up to kBankBlock where they
// stay below 1/256 of it; exact below 8.  A reservation is an atomic whose
// answer the warp waits for, a third of a photon phase's banking at 32 slots
// each: at 128 the photon phases of 1e8 CT histories take 17.9 ms instead of
// 19.1 (64: 18.0, 256: 18.0).
constexpr uint64_t kBankBlock = 128u;
static uint32_t bank_block(uint64_t capacity, uint64_t warps) {
    const uint64_t b = std::max(std::min<uint64_t>(32u, capacity / (8u * warps)),
                                std::min(kBankBlock, capacity / (256u * warps)));
    return b >= 8u ? uint32_t(b) : 0u;
}

int transport_smem(const gdpm_tables* t, int particle) { return int(tables_smem(t->dev, particle)); }

// A phase kernel's launch shape: its own CTA, or the context's
// GDPM_PARAM_BLOCK_THREADS when set (at most 256, within every kernel's
// bound); the tables and counters of a CTA and the warps' stacks in shared
// memory.  Beside large tables a CTA has fewer warps.  fixed_smem: shared
// memory the kernel declares itself, which counts towards the same limit.
constexpr size_t kMaxSmem = size_t(227) << 10;
// A photon phase that starts fewer than kWideItems histories per thread (the
// later generations among them) runs narrow: its last rounds, which few lanes
// fill, cost more than more warps hide.  1e6
// photons on 128^3 (7 a thread) take 0.50 ms of photon phases at 768 threads
// and 0.55 at 896, a 1e5 beamlet 0.26 and 0.27; 1e7 CT photons (73 a thread)
// 2.11 and 2.03, 3.3e7 lung photons 7 % less at 896.
constexpr int kNarrowThreads = std::min(768, PhaseShape<0>::threads);
constexpr uint64_t kWideItems = 64u;
// Beside large tables the electrons' step and event table, two thirds of
// theirs, stays in global memory (PT 2) and is read through the L1, so that
// the warps' stacks find room.  Staged, it leaves 24 warps a CTA beside 4
// materials of 512 energies, 18 beside 8, 11 beside 4 of 1500 and 4 beside the
// largest tables (8 of 1024); in global memory 24, 24, 24 and 22.  The line
// is where the two cost the same (staged -> global; 5e6 histories of the CT
// plan, 5e6 photons and 3e5 20 MeV electrons on 128^3): 24 warps 3.67 -> 3.70,
// 2.66 -> 2.69, 1.90 -> 1.92 ms; 20 warps 3.76 -> 3.73, 2.75 -> 2.71, 1.89 ->
// 1.95; 18 warps 3.85 -> 3.75, 2.82 -> 2.71, 1.93 -> 1.94; 17 warps 3.90 ->
// 3.75, 2.86 -> 2.72, 1.96 -> 1.95; 11 warps 4.31 -> 3.68, 3.25 -> 2.65, 2.22 ->
// 1.94; 4 warps 7.33 -> 3.93, 5.73 -> 2.71, 3.87 -> 1.95.
constexpr int kFarWarps = 18;
struct Launch {
    int pt;            // of the kernel: 0 photons, 1 electrons, 2 electrons beside large tables
    int threads;
    size_t smem;
};
static Launch phase_shape(const gdpm_ctx* ctx, const DevTables& T, int pt, bool narrow, size_t fixed_smem = 0) {
    const size_t stack = pt == 0 ? kPhStack * sizeof(PhRec) : sizeof(ElStack);
    const int want = ctx->block_threads > 0 ? ctx->block_threads
                     : pt == 0              ? (narrow ? kNarrowThreads : PhaseShape<0>::threads)
                                            : PhaseShape<1>::threads;
    auto fit = [&](int k) { return std::min(want, 32 * int((kMaxSmem - fixed_smem - smem_of(T, k)) / stack)); };
    int thr = fit(pt);
    if (pt == 1 && thr < std::min(want, 32 * kFarWarps)) thr = fit(pt = 2);
    return Launch{pt, thr, smem_of(T, pt) + stack * size_t(thr / 32)};
}

// CTAs of n primaries: see kSourceThreads.
static void source_shape(const gdpm_ctx* ctx, uint32_t n, uint32_t& grid, uint32_t& threads) {
    const uint32_t sms = uint32_t(ctx->sm_count);
    threads = n / uint32_t(kSourceThreads) >= sms ? uint32_t(kSourceThreads) : 256u;
    grid = threads == 256u ? n / 256u + 1u : sms;
}

// Persistent grid: SM count x resident CTAs per SM for this shared-memory size.
// share_eighths < 8 gives the grid that many eighths of the GPU: a large
// request that runs while small ones are active leaves SMs free for them,
// since persistent CTAs do not yield until their phase's input is drained.
int launch_phase(gdpm_ctx* ctx, Runner& r, cudaStream_t st, int particle, const SimParams& P,
                 const PhaseArgs& A, uint32_t n_items_hint, uint32_t share_eighths) {
    const uint64_t wide = kWideItems * uint64_t(ctx->sm_count) * uint64_t(PhaseShape<0>::threads);
    const Launch shape = phase_shape(ctx, P.T, particle == GDPM_PHOTON ? 0 : 1, A.n_src < wide);
    const int thr = shape.threads;
    const size_t smem = shape.smem;
    using Kernel = void (*)(const SimParams, const PhaseArgs);
    static const Kernel kernels[3][3] = {{k_phase<0, kPlain>, k_phase<0, kPair>, k_phase<0, kGeneral>},
                                         {k_phase<1, kPlain>, k_phase<1, kPair>, k_phase<1, kGeneral>},
                                         {k_phase<2, kPlain>, k_phase<2, kPair>, k_phase<2, kGeneral>}};
    const Kernel fn = kernels[shape.pt][P.hrec ? kGeneral : P.tally_mode ? kPair : kPlain];
    Runner::Resident* known = nullptr;
    for (Runner::Resident& q : r.resident) {
        if (q.fn == (const void*)fn && q.threads == thr && q.smem == smem) known = &q;
        if (known) break;
    }
    if (!known) {
        int ctas = 0;
        GDPM_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kMaxSmem)));
        GDPM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, fn, thr, smem));
        for (int k = 5; k > 0; --k) r.resident[k] = r.resident[k - 1];
        r.resident[0] = Runner::Resident{(const void*)fn, thr, ctas, smem};
        known = &r.resident[0];
    }
    const int bps = ctx->blocks_per_sm > 0 ? ctx->blocks_per_sm : known->ctas;
    if (bps < 1) return GDPM_E_ARG;
    uint32_t grid = uint32_t(ctx->sm_count) * uint32_t(bps);
    if (share_eighths < 8) grid = std::max(1u, grid * share_eighths / 8);
    if (n_items_hint > 0) {
        grid = std::min(grid, n_items_hint);   // a CTA has at least one particle
    }
    if (grid == 0) grid = 1;
    PhaseArgs B = A;
    const uint64_t warps = uint64_t(grid) * uint64_t(thr / 32);
    B.bank_block = bank_block(std::min(A.out_el.capacity, A.out_ph.capacity), warps);
    B.share_shift = share_shift(uint32_t(warps));
    // This phase's CTAs may start and stage their tables while the last ones of
    // the kernel before it run, except beside other requests, which then find
    // those SMs free.  A start costs some 5 us otherwise: 1e4 pencil photons (4
    // phases) 0.195 -> 0.170 ms, a 1e5 beamlet (8) 0.83 -> 0.77.
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(unsigned(thr));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &early;
    cfg.numAttrs = r.serving ? 0u : 1u;
    GDPM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, P, B));
    return GDPM_OK;
}

int launch_debug_philox(gdpm_ctx* ctx, const uint32_t* ctr, uint32_t k0, uint32_t k1,
                        uint32_t* out, uint64_t n) {
    const uint32_t grid = uint32_t(ctx->sm_count) * 4u;
    k_debug_philox<<<grid, 256, 0, ctx->stream>>>(ctr, k0, k1, out, n);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

int launch_debug_sample(gdpm_ctx* ctx, int kind, double a, double b, uint64_t n, uint64_t seed,
                        double* out1, double* out2) {
    const uint32_t grid = uint32_t(ctx->sm_count) * 4u;
    k_debug_sample<<<grid, 256, 0, ctx->stream>>>(kind, float(a), float(b), n, uint32_t(seed),
                                                   uint32_t(seed >> 32), out1, out2);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

int launch_debug_sources(gdpm_ctx* ctx, const SimParams& P, const PhaseArgs& A, uint64_t n,
                         double* out) {
    const uint32_t grid = uint32_t(ctx->sm_count) * 2u;
    k_debug_sources<<<grid, 256, 0, ctx->stream>>>(P, A, n, out);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

// The device-driven phase loop: a graph holding one conditional WHILE node
// whose body runs [Metropolis picks ->] photon phase -> electron phase ->
// control kernel; the control kernel advances the phase index and ends the
// loop when nothing is left (or at the phase cap).  The phase kernels use
// the persistent grids of launch_phase; L.bank_block is set here.
int build_loop_graph(gdpm_ctx* ctx, const SimParams& P, LoopArgs& L, bool metropolis,
                     cudaGraph_t* graph, cudaGraphExec_t* exec) {
    *graph = nullptr;
    *exec = nullptr;
    uint32_t grid[2];
    size_t smem[2];
    const void* const loops[3] = {(const void*)k_phase_loop<0>, (const void*)k_phase_loop<1>,
                                  (const void*)k_phase_loop<2>};
    const void* fn[2];
    int thr[2];
    uint64_t warps = 0;
    for (int t = 0; t < 2; ++t) {
        cudaFuncAttributes attr{};             // the arguments k_phase_loop derives in shared memory
        GDPM_CUDA_TRY(cudaFuncGetAttributes(&attr, loops[t]));
        const Launch shape = phase_shape(ctx, P.T, t, false, attr.sharedSizeBytes);
        fn[t] = loops[shape.pt];
        thr[t] = shape.threads;
        smem[t] = shape.smem;
        // one limit for every context's graph, as in launch_phase
        GDPM_CUDA_TRY(cudaFuncSetAttribute(fn[t], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           int(kMaxSmem - attr.sharedSizeBytes)));
        int bps = ctx->blocks_per_sm;
        if (bps <= 0) {
            GDPM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn[t], thr[t], smem[t]));
            if (bps < 1) return GDPM_E_ARG;
        }
        grid[t] = uint32_t(ctx->sm_count) * uint32_t(bps);
        warps = std::max<uint64_t>(warps, uint64_t(grid[t]) * uint64_t(thr[t] / 32));
        L.share_shift[t] = share_shift(grid[t] * uint32_t(thr[t] / 32));
    }
    L.bank_block = bank_block(std::min(L.qph.capacity, L.qe0.capacity), warps);

    cudaGraph_t g = nullptr;
    GDPM_CUDA_TRY(cudaGraphCreate(&g, 0));
    cudaGraphConditionalHandle h;
    cudaError_t e = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
    cudaGraphNodeParams cp{};
    cudaGraphNode_t wn = nullptr;
    if (e == cudaSuccess) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        e = cudaGraphAddNode(&wn, g, nullptr, nullptr, 0, &cp);
    }
    cudaGraph_t body = e == cudaSuccess ? cp.conditional.phGraph_out[0] : nullptr;
    SimParams Pc = P;
    LoopArgs Lc = L;
    void* phase_args_v[2] = {&Pc, &Lc};
    void* metro_args_v[2] = {&Pc, &Lc};
    uint32_t np, nc;
    {
        PhaseArgs probe{};
        probe.n_sub = L.n_sub;
        sources_smem(L.prefix_n, cdf_entries(P, probe), np, nc);
    }
    const size_t src_sm = size_t(nc) * 4 + size_t(np) * 4;
    void* src_args_v[4] = {&Pc, &Lc, &np, &nc};
    void* ctl_args_v[2] = {&Lc, &h};
    cudaGraphNode_t prev = nullptr;
    auto add = [&](const void* f, dim3 gd, dim3 bd, size_t sm, void** args) {
        if (e != cudaSuccess) return;
        cudaKernelNodeParams kp{};
        kp.func = const_cast<void*>(f);
        kp.gridDim = gd;
        kp.blockDim = bd;
        kp.sharedMemBytes = unsigned(sm);
        kp.kernelParams = args;
        cudaGraphNode_t n = nullptr;
        e = cudaGraphAddKernelNode(&n, body, prev ? &prev : nullptr, prev ? 1 : 0, &kp);
        prev = n;
    };
    if (metropolis)
        add((const void*)k_metropolis_loop, dim3((P.S.n_chains + kMetroChains - 1) / kMetroChains),
            dim3(kMetroThreads), 0, metro_args_v);
    {
        uint32_t sg, sthr;
        source_shape(ctx, L.chunk, sg, sthr);
        const void* sf = L.src_particle == GDPM_PHOTON ? (const void*)k_sources_loop<0> : (const void*)k_sources_loop<1>;
        add(sf, dim3(sg), dim3(sthr), src_sm, src_args_v);
    }
    add(fn[0], dim3(grid[0]), dim3(thr[0]), smem[0], phase_args_v);
    add(fn[1], dim3(grid[1]), dim3(thr[1]), smem[1], phase_args_v);
    add((const void*)k_loop_ctl, dim3(1), dim3(1), 0, ctl_args_v);
    cudaGraphExec_t x = nullptr;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&x, g, 0);
    if (e != cudaSuccess) {
        cudaGraphDestroy(g);
        last_cuda_error() = e;
        cudaGetLastError();
        return GDPM_E_CUDA;
    }
    *graph = g;
    *exec = x;
    return GDPM_OK;
}

int launch_sources(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, const PhaseArgs& A) {
    uint32_t grid, threads;
    source_shape(ctx, A.n_src, grid, threads);
    uint32_t np, nc;
    sources_smem(A.prefix_n, cdf_entries(P, A), np, nc);
    const size_t sm = size_t(nc) * 4 + size_t(np) * 4;
    if (P.S.particle == GDPM_PHOTON) {
        k_sources<0><<<grid, threads, sm, st>>>(P, A, np, nc);
    } else {
        k_sources<1><<<grid, threads, sm, st>>>(P, A, np, nc);
    }
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

int launch_metropolis_init(cudaStream_t st, const SimParams& P, uint32_t* chains) {
    k_metropolis_init<<<(P.S.n_chains + 255) / 256, 256, 0, st>>>(P, chains);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

int launch_metropolis(cudaStream_t st, const SimParams& P, uint32_t first, uint32_t n,
                      uint32_t* chains, uint32_t* pick) {
    k_metropolis<<<(P.S.n_chains + kMetroChains - 1) / kMetroChains, kMetroThreads, 0, st>>>(P, first, n, chains,
                                                                                              pick);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

int launch_debug_beamlets(cudaStream_t st, const SimParams& P, uint32_t first, uint64_t n,
                          const uint32_t* pick, int32_t* out) {
    const uint32_t grid = uint32_t(std::min<uint64_t>(1024u, (n + 255) / 256));
    k_debug_beamlets<<<grid, 256, 0, st>>>(P, first, n, pick, out);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

}  // namespace gdpm
