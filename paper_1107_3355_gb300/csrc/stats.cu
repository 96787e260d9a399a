// Batch statistics (Sec. 2.2.1: mean dose and uncertainty from N_b batches;
// Sec. 3.1: sigma/Dmax over the D > 0.5 Dmax region) and the per-phantom
// Woodcock majorant.  These kernels stream voxel arrays in coalesced
// grid-stride loops sized to the SM count; the folds are bound by the FP64
// pipe before HBM.
#include <algorithm>
#include <cstring>

#include "internal.h"

namespace gdpm {
namespace {

// Largest density per material index (positive floats order like their bit
// patterns, so an integer atomicMax on the bits is exact); counts voxels whose density is not a
// positive finite number (zero, negative, NaN or infinite).
__global__ void k_rhomax(const uint8_t* __restrict__ mat, const float* __restrict__ rho, size_t V,
                         int* rmax_bits, unsigned int* n_bad) {
    __shared__ int s_max[256];
    for (int k = threadIdx.x; k < 256; k += blockDim.x) s_max[k] = 0;
    __syncthreads();
    unsigned int bad = 0;
    for (size_t v = blockIdx.x * size_t(blockDim.x) + threadIdx.x; v < V;
         v += size_t(gridDim.x) * blockDim.x) {
        const float r = rho[v];
        if (!(r > 0.f) || isinf(r)) { ++bad; continue; }
        atomicMax(&s_max[mat[v]], __float_as_int(r));
    }
    if (bad) atomicAdd(n_bad, bad);
    __syncthreads();
    for (int k = threadIdx.x; k < 256; k += blockDim.x)
        if (s_max[k]) atomicMax(&rmax_bits[k], s_max[k]);
}

// mu_max(E_i) = (1 + 1e-6) max_m mu_m(E_i) rho_max,m over the materials
// present: the interpolated majorant then bounds every voxel's
// interpolated attenuation.
__global__ void k_majorant(const float* __restrict__ tot, const float* __restrict__ rmax, int n_mat,
                           int n_e, float* maj) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_e) return;
    float m = 0.f;
    for (int k = 0; k < n_mat; ++k) m = fmaxf(m, tot[k * n_e + i] * rmax[k]);
    maj[i] = m * (1.0f + 1e-6f);
}

__device__ __forceinline__ double block_sum(double v, double* s_red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        t = threadIdx.x < (blockDim.x >> 5) ? s_red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    return t;
}

// End of batch: x = E_b(v)/n_b (energy per history), sum x and x^2, clear
// the batch tally; accumulate the deposited energy into the ledger.
// Streams 48 B per voxel; every thread issues the loads of its four voxel
// pairs before any store, and the grid covers the data once.
constexpr int kFoldPairs = 4;

__global__ void __launch_bounds__(256) k_fold(SimParams P, size_t V, double inv_nb,
                                              double* __restrict__ s1, double* __restrict__ s2) {
    __shared__ double s_red[32];
    double dep = 0.0;
    const size_t n2 = V / 2;
    const size_t base = size_t(blockIdx.x) * blockDim.x * kFoldPairs + threadIdx.x;
    double2* __restrict__ a2 = reinterpret_cast<double2*>(s1);
    double2* __restrict__ b2 = reinterpret_cast<double2*>(s2);
    double2 e[kFoldPairs], a[kFoldPairs], b[kFoldPairs];
    if (P.tally_mode == 0) {
        double2* __restrict__ e2 = reinterpret_cast<double2*>(P.edep);
#pragma unroll
        for (int u = 0; u < kFoldPairs; ++u) {
            const size_t i = base + size_t(u) * blockDim.x;
            if (i < n2) { e[u] = e2[i]; a[u] = a2[i]; b[u] = b2[i]; }
        }
#pragma unroll
        for (int u = 0; u < kFoldPairs; ++u) {
            const size_t i = base + size_t(u) * blockDim.x;
            if (i < n2) e2[i] = make_double2(0.0, 0.0);
        }
    } else {
        float2* __restrict__ h2 = reinterpret_cast<float2*>(P.edep_hi);
        float2* __restrict__ l2 = reinterpret_cast<float2*>(P.edep_lo);
#pragma unroll
        for (int u = 0; u < kFoldPairs; ++u) {
            const size_t i = base + size_t(u) * blockDim.x;
            if (i < n2) {
                const float2 h = h2[i], l = l2[i];
                e[u] = make_double2(double(h.x) + double(l.x), double(h.y) + double(l.y));
                a[u] = a2[i];
                b[u] = b2[i];
            }
        }
#pragma unroll
        for (int u = 0; u < kFoldPairs; ++u) {
            const size_t i = base + size_t(u) * blockDim.x;
            if (i < n2) { h2[i] = make_float2(0.f, 0.f); l2[i] = make_float2(0.f, 0.f); }
        }
    }
#pragma unroll
    for (int u = 0; u < kFoldPairs; ++u) {
        const size_t i = base + size_t(u) * blockDim.x;
        if (i < n2) {
            dep += e[u].x + e[u].y;
            const double x0 = e[u].x * inv_nb, x1 = e[u].y * inv_nb;
            a2[i] = make_double2(a[u].x + x0, a[u].y + x1);
            b2[i] = make_double2(fma(x0, x0, b[u].x), fma(x1, x1, b[u].y));
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && (V & 1)) {
        double ev;
        if (P.tally_mode == 0) {
            ev = P.edep[V - 1];
            P.edep[V - 1] = 0.0;
        } else {
            ev = double(P.edep_hi[V - 1]) + double(P.edep_lo[V - 1]);
            P.edep_hi[V - 1] = 0.f;
            P.edep_lo[V - 1] = 0.f;
        }
        dep += ev;
        const double x = ev * inv_nb;
        s1[V - 1] += x;
        s2[V - 1] = fma(x, x, s2[V - 1]);
    }
    const double t = block_sum(dep, s_red);
    if (threadIdx.x == 0 && t != 0.0) atomicAdd(&P.ledger[L_DEPOSITED], t);
}

// Mean dose of a voxel and its standard error, MeV/g per history.  With n_b
// batches, x_b = E_b/n_b and volume V, the weights of a voxel's sums make
// x = sum x_b / (n_b V) and q = sum x_b^2 / (n_b (n_b - 1) V^2) at once, so
// that dose = x / rho and sigma = sqrt(q - x^2 / (n_b - 1)) / rho: about 16
// FP64 operations a voxel instead of 30, on a pipe that a fold of 10 grids
// kept three quarters busy (CT phantom, 10 grids of 1e6 histories: 0.54 ->
// 0.46 ms).  FP64 division and square root are slow on this part:
// 1/rho and sqrt() start from FP32 estimates and take one FP64 Newton step
// each (relative error ~1e-14).  The variance is a small difference where all
// batches dose a voxel alike, so the weights of the squares are made from the
// rounded weights of the sums.
struct FoldWeights {
    double xb, xs, qb, qs;     // of the sums over the long batches and over the short ones
    double k;                  // 1 / (n_b - 1)
};
__host__ __device__ __forceinline__ FoldWeights fold_weights(double inv_big, double inv_small, double x_scale,
                                                             double nb_k, double k) {
    const double xb = inv_big * x_scale, xs = inv_small * x_scale;
    return FoldWeights{xb, xs, xb * xb * nb_k, xs * xs * nb_k, k};
}
__device__ __forceinline__ double inverse(float rho) {
    const double y = double(1.0f / rho);
    return y * fma(-double(rho), y, 2.0);
}
// The estimate is taken of the variance's mantissa times 1 or 2 and the result
// given half the exponent, with integers: the variance itself, in MeV^2 per
// cm^6, leaves FP32's range where voxels are large and deposits small.
__device__ __forceinline__ double root(double var) {
    const int hi = __double2hiint(var);
    if (hi < 0x00100000 || hi >= 0x7ff00000) return 0.0;   // negative, zero or subnormal, not finite
    const int e = ((hi >> 20) - 1023) & ~1;
    const double m = __hiloint2double(hi - e * (1 << 20), __double2loint(var));   // var = m 2^e, m in [1, 4)
    const float y = rsqrtf(float(m));
    const double g = m * double(y), r = fma(g, fma(-g, double(0.5f * y), 0.5), g);
    return __hiloint2double(__double2hiint(r) + (e / 2) * (1 << 20), __double2loint(r));
}

// Sums of a thread's batch tallies b in [b0, b1) at its VPT voxels v,
// v + blockDim.x, ... over grids of V cells starting at slot `first`: sum e
// and sum e^2 per voxel, two FP64 operations per tally.  GB300's FP64 rate
// (about 5e11 FMA/s), not HBM, bounds a fold that spends them on every tally,
// and most tallies are zero: even a field of 1e6 histories a batch leaves
// four fifths of the CT phantom's voxels without a deposit in that batch.
// So UB batches are loaded at a time only to see which are nonzero, and the
// thread then walks its nonzero ones, in batch order, from L1 (adding zero
// would change no bit of a sum); a warp spends FP64 operations for the lane
// with the most.  Those tallies are then zeroed, after all of the chunk's
// loads, which leaves the grids ready for the next calculation.
// Measured with the finalize work in the same kernel (below) and the metric:
// CT phantom, 10 grids of one beamlet's 1e5 histories 0.98 -> 0.19 ms; 128^3
// slab, 100 grids of 1e4 histories each 0.93 -> 0.37 ms; CT plan, 100 grids of
// 1e6 histories each 3.7 -> 2.45 ms (6.7 GB read).  10 batches at a time (whole
// chunks of the usual 10, 20 and 100) at five CTAs per SM were best: 16 at
// four +9 to +20 %, 20 to 32 at two or three +15 to +60 %.
template <int VPT, int UB>
__device__ __forceinline__ void batch_sums(const SimParams& P, size_t V, size_t first, size_t v,
                                           int b0, int b1, double (&se)[VPT], double (&sq)[VPT],
                                           uint32_t (&have)[VPT]) {
    const bool pair = P.tally_mode != 0;
    for (int b = b0; b < b1; b += UB) {
        uint32_t mask[VPT] = {};
        const size_t k0 = (first + size_t(b)) * V + v;
        if (!pair) {
            unsigned long long bits[UB][VPT];
#pragma unroll
            for (int u = 0; u < UB; ++u)
#pragma unroll
                for (int i = 0; i < VPT; ++i)
                    bits[u][i] = (b + u < b1 && v + size_t(i) * blockDim.x < V)
                                     ? reinterpret_cast<const unsigned long long*>(P.edep)[k0 + u * V + i * blockDim.x]
                                     : 0ull;
#pragma unroll
            for (int u = 0; u < UB; ++u)
#pragma unroll
                for (int i = 0; i < VPT; ++i) mask[i] |= bits[u][i] ? 1u << u : 0u;
        } else {
#pragma unroll
            for (int u = 0; u < UB; ++u)
#pragma unroll
                for (int i = 0; i < VPT; ++i)
                    if (b + u < b1 && v + size_t(i) * blockDim.x < V) {
                        const size_t k = k0 + u * V + i * blockDim.x;
                        const uint32_t w = reinterpret_cast<const uint32_t*>(P.edep_hi)[k] |
                                           reinterpret_cast<const uint32_t*>(P.edep_lo)[k];
                        mask[i] |= w ? 1u << u : 0u;
                    }
        }
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const size_t ki = k0 + i * blockDim.x;
            have[i] |= mask[i];
            for (uint32_t m = mask[i]; m; m &= m - 1u) {
                const size_t k = ki + size_t(__ffs(m) - 1) * V;
                const double e = pair ? double(P.edep_hi[k]) + double(P.edep_lo[k]) : P.edep[k];
                se[i] += e;
                sq[i] = fma(e, e, sq[i]);
            }
            for (uint32_t m = mask[i]; m; m &= m - 1u) {
                const size_t k = ki + size_t(__ffs(m) - 1) * V;
                if (!pair) {
                    P.edep[k] = 0.0;
                } else {
                    P.edep_hi[k] = 0.f;
                    P.edep_lo[k] = 0.f;
                }
            }
        }
    }
}

// The tallies themselves instead of their sums, for at most 4 batches: the
// sums are then made with the rest of a voxel's FP64 work, by full warps.
template <int VPT, int NB>
__device__ __forceinline__ void batch_tallies(const SimParams& P, size_t V, size_t first, size_t v, int nbatch,
                                              double (&e)[VPT][NB], uint32_t (&have)[VPT]) {
    const bool pair = P.tally_mode != 0;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const size_t vi = v + size_t(i) * blockDim.x, k = (first + size_t(b)) * V + vi;
            const bool in = b < nbatch && vi < V;
            if (!pair) {
                e[i][b] = in ? P.edep[k] : 0.0;
                have[i] |= uint32_t(__double2hiint(e[i][b]) | __double2loint(e[i][b]));
            } else {
                const float hi = in ? P.edep_hi[k] : 0.f, lo = in ? P.edep_lo[k] : 0.f;
                e[i][b] = double(hi) + double(lo);
                have[i] |= __float_as_uint(hi) | __float_as_uint(lo);
            }
        }
#pragma unroll
    for (int i = 0; i < VPT; ++i)
        if (have[i])
#pragma unroll
            for (int b = 0; b < NB; ++b)
                if (b < nbatch) {
                    const size_t k = (first + size_t(b)) * V + v + size_t(i) * blockDim.x;
                    if (!pair) {
                        P.edep[k] = 0.0;
                    } else {
                        P.edep_hi[k] = 0.f;
                        P.edep_lo[k] = 0.f;
                    }
                }
}

// Voxels with dose, gathered by the threads of a CTA so that the FP64 work
// per voxel (weights, mean, 1/density, square root: about 16 operations) runs
// with full warps however few of a warp's voxels hold dose.
struct FoldItem {
    double v[4];      // sums over the long batches (e, e^2) and over the short ones, or the tallies
};
constexpr int kFoldThreads = 256;
struct FoldList {
    FoldItem item[2 * kFoldThreads];
    uint32_t vox[2 * kFoldThreads];
    uint32_t n;
};

// Loop of a fold over the CTA's voxels: read each voxel's tallies, hand a
// voxel without dose to `empty(voxel)` and the others, in full CTA-loads, to
// `full(voxel, eb, qb, es, qs)`.  UB: batches read at a time (batch_sums), or
// 0 for at most 4 batches (batch_tallies).
template <int VPT, int UB, class Full, class Empty>
__device__ __forceinline__ void fold_voxels(const SimParams& P, size_t V, size_t first, int nbig, int nbatch,
                                            FoldList& L, Full full, Empty empty) {
    auto item = [&](uint32_t j) {
        const FoldItem t = L.item[j];
        if constexpr (UB > 0) {
            full(size_t(L.vox[j]), t.v[0], t.v[1], t.v[2], t.v[3]);
        } else {
            double s[2] = {0.0, 0.0}, q[2] = {0.0, 0.0};
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (b < nbatch) {
                    if (b < nbig) {
                        s[0] += t.v[b];
                        q[0] = fma(t.v[b], t.v[b], q[0]);
                    } else {
                        s[1] += t.v[b];
                        q[1] = fma(t.v[b], t.v[b], q[1]);
                    }
                }
            full(size_t(L.vox[j]), s[0], q[0], s[1], q[1]);
        }
    };
    if (threadIdx.x == 0) L.n = 0u;
    __syncthreads();
    for (size_t base = size_t(blockIdx.x) * kFoldThreads * VPT; base < V;
         base += size_t(gridDim.x) * kFoldThreads * VPT) {
        const size_t v = base + threadIdx.x;
        FoldItem it[VPT];
        uint32_t some[VPT] = {};
        if constexpr (UB > 0) {
            double eb[VPT] = {}, qb[VPT] = {}, es[VPT] = {}, qs[VPT] = {};
            if (nbig > 0) batch_sums<VPT, UB>(P, V, first, v, 0, nbig, eb, qb, some);
            batch_sums<VPT, UB>(P, V, first, v, nbig, nbatch, es, qs, some);
#pragma unroll
            for (int i = 0; i < VPT; ++i) it[i] = FoldItem{{eb[i], qb[i], es[i], qs[i]}};
        } else {
            double e[VPT][4];
            batch_tallies<VPT, 4>(P, V, first, v, nbatch, e, some);
#pragma unroll
            for (int i = 0; i < VPT; ++i) it[i] = FoldItem{{e[i][0], e[i][1], e[i][2], e[i][3]}};
        }
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const size_t vi = v + size_t(i) * kFoldThreads;
            const bool have = some[i] != 0u;
            if (vi < V && !have) empty(vi);
            const uint32_t m = __ballot_sync(0xffffffffu, have);
            uint32_t at = 0u;
            if (m && (threadIdx.x & 31u) == 0u) at = atomicAdd(&L.n, uint32_t(__popc(m)));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & lanemask_lt());
            if (have) {
                L.item[at] = it[i];
                L.vox[at] = uint32_t(vi);
            }
            __syncthreads();
            // at most 255 left over plus 256 new ones: one full load at a time
            const uint32_t n = L.n;
            if (n >= uint32_t(kFoldThreads)) {
                item(n - kFoldThreads + threadIdx.x);
                __syncthreads();
                if (threadIdx.x == 0) L.n = n - kFoldThreads;
            }
            __syncthreads();
        }
    }
    if (threadIdx.x < L.n) item(threadIdx.x);
}

// All batches at once (batches run side by side, one tally grid each): per
// voxel a1 = sum_b E_b/n_b and a2 = sum_b (E_b/n_b)^2; the first n_big
// batches hold one history more.  FINAL: the grids hold the whole
// calculation, so the voxel's dose and sigma follow at once (out1, out2; and
// Dmax), with no sums written and read back.  Otherwise the sums of a run in
// parts accumulate in out1, out2.  The grids are left zeroed.
template <bool FINAL, int VPT, int UB>
__global__ void __launch_bounds__(kFoldThreads, 5) k_fold_batches(SimParams P, size_t V, int nbatch,
                                                               FoldWeights W, int n_big,
                                                               double* __restrict__ out1,
                                                               double* __restrict__ out2,
                                                               unsigned long long* dmax_bits,
                                                               float metric_min_rho) {
    __shared__ double s_red[32];
    __shared__ FoldList L;
    double dep = 0.0, mx = 0.0;
    fold_voxels<VPT, UB>(
        P, V, 0, min(n_big, nbatch), nbatch, L,
        [&](size_t v, double eb, double qb, double es, double qs) {
            double x = es * W.xs, q = qs * W.qs;
            dep += es;
            if (n_big > 0) {
                x = fma(eb, W.xb, x);
                q = fma(qb, W.qb, q);
                dep += eb;
            }
            if (FINAL) {
                const float r = P.rho[v];
                const double ir = inverse(r), d = x * ir;
                out1[v] = d;
                out2[v] = root(fma(-W.k * x, x, q)) * ir;
                if (r >= metric_min_rho) mx = fmax(mx, d);
            } else {
                out1[v] += x;
                out2[v] += q;
            }
        },
        [&](size_t v) {
            if (FINAL) {
                out1[v] = 0.0;
                out2[v] = 0.0;
            }
        });
    const double t = block_sum(dep, s_red);
    if (threadIdx.x == 0 && t != 0.0) atomicAdd(&P.ledger[L_DEPOSITED], t);
    if (FINAL) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0 && mx > 0.0)
            atomicMax(dmax_bits, (unsigned long long)__double_as_longlong(mx));
    }
}

// Dose matrix: sub-problem k (row k of the fluence map; blockIdx.y) tallied
// into slots k*nb .. k*nb+nb-1.  Writes its mean dose and standard error per
// voxel (MeV/g per history of that sub-problem) to dose[(k-k0)*V + v] and
// sigma[...]; with one batch only the dose.  inv_n[2k], inv_n[2k+1] are
// 1/(histories of a long batch) and 1/(histories of a short batch) of
// sub-problem k, whose first nbig[k] batches are the long ones.  The grids
// are left zeroed.  With two batches a thread has only two tallies a voxel to
// load, so it takes four voxels.  64 beamlets x 2 batches on the 128^3 slab
// (134M voxels of output, 12 % of them with dose): memset and fold 17 -> 1.5 ms.
template <int VPT, int UB>
__global__ void __launch_bounds__(kFoldThreads) k_fold_sub(SimParams P, size_t V, uint32_t k0, int nb,
                                                           const double* __restrict__ inv_n,
                                                           const uint32_t* __restrict__ nbig, double x_scale,
                                                           double k_sigma, double* __restrict__ dose,
                                                           double* __restrict__ sigma) {
    __shared__ double s_red[32];
    __shared__ FoldList L;
    const uint32_t k = k0 + blockIdx.y;
    const int n_big = int(min(nbig[k], uint32_t(nb)));
    __shared__ FoldWeights W;      // visible after fold_voxels' first barrier
    if (threadIdx.x == 0) W = fold_weights(inv_n[2 * k], inv_n[2 * k + 1], x_scale, nb * k_sigma, k_sigma);
    const bool with_sigma = sigma && nb > 1;
    double* const dk = dose + size_t(blockIdx.y) * V;
    double* const sk = with_sigma ? sigma + size_t(blockIdx.y) * V : nullptr;
    double dep = 0.0;
    fold_voxels<VPT, UB>(
        P, V, size_t(k) * nb, n_big, nb, L,
        [&](size_t v, double eb, double qb, double es, double qs) {
            double x = es * W.xs, q = qs * W.qs;
            dep += es;
            if (n_big > 0) {
                x = fma(eb, W.xb, x);
                q = fma(qb, W.qb, q);
                dep += eb;
            }
            const double ir = inverse(P.rho[v]);
            dk[v] = x * ir;
            if (with_sigma) sk[v] = root(fma(-W.k * x, x, q)) * ir;
        },
        [&](size_t v) {
            dk[v] = 0.0;
            if (with_sigma) sk[v] = 0.0;
        });
    const double t = block_sum(dep, s_red);
    if (threadIdx.x == 0 && t != 0.0) atomicAdd(&P.ledger[L_DEPOSITED], t);
}

// Mean and standard error per voxel in MeV/g per history, and Dmax, from the
// sums of all batches (batches run one after another, or in parts).  A voxel
// without dose skips the FP64 arithmetic.
__global__ void k_finalize(const double* __restrict__ s1, const double* __restrict__ s2,
                           const float* __restrict__ rho, size_t V, int nb, double dvol,
                           double* __restrict__ dose, double* __restrict__ sigma,
                           unsigned long long* dmax_bits, float metric_min_rho) {
    double mx = 0.0;
    const double x_scale = 1.0 / (nb * dvol), k = 1.0 / (nb - 1), q_scale = x_scale * x_scale * (nb * k);
    for (size_t v = blockIdx.x * size_t(blockDim.x) + threadIdx.x; v < V;
         v += size_t(gridDim.x) * blockDim.x) {
        const double a1 = s1[v], a2 = s2[v];
        double d = 0.0, sd = 0.0;
        if (a1 != 0.0 || a2 != 0.0) {
            const double x = a1 * x_scale;
            const float r = rho[v];
            const double ir = inverse(r);
            d = x * ir;
            sd = root(fma(-k * x, x, a2 * q_scale)) * ir;
            if (r >= metric_min_rho) mx = fmax(mx, d);
        }
        if (dose) dose[v] = d;
        if (sigma) sigma[v] = sd;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx > 0.0)
        atomicMax(dmax_bits, (unsigned long long)__double_as_longlong(mx));
}

// Sec. 3.1 precision metric: mean of sigma over voxels with D > 0.5 Dmax
// (both over voxels at least as dense as metric_min_rho: air voxels of tiny
// mass have meaningless dose noise).
__global__ void k_metric(const double* __restrict__ dose, const double* __restrict__ sigma,
                         const float* __restrict__ rho, size_t V,
                         const unsigned long long* dmax_bits, double* ledger, float metric_min_rho) {
    __shared__ double s_red[32];
    const double dmax = __longlong_as_double((long long)*dmax_bits);
    double acc = 0.0, cnt = 0.0;
    // Doses are not negative, so their order is that of their high words up to
    // a tie: an FP64 comparison of every voxel would take longer than reading
    // them (CT phantom 29 -> 13 us).
    const double half = 0.5 * dmax;
    const int half_hi = __double2hiint(half);
    const size_t step = size_t(gridDim.x) * blockDim.x;
    for (size_t v = blockIdx.x * size_t(blockDim.x) + threadIdx.x; v < V; v += 8 * step) {
        double d[8];                        // eight loads in flight
#pragma unroll
        for (int u = 0; u < 8; ++u) d[u] = v + u * step < V ? dose[v + u * step] : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (__double2hiint(d[u]) >= half_hi && v + u * step < V && d[u] > half && rho[v + u * step] >= metric_min_rho) {
                acc += sigma[v + u * step];
                cnt += 1.0;
            }
    }
    const double a = block_sum(acc, s_red);
    __syncthreads();
    const double c = block_sum(cnt, s_red);
    if (threadIdx.x == 0) {
        if (a != 0.0) atomicAdd(&ledger[L_SIGSUM], a);
        if (c != 0.0) atomicAdd(&ledger[L_SIGCNT], c);
    }
}

}  // namespace

int phantom_density_max(gdpm_ctx* ctx, gdpm_phantom* ph) {
    const size_t V = size_t(ph->nx) * ph->ny * ph->nz;
    int rc = ensure(ph->rhomax, 256 * sizeof(float) + 16);
    if (rc) return rc;
    GDPM_CUDA_TRY(cudaMemsetAsync(ph->rhomax.p, 0, 256 * sizeof(float) + 16, ctx->stream));
    int* bits = static_cast<int*>(ph->rhomax.p);
    unsigned int* bad = reinterpret_cast<unsigned int*>(bits + 256);
    k_rhomax<<<ctx->sm_count * 4, 256, 0, ctx->stream>>>(static_cast<const uint8_t*>(ph->mat.p),
                                                          static_cast<const float*>(ph->rho.p), V,
                                                          bits, bad);
    GDPM_CUDA_TRY(cudaGetLastError());
    unsigned int h[260];
    GDPM_CUDA_TRY(cudaMemcpyAsync(h, ph->rhomax.p, 257 * sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    GDPM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    if (h[256] != 0) return GDPM_E_ARG;
    for (int k = 0; k < 256; ++k) {
        float f;
        std::memcpy(&f, &h[k], 4);
        ph->rhomax_host[k] = f;
    }
    return GDPM_OK;
}

}  // namespace gdpm

namespace gdpm {

// Launchers with every buffer and the stream explicit (a dose calculation's
// buffers belong to its runner, or to the no-allocation static array).
int launch_majorant_into(cudaStream_t st, gdpm_phantom* ph, gdpm_tables* t, float* maj) {
    k_majorant<<<(t->n_e + 127) / 128, 128, 0, st>>>(static_cast<const float*>(t->ph_tot.p),
                                                     static_cast<const float*>(ph->rhomax.p),
                                                     t->n_mat, t->n_e, maj);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

int launch_fold_into(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, uint32_t nb,
                     double* s1, double* s2) {
    const size_t per_block = size_t(256) * kFoldPairs;
    const unsigned grid = unsigned(std::max<size_t>(1, (V / 2 + per_block - 1) / per_block));
    k_fold<<<grid, 256, 0, st>>>(P, V, 1.0 / double(nb), s1, s2);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

// Thread blocks of a fold over V voxels, VPT a thread: one wave of CTAs at
// most (each loops over its share), so that the per-CTA reductions stay few.
static unsigned fold_grid(gdpm_ctx* ctx, size_t V, int vpt, int ctas_per_sm) {
    const size_t need = (V + size_t(256) * vpt - 1) / (size_t(256) * vpt);
    return unsigned(std::max<size_t>(1, std::min<size_t>(need, size_t(ctx->sm_count) * ctas_per_sm)));
}

int launch_fold_batches(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, int n_batches,
                        uint32_t nb_small, uint32_t nb_rem, double* s1, double* s2) {
    k_fold_batches<false, 1, 10><<<fold_grid(ctx, V, 1, 5), kFoldThreads, 0, st>>>(
        P, V, n_batches, fold_weights(1.0 / double(nb_small + 1), 1.0 / double(nb_small), 1.0, 1.0, 0.0), int(nb_rem),
        s1, s2, nullptr, 0.f);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

static int launch_metric(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, const double* dose,
                         const double* sigma) {
    const unsigned long long* dmax_bits = reinterpret_cast<const unsigned long long*>(&P.ledger[L_DMAX]);
    const size_t need = (V + 1023) / 1024;
    const unsigned grid = unsigned(std::min<size_t>(std::max<size_t>(need, 1), size_t(ctx->sm_count) * 4));
    k_metric<<<grid, 256, 0, st>>>(dose, sigma, P.rho, V, dmax_bits, P.ledger, ctx->metric_min_rho);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

int launch_fold_final(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, int n_batches,
                      uint32_t nb_small, uint32_t nb_rem, double* dose, double* sigma) {
    const double dvol = double(P.dx) * P.dy * P.dz;
    unsigned long long* dmax_bits = reinterpret_cast<unsigned long long*>(&P.ledger[L_DMAX]);
    const double k = 1.0 / (n_batches - 1);
    k_fold_batches<true, 1, 10><<<fold_grid(ctx, V, 1, 5), kFoldThreads, 0, st>>>(
        P, V, n_batches,
        fold_weights(1.0 / double(nb_small + 1), 1.0 / double(nb_small), 1.0 / (n_batches * dvol), n_batches * k, k),
        int(nb_rem), dose, sigma, dmax_bits, ctx->metric_min_rho);
    GDPM_CUDA_TRY(cudaGetLastError());
    return launch_metric(ctx, st, P, V, dose, sigma);
}

int launch_fold_sub(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, uint32_t k0,
                    uint32_t nk, int nb, const double* inv_n, const uint32_t* nbig, double* dose,
                    double* sigma) {
    const double dvol = double(P.dx) * P.dy * P.dz;
    const double x = 1.0 / (nb * dvol), k = nb > 1 ? 1.0 / (nb - 1) : 0.0;
    const dim3 grid(fold_grid(ctx, V, 4, 2), nk);   // two CTAs per SM and beamlet: 8 were 6 % slower
    if (nb <= 4) k_fold_sub<4, 0><<<grid, kFoldThreads, 0, st>>>(P, V, k0, nb, inv_n, nbig, x, k, dose, sigma);
    else k_fold_sub<4, 4><<<grid, kFoldThreads, 0, st>>>(P, V, k0, nb, inv_n, nbig, x, k, dose, sigma);
    GDPM_CUDA_TRY(cudaGetLastError());
    return GDPM_OK;
}

int launch_finalize_into(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V,
                         int n_batches, const double* s1, const double* s2, double* dose,
                         double* sigma) {
    const double dvol = double(P.dx) * P.dy * P.dz;
    unsigned long long* dmax_bits = reinterpret_cast<unsigned long long*>(&P.ledger[L_DMAX]);
    k_finalize<<<ctx->sm_count * 4, 256, 0, st>>>(s1, s2, P.rho, V, n_batches, dvol, dose, sigma,
                                                    dmax_bits, ctx->metric_min_rho);
    GDPM_CUDA_TRY(cudaGetLastError());
    if (dose && sigma) {
        return launch_metric(ctx, st, P, V, dose, sigma);
    }
    return GDPM_OK;
}

}  // namespace gdpm
