// Host-side definitions shared by the library's translation units.
#pragma once
#include <atomic>
#include <condition_variable>
#include <cstdint>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "common.cuh"

struct gdpm_source_state;   // a context's source (below)

namespace gdpm {

// The runtime's own record of the error is cleared: left there, it would fail
// the next call of this thread at its first launch check.
#define GDPM_CUDA_TRY(expr)                                   \
    do {                                                      \
        cudaError_t _e = (expr);                              \
        if (_e != cudaSuccess) {                              \
            last_cuda_error() = _e;                           \
            cudaGetLastError();                               \
            return GDPM_E_CUDA;                               \
        }                                                     \
    } while (0)

cudaError_t& last_cuda_error();

// Material constants needed by the table builder (device copy).
struct MatDev {
    int n;
    int Z[GDPM_MAX_ELEMENTS];
    double A[GDPM_MAX_ELEMENTS];
    double w[GDPM_MAX_ELEMENTS];
    double I;
};

// Source description as the kernels see it.
struct DevSource {
    int particle, geometry, annihilation, n_bins, n_beamlets;
    float origin[3], direction[3], center[3], axis_u[3], axis_v[3];
    float half_u, half_v;
    const float* edges;        // n_bins + 1
    // fluence map (Sec. 2.3.1), over the n_beamlets beamlets of positive weight
    const float* beamlets;     // n_beamlets * 16 (geometry rows, no weight)
    const float* bl_cdf;       // cumulative weights P(I+1), rounded up to FP32 (see BeamletHost)
    const int* bl_row;         // row of each listed beamlet in the caller's map
    const double* bl_f;        // weights f
    const uint64_t* al_cut;    // Walker alias cut-offs as Philox-word thresholds, and aliases
    const int* al_alias;
    int sampler;               // GDPM_SAMPLE_*
    uint32_t n_chains;         // Metropolis chains C
};

// Beamlet list and sampler tables of a fluence map, built on the host.
// cdf_up[k] is the smallest float >= cdf[k]: for a float uniform r,
// r < cdf_up[k] exactly when double(r) < cdf[k].  cut_t[k] counts the words
// x with (x + 1/2) / 2^32 < cut[k]: x < cut_t[k] exactly when that FP64
// comparison holds.  The device compares in FP32 and integers.
struct BeamletHost {
    std::vector<float> rows;   // 16 floats per listed beamlet
    std::vector<int> row;      // its row in the caller's map
    std::vector<double> f, cdf, cut;
    std::vector<int> alias;
    std::vector<float> cdf_up;
    std::vector<uint64_t> cut_t;
};
// all_rows keeps every row (in order) for dose-matrix runs, where row k is
// sub-problem k whatever its weight.
void beamlet_tables_host(const std::vector<double>& rows17, BeamletHost& out, bool all_rows = false);

// One transport phase (Sec. 2.2.1 Step 3f) in queue terms.
struct PhaseArgs {
    uint32_t n_src;            // primaries generated by this phase
    uint32_t src_first;        // global history id of the first of them
    uint32_t nb_small, nb_rem; // batches: the first nb_rem hold nb_small+1 histories, the rest nb_small
    const uint32_t* bin_prefix;// per batch: n_bins + 1 spectrum prefix counts
    uint32_t prefix_n;         // entries of bin_prefix
    const uint32_t* bl_pick;   // Metropolis: list position of each primary's beamlet
    Queue src;                 // this phase's primaries (slot i = primary i; E < 0: missed)
    Queue in;                  // particles consumed
    const uint32_t* in_count;  // count of `in` (device)
    uint32_t* head;            // pop counter of this phase (zeroed per batch)
    Queue out_ph, out_el;      // where secondaries are banked
    uint32_t* out_ph_count;
    uint32_t* out_el_count;
    // queue slots a warp reserves at a time (0: exactly what it pushes), and at
    // most half its even share of the phase's input (an eighth beyond 32
    // slots): a small phase would leave the next one mostly reserved slots
    // that were never written
    uint32_t bank_block;
    uint32_t share_shift;      // items >> share_shift: at most half a warp's even share of them
    // dose matrix: n_sub sub-problems (one per fluence-map row), sub-problem
    // k owning histories [sub_first[k], sub_first[k+1]) in nb_small batches
    // each; 0 for a single problem
    uint32_t n_sub, sub_batches;
    const uint32_t* sub_first;
};

// What the device-driven phase loop (a CUDA graph whose conditional WHILE
// node repeats photon phase k, electron phase k+1) needs to derive each
// phase's PhaseArgs from the phase index k held in device memory.
struct LoopArgs {
    Queue qph, qe0, qe1, qsrc;
    uint32_t* ctl;             // per-phase counter rows
    uint32_t* k;               // phase index of the current pass (even)
    uint32_t* status;
    const uint32_t* bin_prefix;
    uint32_t prefix_n;
    const uint32_t* sub_first;
    uint32_t* chains;          // Metropolis chain states and picks (or null)
    uint32_t* pick;
    uint32_t n_src, first, chunk;
    uint32_t nb_small, nb_rem, n_sub, sub_batches, bank_block;
    uint32_t share_shift[2];   // of the photon and the electron phases
    int src_particle, max_phases;
};

// Everything a transport kernel reads that does not change within a run.
struct SimParams {
    int nx, ny, nz;
    float dx, dy, dz, inv_dx, inv_dy, inv_dz, Lx, Ly, Lz;
    const uint8_t* mat;
    const float* rho;
    const float* maj;          // Woodcock majorant, n_e
    DevTables T;
    DevSource S;
    uint32_t key0, key1;
    RoundKeys keys;            // of (key0, key1)
    double* edep;              // FP64 batch tally (MeV)
    uint32_t batch_stride;     // voxels between batch grids (0: one grid for the current batch)
    float* edep_hi;            // FP32 compensated tally
    float* edep_lo;
    int tally_mode;
    int walk_trips;            // stretches of an electron's voxel walk per round of the phase loop
    unsigned long long* counters;
    double* ledger;
    uint32_t* status;
    int32_t* hrec;             // optional per-history records
    double* hrecd;
    uint32_t max_iters;
    // ranges the checked build tests indices against: tally cells
    // [tally_lo, tally_hi) of edep (or edep_hi/edep_lo), history records
    uint64_t tally_lo, tally_hi;
    uint64_t n_records;
};

struct Buffer {
    void* p = nullptr;
    size_t bytes = 0;
};
int ensure(Buffer& b, size_t bytes);
void release(Buffer& b);

}  // namespace gdpm

struct gdpm_tables {
    gdpm_ctx* ctx = nullptr;
    uint64_t id = 0;
    int n_mat = 0, n_e = 0, n_r = 0, n_a = 0;
    double e_min = 0, e_max = 0, eabs_ph = 0, eabs_el = 0, ms_loss = 0;
    int flags = 0;
    gdpm::Buffer ph_tot, ph_cum, el, rinv, atab;
    gdpm::DevTables dev{};
    size_t smem_photon = 0, smem_electron = 0;
};

struct gdpm_phantom {
    gdpm_ctx* ctx = nullptr;
    int nx = 0, ny = 0, nz = 0;
    float dx = 0, dy = 0, dz = 0;
    gdpm::Buffer mat, rho, rhomax;   // rhomax: 256 floats, max density per material index
    float rhomax_host[256] = {};
    std::map<uint64_t, gdpm::Buffer> maj;    // Woodcock majorant per table set id
};

namespace gdpm {

// A named NVTX range over a scope (seen by nsys and other NVTX tools; costs
// nothing when no tool is attached).
struct Range {
    explicit Range(const char* name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
    Range(const Range&) = delete;
    Range& operator=(const Range&) = delete;
};

// Device work buffers of a context, grown on demand.
struct Workspace {
    Buffer edep, s1, s2, hi, lo;          // tallies (V doubles / floats)
    Buffer edep2, hi2, lo2;               // second batch tally (folded while the next batch runs)
    size_t tally_bytes = 0;               // bytes of the all-batches tally (concurrent batches)
    // Leading bytes of edep known to be zero: set when a calculation's fold
    // (which clears the grids it reads) has completed; taken and reset by
    // prepare_workspace, which hands it to the calculation it sets up as
    // edep_zero (0 if edep was reallocated).
    size_t edep_clean = 0, edep_zero = 0;
    Buffer qph, qel0, qel1;               // particle queues
    uint32_t cap_ph = 0, cap_el = 0;
    Buffer qsrc;                           // primaries of one source phase
    uint32_t cap_src = 0;
    Buffer ctl;                            // per-phase counters (uint32)
    Buffer inputs;                         // a calculation's small inputs (source_upload):
    const uint32_t* prefix = nullptr;      //   per-batch spectrum prefix counts,
    uint32_t prefix_n = 0;                 //   how many; edges, fluence map, samplers
    Buffer run;                            // run statistics: counters, ledger, status
    Buffer chains, pick;                   // Metropolis chain states; picks of one phase
    Buffer sub_first, sub_inv, sub_nbig;   // dose matrix: sub-problem history ranges, batch sizes
    Buffer loop_k;                         // device-driven phase loop: the phase index
    Buffer stage;                          // device staging for host outputs
    Buffer pinned_host;                    // pinned host block for small readbacks
    Buffer pinned_stage;                   // pinned staging block of the inputs
};

// Launch wrappers (defined next to their kernels); all work goes to `st`.
int build_tables_device(gdpm_ctx* ctx, gdpm_tables* t, const gdpm_material_desc* mats);
int phantom_density_max(gdpm_ctx* ctx, gdpm_phantom* ph);
int launch_majorant_into(cudaStream_t st, gdpm_phantom* ph, gdpm_tables* t, float* maj);
struct Runner;
int launch_phase(gdpm_ctx* ctx, Runner& r, cudaStream_t st, int particle, const SimParams& P,
                 const PhaseArgs& A, uint32_t n_items_hint, uint32_t share_eighths = 8);
int launch_fold_into(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, uint32_t nb,
                     double* s1, double* s2);
int launch_fold_batches(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, int n_batches,
                        uint32_t nb_small, uint32_t nb_rem, double* s1, double* s2);
// The whole calculation's grids into dose and sigma, Dmax and the Sec. 3.1
// metric (both outputs are needed); the grids are left zeroed.
int launch_fold_final(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, int n_batches,
                      uint32_t nb_small, uint32_t nb_rem, double* dose, double* sigma);
int launch_finalize_into(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V,
                         int n_batches, const double* s1, const double* s2, double* dose,
                         double* sigma);
int launch_debug_philox(gdpm_ctx* ctx, const uint32_t* ctr, uint32_t k0, uint32_t k1,
                        uint32_t* out, uint64_t n);
int launch_debug_sample(gdpm_ctx* ctx, int kind, double a, double b, uint64_t n, uint64_t seed,
                        double* out1, double* out2);
int launch_debug_sources(gdpm_ctx* ctx, const SimParams& P, const PhaseArgs& A, uint64_t n,
                         double* out);
int launch_metropolis_init(cudaStream_t st, const SimParams& P, uint32_t* chains);
// Make the A.n_src primaries of a source phase into A.src (before the phase).
int launch_sources(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, const PhaseArgs& A);
// Build the device-driven phase loop as an instantiated CUDA graph.
int build_loop_graph(gdpm_ctx* ctx, const SimParams& P, LoopArgs& L, bool metropolis,
                     cudaGraph_t* graph, cudaGraphExec_t* exec);
int launch_metropolis(cudaStream_t st, const SimParams& P, uint32_t first, uint32_t n,
                      uint32_t* chains, uint32_t* pick);
int launch_debug_beamlets(cudaStream_t st, const SimParams& P, uint32_t first, uint64_t n,
                          const uint32_t* pick, int32_t* out);
int launch_fold_sub(gdpm_ctx* ctx, cudaStream_t st, const SimParams& P, size_t V, uint32_t k0,
                    uint32_t nk, int nb, const double* inv_n, const uint32_t* nbig, double* dose,
                    double* sigma);
int transport_smem(const gdpm_tables* t, int particle);

// Everything one dose calculation needs besides its inputs: streams, events,
// work buffers and profiling state.  A context has one for gdpm_simulate;
// each serving slot has its own, so calculations can run side by side.
struct Runner {
    cudaStream_t stream = nullptr;        // main stream (the context's, or owned)
    cudaStream_t side = nullptr;          // batch folds overlap the next batch here
    bool owns_stream = false;
    bool serving = false;                 // a serving slot: shares the GPU with the other slots
    bool small = false;                   // serving a small request now
    cudaStream_t prio_hi = nullptr, prio_lo = nullptr;   // serving: small / large requests
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    cudaEvent_t batch_done[2] = {nullptr, nullptr}, fold_done[2] = {nullptr, nullptr};
    Workspace ws;
    std::vector<cudaEvent_t> prof_events;
    std::vector<int> prof_kind;
    // device-driven phase loop: the instantiated graph and what it was built for
    cudaGraph_t loop_graph = nullptr;
    cudaGraphExec_t loop_exec = nullptr;
    std::vector<unsigned char> loop_key;
    // resident CTAs per SM of the phase kernels this runner launched (asking
    // the runtime costs as much as a launch)
    struct Resident {
        const void* fn = nullptr;
        int threads = 0, ctas = 0;
        size_t smem = 0;
    } resident[6];
};
int runner_init(Runner& r, cudaStream_t stream, bool own_stream);
// Electron phase form of a run: 1 resumable steps, 0 whole steps.
int walk_form(const gdpm_ctx* ctx);

// Host helpers shared by gdpm_simulate's runner and the allocation-free
// entry point (api.cu).
// Histories of one batch allotted to the spectrum intervals (n_bins + 1
// prefix counts): floor, then the remainder to the largest fractional parts.
void allot_prefix(const std::vector<double>& w, uint64_t nb, uint32_t* prefix);
// True for device or managed memory.
bool is_device_ptr(const void* p);
// View of a queue of `cap` slots at `base`.
Queue queue_view(void* base, uint32_t cap);
// The transport parameters of a calculation on this phantom and table set
// (geometry, tables, Philox key, tally mode, electron phase form, one grid).
SimParams base_params(gdpm_ctx* ctx, gdpm_phantom* ph, gdpm_tables* tb, uint32_t request_id);
// The source's scalar fields; its device arrays are left unset.
void source_fields(const ::gdpm_source_state& s, DevSource& d);
void runner_free(Runner& r);

}  // namespace gdpm

struct gdpm_source_state {
    gdpm_source_desc desc{};
    std::vector<double> edges, weights, beamlets;
    bool set = false;
};

// A serving request and its resident results.
struct gdpm_request {
    uint64_t id = 0;
    gdpm_request_desc desc{};
    gdpm_source_state src;
    int status = 1;          // 1 queued/running, 0 done ok, <0 failed
    gdpm::Buffer result;     // device: dose then sigma (2 x V doubles)
    gdpm_stats stats{};
};

struct gdpm_ctx {
    int device = 0;
    uint64_t seed = 0;
    int sm_count = 0;
    // parameters
    uint32_t queue_capacity = 0;
    int block_threads = 0;          // 0: each phase kernel's own CTA shape
    int blocks_per_sm = 0;
    int tally_mode = 0;
    uint32_t source_chunk = 0;
    uint32_t auto_chunk = 1u << 23;            // side-by-side phase length when source_chunk is 0
    int max_phases = 512;
    uint32_t max_iters = 1u << 22;             // loop trips per warp and phase
    gdpm::Buffer atab_cache;                   // ln A(ln G1) table: the same for every material set
    uint32_t request_id = 0;
    int speculative = 2;
    int profile = 0;
    int overlap_fold = 1;
    int use_graph = 0;                         // device-driven phase loop (CUDA graph)
    int electron_walk = 2;                     // GDPM_PARAM_ELECTRON_WALK
    float metric_min_rho = 0.05f;              // sigma/Dmax over voxels at least this dense
    int batch_mode = 0;                        // 0 auto, 1 sequential, 2 side by side
    uint64_t concurrent_max_hist = 4000000000ull;   // auto: histories per batch for side by side
    size_t concurrent_max_bytes = size_t(16384) << 20;
    int serve_slots = 4;
    size_t serve_reserve = size_t(1) << 30;   // device bytes kept free when admitting
    uint64_t serve_small_hist = 1000000;       // requests up to this size are "small"
    int serve_big_slots = 1;                   // slots for large requests (the rest serve small ones)
    uint32_t serve_phase_cap = 0;              // primaries per phase of a served request (0: as alone)
    int serve_share8 = 7;                      // eighths of the SMs large requests launch on while
                                               // small ones run
    // source
    gdpm_source_state src;
    // work of gdpm_simulate; `stream` aliases run.stream for the no-allocation path
    gdpm::Runner run;
    cudaStream_t stream = nullptr;
    int32_t* hrec = nullptr;
    double* hrecd = nullptr;
    uint64_t hrec_n = 0;
    uint64_t next_tables_id = 1;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;   // aliases of run.ev0/ev1
    std::mutex maj_mu;                           // majorant cache of shared phantoms
    // serving
    std::mutex mu;
    std::condition_variable cv;
    std::deque<gdpm_request*> pending;
    std::map<uint64_t, std::unique_ptr<gdpm_request>> requests;
    std::vector<std::thread> workers;
    std::vector<gdpm::Buffer> result_pool;     // finished results' buffers, reused (no cudaFree,
                                               // which would synchronize the whole device)
    std::atomic<int> running{0};
    std::atomic<int> small_running{0};         // small requests running now
    bool stop = false;
    uint64_t next_request = 1;
};
