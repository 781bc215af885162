// Internal declarations of the CUDA library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <string>
#include <vector>

#include "qaoa.h"

namespace qaoa {

// ---------------------------------------------------------------------------
// Errors: every ABI entry point returns a status; the message is thread-local.
int set_error(int code, const char *fmt, ...);
int cuda_error(cudaError_t e, const char *what);
#define QAOA_CUDA_TRY(call)                                   \
    do {                                                      \
        cudaError_t e_ = (call);                              \
        if (e_ != cudaSuccess) return ::qaoa::cuda_error(e_, #call); \
    } while (0)

// ---------------------------------------------------------------------------
// Device facts, queried once per device.
struct DeviceInfo {
    int device = -1;
    int sms = 0;
    size_t smem_optin = 0;
    bool pageable = false;  // reads the host's pageable memory through its page tables
};
int device_info(DeviceInfo *out);

// ---------------------------------------------------------------------------
// Per-(device, stream) scratch owned by the library.  Grows on demand; the
// pinned host block receives results of device reductions.
// Pinned host memory that an asynchronous upload reads after the call that
// filled it has returned.
struct Upload {
    void *host = nullptr;
    size_t bytes = 0;
    cudaEvent_t sent = nullptr;  // recorded behind the upload
    bool pending = false;
};
constexpr unsigned UPLOADS = 32;  // uploads in flight per stream before a call waits for the oldest

struct Scratch {
    void *dev = nullptr;   // device bytes
    size_t dev_bytes = 0;
    void *host = nullptr;  // pinned host bytes
    size_t host_bytes = 0;
    int *fault = nullptr;  // pinned: set by a kernel whose grid barrier ran out of time
    Upload up[UPLOADS];
    unsigned next_up = 0;
};
// Returns scratch for `stream` on the current device with at least the given
// capacities (device, pinned host).  Not thread-safe per stream: one caller
// thread per stream at a time, as for any CUDA stream.
int scratch_for(cudaStream_t stream, size_t dev_bytes, size_t host_bytes, Scratch **out);
// Pinned memory of at least `bytes` for one upload, free of earlier ones (waits
// for the oldest when UPLOADS are in flight); upload_sent once its copy is
// enqueued.  The runtime may read a pageable source after cudaMemcpyAsync returns,
// where it does not stage it; this memory stays until the copy is done.
int upload_buffer(Scratch *s, size_t bytes, Upload **out);
int upload_sent(Upload *u, cudaStream_t stream);
// The stream's fault word, kept apart from the blocks that calls reuse.  A kernel may
// set it after its call has returned: scratch_for then refuses the next call on
// the stream, and stream_fault reports it to a call that has waited for the
// stream.  Reporting clears it.
int fault_word(cudaStream_t stream, int **out);
int stream_fault(cudaStream_t stream);
// Kernel attributes (the dynamic shared-memory limit) belong to a device:
// the current device's ordinal for per-device set-up state, or -1 with the
// error recorded when it is out of [0, MAX_DEVICES).
constexpr int MAX_DEVICES = 64;
int current_device_slot();

// ---------------------------------------------------------------------------
// Instrumentation: kernel kinds, launch counting and optional event timing.
enum KernelKind {
    K_COST_TABLE = 0,
    K_PASS_LOW,
    K_PASS_HIGH,
    K_SMALL_N,
    K_REDUCE,
    K_PSUCC,
    K_ADJ_LOW,
    K_ADJ_HIGH,
    K_ADJ_SEED,
    K_SERVE_SMALL,
    K_SAMPLE,
    K_FLIP_CHECK,
    K_MIRROR,
    K_ENCODE,
    K_MID,
    K_NUM_KINDS
};
// Call before / after a launch on `stream`.  `after` checks the launch status.
void profile_before(int kind, cudaStream_t stream);
int profile_after(int kind, cudaStream_t stream);

// Launches `k` with its launch overlapping the end of the kernel before it on the
// stream (programmatic stream serialization): its CTAs are placed as that one's
// leave, and prepare until pdl_wait.  Every kernel launched this way calls
// pdl_wait in every CTA, before it touches global memory, so it ends only after
// the kernels before it have.  n = 21, p = 7 (12 launches): 150 -> 115 us per
// evolution.  No kernel triggers its dependents early (griddepcontrol.
// launch_dependents): their waiting CTAs then shared the SMs with the running
// ones (n = 21: 135 us; n = 30, p = 10: 30.2 -> 31.8 ms).
template <class... P, class... A>
inline void launch_pdl(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const A &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k, args...);  // the status is taken by profile_after
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

// ---------------------------------------------------------------------------
// Pass plan: how one layer's mixer is split into HBM passes.  Pass 0 is the
// "low" pass over the contiguous tile bits [0, T); each further pass is a
// "high" pass whose tile is 2^row contiguous elements times 2^G rows strided
// by 2^lo (G = T - row, state bits [lo, lo + G)); it butterflies the top `bits`
// of those G bits (the others were mixed by an earlier pass).
struct Pass {
    int lo;    // lowest state bit of the tile's strided group
    int bits;  // qubits butterflied by this pass (the low pass: T)
    int row;   // contiguous low bits per tile row (the low pass: T)
};
struct Plan {
    int n = 0;
    int state_bits = 0;  // index bits of the stored state (n, or n - 1 when halved)
    int z2 = 0;          // halved by the global-flip symmetry
    int tile_bits = 0;   // T
    int n_passes = 0;
    Pass pass[8];
};
constexpr int T_C64 = 13;   // 2^13 complex64 = 64 KiB tile
constexpr int T_C128 = 12;  // 2^12 complex128 = 64 KiB tile
constexpr int G_MAX_C64 = 9;
constexpr int G_MAX_C128 = 8;
int make_plan(int n, int dtype, Plan *plan, bool z2 = false);
// Plan for a tile of 2^T amplitudes and high groups of at most gmax bits.
// With `wide`, groups that can spare a bit take gmax - 1 bits and rows of
// T - gmax + 1 bits instead (twice the contiguous bytes per row, which the
// HBM streams more efficiently at large strides); the top groups go wide first.
int make_plan_geo(int n, int T, int gmax, Plan *plan, bool z2 = false, bool wide = false);

// One launch of the forward evolution: pass `pass` of the plan for layer `la`.
// Modes: 0 = first pass of layer 0 (the state |+> is generated from the phase
// table), 1 = butterflies of one layer, 2 = butterflies of layer la, the phase
// of layer la + 1 and the butterflies of layer la + 1 on the same tile,
// 3 = the phase of layer la applied at load, then its butterflies.
// The qubit groups of a layer commute, so their order alternates between
// layers and the last pass of a layer fuses with the first of the next; the
// low pass always sits inside a layer (its fused form would be bound by the
// SMs rather than by HBM), so only high passes fuse.
struct Launch {
    int pass, la, mode;
};
enum PassMode { MODE_INIT = 0, MODE_PLAIN = 1, MODE_FUSED = 2, MODE_PHASE = 3 };
std::vector<Launch> make_schedule(int n_passes, int p);

// The backward (adjoint) sweep, layers p-1 down to 0.  Each launch undoes the
// butterflies of layer la on one group; the last pass of a layer also takes
// the phase term and undoes D_la (A_PHASE), and when layer la - 1 starts with
// the same group it goes on to undo that layer's butterflies too (A_FUSED).
// With two or more high groups the orders alternate ([1, 0, 2, ..., k] and
// [k, 0, k-1, ..., 1]) so every layer boundary fuses on a high group; with one
// high group each layer is [1, 0] with the phase in the low pass.
enum AdjMode { A_PLAIN = 0, A_PHASE = 1, A_FUSED = 2 };
std::vector<Launch> make_adj_schedule(int n_passes, int p);

// ---------------------------------------------------------------------------
// Host-side per-layer coefficients.  One mixer layer is
//   prod_j [c I + i S X_j] = sigma^n prod_j [A I + i B X_j]
// with (sigma, A, B) chosen so that A = 1 or B = 1 (one FMA per component).
// `arith` is the arithmetic of the kernels that take A and B: the non-unit
// coefficient is returned already rounded to it (exactly representable there)
// and sigma is derived from that rounded value.
enum Arith { ARITH_F32 = 0, ARITH_F64 = 1, ARITH_DF = 2 };
struct LayerCoef {
    double sigma, A, B;
    bool unit_a;  // true: A == 1, else B == 1
    double s2 = 1.0, s2_lo = 0.0;  // 1 / sigma^2 = s2 + s2_lo (beyond FP64)
};
// sigma^n and sigma^2, each within an ulp or two: the n-th power of a rounded
// sigma is off by n roundings, the same on every amplitude of a layer.
double layer_scale(const LayerCoef &k, int n);
double layer_sigma2(const LayerCoef &k);
LayerCoef layer_coef(double beta, int sign, int arith);
inline int arith_of(int dtype, int flags) {
    return dtype == QAOA_C64 ? ARITH_F32 : ((flags & QAOA_DF64) ? ARITH_DF : ARITH_F64);
}

// Phase table of one layer: T[c] = scale * exp(-i gamma c), c = 0..m (FP64 on
// the host; cast to the state's element type by the caller).  For complex64 and
// double-float tables (ARITH_F32, ARITH_DF) only every eighth entry is evaluated,
// the others are its products with exp(-i gamma b), b < 8, at a fifth of the time (a
// host that fills 10 layers of 129 entries ahead of one launch waits 30 us for them
// otherwise).  Their error is no larger for it, since the arguments' rounding is
// undone: against 80 bits, m up to 255, largest error of a complex64 entry 5.9e-8 of
// the scale either way; of a double-float one, |gamma| in 0.05 .. 0.8, 1.5e-14 with
// a cosine and sine of each rounded gamma c and 2.0e-15 this way, in 0.8 .. 3.2 5.8e-14
// and 2.0e-15.
void phase_table(double gamma, double scale, int m, int arith, double *re, double *im);

// Largest cost a phase table indexes.  The cost table is uint8, so
// C(x) <= 255 whatever m is: a table holds entries 0..table_top(m).
inline int table_top(int m) { return m < 255 ? m : 255; }
// Number of clause-count entries a phase table must hold.
constexpr int MAX_TABLE = 256;

// ---------------------------------------------------------------------------
// Cost-table internals shared by the cost-table and serving code.
struct ClauseRec {
    uint32_t hi_mask;  // mask of the clause's variables >= 5 (as bits of x)
    uint32_t hi_neg;   // negation pattern on those variables
    uint32_t all_true; // bit b: every literal on a variable < 5 is true at x = b (mod 32)
    uint32_t all_false;// bit b: every such literal is false at x = b (mod 32)
};
int encode_instance(const naesat_instance *inst, ClauseRec *out);
int validate_instance(const naesat_instance *inst);
// Launches the batched cost-table kernel: recs [batch][m_stride] on the device,
// m per instance on the device, results into d_stats [batch][2] (uint64 n_sol,
// uint64 max C) which must be zeroed first; nothing is written when *d_bad is set.  With d_ns == nullptr all
// instances have n qubits and consecutive tables; otherwise instance b has
// d_ns[b] <= n qubits and its table at d_costs + d_offs[b].  `mirror`: the
// tables are full ones (2^n entries), counted on their lower half and
// completed by the global-flip symmetry; false for the lower-half tables of
// the halved state (n then counts their index bits).
int launch_cost_table_batch(int batch, int n, const int *d_ns, const uint64_t *d_offs, const ClauseRec *d_recs,
                            const int *d_m, int m_stride, uint8_t *d_costs, unsigned long long *d_stats,
                            cudaStream_t stream, bool mirror, const unsigned long long *d_bad = nullptr);
// One table.  Up to 1023 clauses the records go as kernel parameters (no
// staging); a longer list is copied from h_big (pinned, and left alone until the
// copy is done) to d_big (device), cost_table_big_bytes(m) bytes each, 16-byte
// aligned, and counted chunk by chunk.
int launch_cost_table_one(const naesat_instance *inst, uint8_t *d_cost, unsigned long long *d_stats,
                          cudaStream_t stream, bool half, void *d_big, void *h_big);
size_t cost_table_big_bytes(int m);

// Multi-pass evolution of `batch` states (device side only, no host sync).
// `tables` holds p layers x (m + 1) complex FP64 entries (interleaved).
struct EvolveReq {
    int batch, n, m, p, dtype, flags;  // flags & QAOA_Z2_HALF: halved state and half cost tables
    const uint8_t *cost;
    void *state;
    void *adj;          // nullable: if set, the last pass also writes P psi into it
    const double *gamma, *beta;
    double *d_result;   // nullable: device [batch][2] (p_succ, norm)
    // Full tables, p > 0: device [batch][nslots] verdicts of the flip-symmetry
    // check, which the evolution fills first; a symmetric instance then evolves
    // half of its amplitudes.  Null: every amplitude is evolved.
    int *slots = nullptr;
    int nslots = 0;
};
// Runs the passes of `r` on `stream`; d_partials holds batch x gx x 2 doubles
// (gx from pass_grid_x); r.d_result (if set) receives [batch][2].
int evolve_device_impl(const EvolveReq &r, cudaStream_t stream, double *d_partials, int gx);
// `checked`: full tables that the passes check for flip symmetry.
int pass_grid_x(int dtype, int n, int batch, bool checked = false);
// Slots per instance of the flip-symmetry check.
int flip_slots(int n, int batch, int sms);
// Grid width per instance for `batch` instances of `tiles` tiles on `slots`
// resident CTAs (the wave-balanced choice; 1 <= result <= min(slots, tiles)).
int balanced_grid_x(int slots, int batch, uint64_t tiles);
// The same where `tiles` are halved on the device for flip-symmetric instances.
int checked_grid_x(int sms, int slots, int batch, uint64_t tiles);
// Fixed-order sums: out[g][k] = sum_j part[g][j][k] for g < groups, k < nv <= 4.
int launch_reduce(const double *part, int groups, int nblk, int nv, double *out, cudaStream_t stream);

// Small-n whole-evolution kernel for a packed batch (serving and n <= T).
struct SmallJob {
    const uint8_t *cost;  // device [2^n]
    void *state;          // device [2^n] (may be null: state not kept)
    double *result;       // device [2] (p_succ, norm)
    int n, m, p;
    int table_off;        // offset (in complex entries) of this job's tables
    int coef_off;         // offset (in layers) of this job's coefficients
};
// Tables and coefficients are in the kernel's own types (small_fill_layers:
// small_entry_bytes per table entry, small_coef_bytes per layer, 16-byte aligned).
// A job's arithmetic and sums depend on its own inputs only, whatever it is
// packed with.
size_t small_entry_bytes(int dtype);
size_t small_coef_bytes(int dtype);
void small_fill_layers(int dtype, int flags, int n, int m, int p, const double *gamma, const double *beta, void *tab,
                       void *coef);
int launch_small_batch(int dtype, int n_jobs, const SmallJob *d_jobs, const void *d_tables, const void *d_coefs,
                       int max_n, int flags, cudaStream_t stream);
// The evolutions of r (n at most small_n_limit) through the same kernel;
// r.d_result may be pinned host memory.  Tables too long for kernel parameters
// are staged: small_stage_bytes on the host (pinned) and the device.  Waits for
// the stream when it staged them or r.d_result is set.
size_t small_stage_bytes(int dtype, int m, int p);
int evolve_small(const EvolveReq &r, void *h_stage, void *d_stage, cudaStream_t stream);
// Whole evolutions (p >= 1, no adjoint seed) of as many mid-sized instances as
// the device holds at once, in one cooperative launch: *taken is false (and
// nothing was done) when r is not such a request.  With h_result (host [batch][2])
// waits for the results.
int evolve_mid(const EvolveReq &r, cudaStream_t stream, double *h_result, bool *taken);
// Gradients for n at most small_n_limit (through the stream's scratch).  Waits
// for the stream.
int grad_small(int batch, int n, const uint8_t *cost, int m, int p, const double *gamma, const double *beta, int dtype,
               int flags, cudaStream_t stream, double *p_succ, double *dgamma, double *dbeta);
// Largest n that the single-instance evolution runs in one CTA (the pass path
// needs n > T), and the largest n the packed small-n kernel accepts.
int small_n_limit(int dtype);
int small_n_pack_limit(int dtype);

}  // namespace qaoa
