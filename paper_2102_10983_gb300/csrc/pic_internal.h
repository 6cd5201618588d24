// Internal declarations shared by the translation units of libpic_gb300.so.
// Nothing here is part of the public ABI (include/pic_gb300.h is).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pic_gb300.h"

namespace pic {

constexpr int kMaxOrder = 5;
constexpr int kMaxK = 7;
// Binned schedule: smallest k whose sub-cycle is deferred to the next launch's
// first work items (shorter ones are compacted inside the warp); also the
// smallest predicted k the predicted schedule bins before a launch.
#ifndef PIC_DEFER_MIN
#define PIC_DEFER_MIN 3
#endif
constexpr int kDeferMin = PIC_DEFER_MIN;
// Predicted schedule: smallest predicted k that puts a particle in the
// predicted queue.  The long sub-cycles only: binning the short ones too (1)
// took them out of the stream's stashes but measured slower, the network
// over-predicting k = 2 and a predicted item costing more than a stream slot.
#ifndef PIC_PRED_MIN_K
#define PIC_PRED_MIN_K 3
#endif
constexpr int kPredMinK = PIC_PRED_MIN_K;

// Device counters of one context (accumulated by every push launch).
struct DevStats {
  unsigned long long k_hist[8];
  unsigned long long substeps;
  unsigned long long n_star;
  unsigned long long clamped;
  unsigned long long lost;
  int error;
  int pad;
};

// Row of the weight table for sub-step j (1-based) of a macro step with
// exponent k: rows are grouped by k, 4^k rows per k.
__host__ __device__ inline int64_t wrow(int k, int64_t j) {
  return (((int64_t)1 << (2 * k)) - 1) / 3 + (j - 1);
}
inline int64_t wrows_total(int k_max) { return wrow(k_max + 1, 1) + 1; }  // + criterion row

// The scale |q/m| dt / (2 Psi_max) of the FP64 kernels' FP32 criterion
// (criterion_f64_guess), 0 where that test does not apply.
__host__ __device__ inline float criterion_f64_scale(double qm_abs, double dt, double psi_max) {
  const double c = qm_abs * dt / (2.0 * psi_max);
  return (c >= 0x1p-60 && c <= 0x1p60 && psi_max >= 0x1p-500 && psi_max <= 0x1p500) ? (float)c : 0.0f;
}

// Whether the FP64 forms' node fields pay: one pass over the grid's entries per
// step, then one multiplication and one addition per grid and electron instead
// of its gather.  Per entry that pass costs what an electron's gather does (57
// ps: 30 FP64 operations), so a grid of more entries than electrons is not worth
// it.  Steps of m = 1 pushes, with the pass and without: 256 electrons in a
// window of 2^22 nodes 276 and 16 us; 1,048,576 electrons in 2^15 128 and 196;
// as many nodes as electrons, 131,072 41 and 40, 1,048,576 190 and 197.
__host__ __device__ inline bool node_fields_pay(int64_t electrons, int64_t entries) {
  return electrons >= entries;
}

// The electrons of a step that sub-cycle: k_sub[i] = their k (else 0), bin[1..7]
// the counts per k, bin[8..15] places taken so far, bin[16] the item cursor.
constexpr int kBinF64 = 32;  // counters in bin
struct BinF64 {
  int64_t n;
  const uint8_t* k_sub;
  int32_t* queue;
  int32_t* bin;
};

// Device memory for that, of at most `most` electrons (a power of two): queue,
// then k_sub, 5 bytes each in one allocation.  Without room for all of them
// (down to 65,536) for fewer, *slice: the passes then take that many at a time.
inline cudaError_t alloc_bin_f64(int64_t electrons, int64_t most, int32_t** queue, uint8_t** k_sub, int64_t* slice) {
  int64_t n = electrons < most ? electrons : most;
  for (;; n /= 2) {
    n = (n + 15) & ~(int64_t)15;  // k_sub is read in 16-byte words
    const cudaError_t e = cudaMalloc((void**)queue, (size_t)n * 5);
    if (e == cudaSuccess) {
      *k_sub = (uint8_t*)(*queue + n);
      *slice = n;
      return e;
    }
    *queue = nullptr;
    if (e != cudaErrorMemoryAllocation || n <= 65536) return e;
    cudaGetLastError();
  }
}

// Arguments of the FP64 push (one macro step).
struct PushArgsF64 {
  int64_t n;
  double* x;
  double* px;
  double* py;
  double* pz;
  uint8_t* status;
  const double* E[kMaxOrder + 1];  // ring slot of level n-p+l, l = 0..p
  const double* B[kMaxOrder + 1];
  double lo, hi;  // s = x/dx must satisfy lo <= s < hi (and s - 1/2 too)
  int32_t lo_i, hi_i;  // the same, clamped to 32 bits
  int64_t mask;   // W - 1
  double dt, inv_dx, psi_max, qm, qm_abs;
  int k_max;
  const double* wtab;  // rows of [E weights p+1 | B weights p+1]
  int64_t crit_row;
  DevStats* stats;
  double* work;  // nullptr, or per particle the accumulated work of E (App. B)
  float crit_scale;   // criterion_f64_scale: 0 = the exact criterion only
  double* nodes;      // nullptr, or 4 W: each node's fields at t_n (nodes_f64_kernel; node_fields_pay)
  int64_t slice;      // particles the passes take at a time (alloc_bin_f64)
  uint8_t* k_sub;     // per particle of a slice: k of the step where k > 0 (written every step)
  int32_t* queue;     // the slice's particles with k > 0, grouped by k
  int32_t* bin;       // [kBinF64] the step's counts and cursors, zeroed by its first launch
  int sms;            // set by the launcher
};

// From which k on, and in stretches of 4^k >> half sub-steps, the mixed form's
// sub-cycles run without a branch (subcycle_f32).
struct Stretches {
  int k_min, half;
};
constexpr int kNearMin = 2, kHalfMin = 3, kStretchMin = 8;
// cells: c dt / dx; k_min: the smallest k where that is at most one (kNearMin; 1
// for the plain schedule, whose warps of mixed k would run both loops one after the
// other).  With more cells per macro step a stretch of half a cell is a smaller part
// of it; k whose stretch would be shorter than kStretchMin, and k < kHalfMin, whose
// one stretch an electron could leave, look at the nodes in each sub-step.  262,144
// gyrating electrons at c dt = 4 dx, us per step, before these loops, in halves of a
// macro step (which nearly all electrons left, to be taken again), and so: plain
// schedule, k = 4 251, 335, 169; binned, k = 4 292, 380, 191; batch, k = 2 92, 120, 95.
inline Stretches stretches(double cells, int k_min) {
  Stretches r{k_min, 1};
  while (cells > (double)(1 << (r.half - 1)) && r.half < 16) ++r.half;
  if (r.half > 1)
    for (r.k_min = kHalfMin; r.k_min <= kMaxK && ((1 << (2 * r.k_min)) >> r.half) < kStretchMin;) ++r.k_min;
  return r;
}

// Arguments of the mixed-precision push.  Position = (cell + frac) * dx with
// an exact int32 cell and an FP32 offset.
struct PushArgsMixed {
  int64_t n;
  int32_t* cell;
  float* frac;
  float* px;
  float* py;
  float* pz;
  uint8_t* status;
  // fields, ring form (ringE != nullptr): a mirrored ring of 2R slots of lstride
  // floats, every level stored in slot (level mod R) and in that slot + R, so a
  // step's p+1 levels are consecutive from slot start_cur (previous step:
  // start_prev).  Pointer form (ringE == nullptr): one pointer per level.
  const float* ringE;
  const float* ringB;
  int64_t lstride;
  int64_t start_cur, start_prev;
  const float* E[kMaxOrder + 1];   // this step's levels n-p .. n
  const float* B[kMaxOrder + 1];
  const float* Ep[kMaxOrder + 1];  // previous step's levels (binned: deferred work)
  const float* Bp[kMaxOrder + 1];
  // per window node, E_y and B_z at t_n (theta = 1/2) and the steps to the next
  // node, {E, dE, B, dB}, written by the step's half-step kernel; nullptr = not
  // provided (gather the levels)
  const float4* nodes;
  // the predictor's feature nodes, E_y and B_z of every window node at t_{n+1}, W
  // + 1 each (node W repeats node 0)
  const float* featE;
  const float* featB;
  // per window node, the monomial coefficients of the temporal interpolant of
  // E_y (p+1) then B_z (p+1) for this step (coef) and the previous one
  // (coef_p); nullptr = form them from the levels
  const float* coef;
  const float* coef_p;
  // the tables of the last coef_steps steps, step s's at (s mod coef_steps)
  // coef_stride; a deferred particle in a step before coef_oldest (or the run's
  // first) forms its coefficients from the levels
  const float* coef_all;
  int64_t coef_stride, coef_oldest;
  int32_t coef_steps;
  int32_t item_tiles;  // tiles per stream item
  int32_t lo, hi;      // tent node j must satisfy lo <= j and j+1 <= hi
  int32_t lo_p, hi_p;  // same for the previous step
  int32_t mask;
  float dt, psi_max, qm, qm_abs;
  float inv_dx;
  int k_max;
  int field_time;  // 0: theta_j = 1/2 + (j-1)/m; 1: theta_j = (j - 1/2)/m
  Stretches near;
  // monomial coefficients, in u = theta - 1, of the Lagrange basis polynomials:
  // L^E_{p,l}(theta) = sum_q mono[0][l][q] u^q, L^B likewise with mono[1]
  float mono[2][kMaxOrder + 1][kMaxOrder + 1];
  const float* wtab;
  int64_t crit_row;
  DevStats* stats;
  // binned schedule: per-k queues (k = 1..7, qcap entries each), double-buffered
  const int32_t* queue_in;
  int32_t* queue_out;
  int32_t* qcount_in;   // [8], consumed by this launch, zeroed by its last block
  int32_t* qcount_out;  // [8], filled by this launch
  int64_t qcap;
  int* cursor;            // work cursor of the launch
  unsigned* blocks_done;  // blocks finished
  int parity_cur, parity_next;
  int finalize;
  int tma;  // 1: the six particle arrays are 16-byte aligned (stream tiles by bulk copy)
  // resumable long sub-cycles (ring form; lag_step == nullptr: every deferred
  // step is finished by the next launch).  A deferred particle is in macro
  // step step0 + lag_step[i] with lag_j[i] of its sub-steps done; a deferred
  // item spends at most heavy_budget sub-steps of long (k >= kDeferMin)
  // sub-cycles per launch and catches a lagging particle up with the stream.
  int32_t* lag_step;
  uint16_t* lag_j;
  int64_t step0;          // base of lag_step: the first step of the call (of the
                          // first call of a run of carried calls)
  int64_t step_cur;       // this launch's stream step (closing launch: last step + 1)
  int64_t keep_step;      // a particle may be left out of budget only in a step
                          // >= keep_step (INT64_MIN: any); below it the budget
                          // does not apply
  int32_t heavy_budget;   // <= 0: no limit
  int32_t ring_R;         // ring slots (levels at slot level mod R, mirrored at + R)
  const int64_t* slot_i0; // device copy of each slot's window origin
  // predicted schedule: electrons binned by predicted k at the last refresh of
  // the predictions (per-k queues, qcap entries each), marked in their status
  // byte; every launch until the next refresh pushes those still marked
  const int32_t* pred_queue;
  int32_t* pred_count;  // [8], set by the refresh's binning pass
};

// Fills PushArgsMixed::mono for order p (host side, FP64 expansion).
void lagrange_monomials(int p, float (&mono)[2][kMaxOrder + 1][kMaxOrder + 1]);

// The node coefficient tables (table_bytes each) of the steps a context keeps: a
// deferred particle a few steps behind the stream then reads a table as the
// others of its warp do, instead of a path of its own; as many as 256 MB hold,
// fewer (two at least) where there is no room.  Allocated after everything else
// that a context cannot do without.
inline cudaError_t alloc_coef_tables(size_t table_bytes, float** coef, int32_t* steps) {
  const size_t most = ((size_t)256 << 20) / (table_bytes > 0 ? table_bytes : 1);
  for (*steps = (int32_t)(most < 2 ? 2 : most > 16 ? 16 : most);; *steps = *steps > 4 ? *steps / 2 : 2) {
    const cudaError_t e = cudaMalloc((void**)coef, *steps * table_bytes);
    if (e == cudaSuccess) return e;
    *coef = nullptr;
    if (e != cudaErrorMemoryAllocation || *steps <= 2) return e;
    cudaGetLastError();
  }
}

// Sets the reason pic_last_error(NULL) reports.
void set_global_error(const char* msg);

// One ensemble of a batch, as the batched kernel reads it.
struct EnsDev {
  float dt, psi_max, qm, qm_abs, inv_dx;
  int32_t k_max, field_time, pad;
  const float* ringE;  // mirrored ring of this ensemble (2R slots x W)
  const float* ringB;
  const int64_t* slot_i0;  // [R] window origin of each ring slot
  double dx, inv_dx64;     // the cell and its reciprocal in FP64 (loading and reading particles)
  int64_t first, count;    // particle range in the concatenated store
  int64_t chunk_first;     // index of its first stream item
};

// Arguments of one batched macro step.
struct BatchArgs {
  int32_t n_ens;
  const EnsDev* ens;
  int64_t n_total, n_chunks;
  int32_t chunk_tiles;       // tiles per stream item
  const int32_t* chunk_ens;  // [n_chunks] the stream items' ensembles
  int32_t* cell;
  float* frac;
  float* px;
  float* py;
  float* pz;
  uint8_t* status;
  int64_t R, lstride;  // ring slots, W
  int32_t mask;
  int64_t start_cur, start_prev;
  Stretches near;  // for the ensemble with the most cells per macro step
  const float* wtab;
  int64_t crit_row;
  float mono[2][kMaxOrder + 1][kMaxOrder + 1];
  DevStats* stats;
  const int32_t* queue_in;  // ensemble e, k: entries from 7*first_e + (k-1)*count_e
  int32_t* queue_out;
  int32_t* qcount_in;   // [n_ens][8]
  int32_t* qcount_out;
  const int64_t* prefix;  // [7*n_ens + 1] heavy-item prefix (filled per launch)
  float4* nodes;          // [n_ens][W]: step_node_f32 of every node (filled per launch)
  int2* win;              // [n_ens] this step's windows [lo, hi] (filled per launch)
  const int2* win_p;      // and the previous step's
  const int2* win_all;    // the steps' kept, as coef_all, n_ens apart
  // [n_ens][W][2(p+1)]: every node's monomial coefficients of the temporal
  // interpolant (E_y then B_z) of this step (coef, filled per launch) and of
  // the previous one (coef_p); coef_all: the tables of the last steps kept,
  // step s's at (s mod steps_kept) coef_stride, from step oldest_kept on
  float* coef;
  const float* coef_p;
  const float* coef_all;
  int64_t coef_stride, oldest_kept;
  int32_t steps_kept;
  int* cursor;
  unsigned* blocks_done;
  int parity_cur, parity_next, finalize;
  // resumable long sub-cycles, as in PushArgsMixed: a deferred particle is in
  // step step0 + lag_step[i] with lag_j[i] of its sub-steps done; a deferred
  // item spends at most heavy_budget sub-steps of long sub-cycles per launch
  int32_t* lag_step;
  uint16_t* lag_j;
  int64_t step0, step_cur;
  int32_t heavy_budget;  // <= 0: no limit
};

cudaError_t launch_batch_step(const BatchArgs& a, int order, int blocks, cudaStream_t s,
                              int* launches);
int batch_max_blocks_per_sm(int order);
int batch_tile();  // particles per tile of the stream
cudaError_t launch_batch_chunks(const EnsDev* ens, int32_t n_ens, int64_t n_chunks, int32_t* chunk_ens,
                                cudaStream_t s);
cudaError_t launch_batch_scatter(const EnsDev* ens, int32_t n_ens, int64_t slot, int64_t R,
                                 int64_t W, const double* Ey, const double* Bz, const int64_t* i0,
                                 int64_t* slot_i0_all, cudaStream_t s);
// The mixed form's particle arrays (momenta and position) from some particle on.
struct MixedStore {
  int32_t* cell;
  float *frac, *px, *py, *pz;
};
// FP64 arrays <-> the mixed layout (convert.cu): n particles of one problem; of
// a batch, particles off .. off + n - 1 of the concatenated store, x .. pz (and
// what they point to) starting at particle off.  Outputs of launch_from_*
// may be NULL.
cudaError_t launch_to_mixed(const double* x, const double* px, const double* py, const double* pz,
                            const MixedStore& m, double inv_dx, int64_t n, cudaStream_t s);
cudaError_t launch_from_mixed(const MixedStore& m, double* x, double* px, double* py, double* pz,
                              double dx, int64_t n, cudaStream_t s);
cudaError_t launch_to_mixed_batch(const double* x, const double* px, const double* py, const double* pz,
                                  const MixedStore& m, const EnsDev* ens, int32_t n_ens, int64_t off,
                                  int64_t n, cudaStream_t s);
cudaError_t launch_from_mixed_batch(const MixedStore& m, double* x, double* px, double* py, double* pz,
                                    const EnsDev* ens, int32_t n_ens, int64_t n, cudaStream_t s);

// Launchers (return cudaError_t of the launch).
cudaError_t build_wtab_f64(double* wtab, int order, int k_max, int field_time, cudaStream_t s);
cudaError_t build_wtab_f32(float* wtab, const double* wtab64, int64_t count, cudaStream_t s);
// Groups the particles whose k_sub is set by k, k = 7 first (push_f64.cu).
cudaError_t launch_bin_f64(const BinF64& a, int sms, cudaStream_t s);
cudaError_t launch_push_f64(const PushArgsF64& a, int order, cudaStream_t s, int* launches);
cudaError_t launch_push_mixed(const PushArgsMixed& a, int order, int schedule, int sm_count,
                              cudaStream_t s, int* launches);
// One binned step (one launch); with a.finalize set, the closing launch of a
// call (the last step's deferred particles, then public status bytes).
cudaError_t launch_binned_step(const PushArgsMixed& a, int order, int sm_count, cudaStream_t main,
                               int* launches);
// E_y, B_z of every window node at t_n (the theta = 1/2 weights of a's step),
// and (coef != nullptr) every node's monomial coefficients, 2(p+1) floats.
cudaError_t launch_halfstep(const PushArgsMixed& a, int order, int64_t W, float4* nodes, float* coef,
                            cudaStream_t s);
// E_y, B_z of every window node extrapolated to t_{n+1} (theta = 3/2) from step
// a's levels, W + 1 nodes each: the predictor's field features.
cudaError_t launch_feature_nodes(const PushArgsMixed& a, int order, int64_t W, float* outE,
                                 float* outB, cudaStream_t s);
// Features of every particle (a.featE / a.featB: the feature nodes of a's step).
cudaError_t launch_features_mixed(const PushArgsMixed& a, int order, float* phi, cudaStream_t s);

// Rebuilds the predicted queue: clears the old queue's marks, then bins and
// marks the particles whose predicted k is >= min_k (and that the stream would
// take this step) into per-k queues; pred_count must be zero on entry.
cudaError_t launch_bin_predicted(const uint8_t* pred, uint8_t* status, int64_t n, int parity_cur,
                                 int min_k, int32_t* pred_queue, int32_t* pred_count, int64_t qcap,
                                 cudaStream_t s);

// predictor (mlp_bf16.cu, mlp_api.cu)
const float* mlp_device_params(const struct ::pic_mlp* m);
int mlp_param_count();
cudaError_t launch_mlp_infer(const float* P, const float* phi, int64_t n, uint8_t* pred,
                             int sm_count, cudaStream_t s);
// Features of step a's levels (theta = 3/2; a.featE / a.featB: the feature
// nodes) and the predicted class of every particle in one pass (the same
// predictions as features + launch_mlp_infer).  fieldless_zero: a particle
// that sees no field (E_y = B_z = 0 at its position) gets class 0 without the
// network, and a tile of such particles skips the network.
cudaError_t launch_predict_fused(const PushArgsMixed& a, int order, const float* P, uint8_t* pred,
                                 int sm_count, cudaStream_t s, bool fieldless_zero = false);
// Gradients of a batch as partial results per block (mlp_partial_floats), then
// their sum: into grad (optional) and *loss, and, lr > 0, the Adam step.
size_t mlp_partial_floats(int sm_count);
cudaError_t launch_mlp_grad(const float* P, const float* phi, const uint8_t* label, int64_t n,
                            float* part, int sm_count, cudaStream_t s);
cudaError_t launch_mlp_finish(const float* part, int64_t n, float* grad, float* loss, float* P, float* m1,
                              float* m2, float lr, int step, int sm_count, cudaStream_t s);

}  // namespace pic
