// Batched ensembles: many independent problems (each its own dt, dx, Psi_max,
// q/m, k cap and sub-step field-time reading, and its own field ring; one
// Lagrange order and window size for all) advanced together, one persistent
// launch per macro step, the mixed-precision binned push of push_mixed.cu per
// particle.
//
// Work items, from one atomic cursor:
//  1. deferred items (k >= kDeferMin) of every ensemble, largest k first;
//  2. stream items: runs of tiles of one ensemble's particles, so a warp
//     streams one ensemble at a time (k = 1, 2 go to the warp stashes, whose
//     entries remember their ensemble).
// The chunk length and the grid are launch parameters (tuned by
// pic_batch_autotune).
#include <math.h>
#include <string.h>

#include "pic_internal.h"
#include "push_device.cuh"

namespace pic {

// Field view of ensemble e for the current (prev = false) or previous step;
// the steps' windows are formed once per step and ensemble (batch_halfstep_kernel).
template <int P>
__device__ __forceinline__ void ens_fields(const BatchArgs& a, const EnsDev& e, bool prev,
                                           StepFields<P, true>& F) {
  const int64_t q = &e - a.ens;
  const int64_t start = prev ? a.start_prev : a.start_cur;
  F.E.base = e.ringE + start * a.lstride;
  F.B.base = e.ringB + start * a.lstride;
  F.E.lstride = (int32_t)a.lstride;
  F.B.lstride = (int32_t)a.lstride;
  F.coef = (prev ? a.coef_p : a.coef) + q * a.lstride * (2 * (P + 1));
  const int2 win = __ldg((prev ? a.win_p : a.win) + q);
  F.lo = win.x;
  F.hi = win.y;
}

// The nodes all p + 1 levels from ring slot `start` cover, [lo, hi].
template <int P>
__device__ __forceinline__ int2 ens_window(const BatchArgs& a, const EnsDev& e, int64_t start) {
  int64_t lo = INT64_MIN, hi = INT64_MAX;
#pragma unroll
  for (int l = 0; l <= P; ++l) {
    const int64_t o = e.slot_i0[(start + l) % a.R];
    lo = o > lo ? o : lo;
    hi = o + a.lstride - 1 < hi ? o + a.lstride - 1 : hi;
  }
  return make_int2((int32_t)lo, (int32_t)hi);
}

__device__ __forceinline__ int64_t queue_slot(const BatchArgs& a, const EnsDev& e, int k,
                                              int64_t entry) {
  return 7 * e.first + (int64_t)(k - 1) * e.count + entry;
}

// Warp-aggregated enqueue into ensemble ens's queue of k (key = ens * 8 + k;
// key < 0: nothing).  All 32 lanes call this.
__device__ __forceinline__ void batch_enqueue(const BatchArgs& a, int key, int32_t i) {
  if (!__any_sync(0xffffffffu, key >= 0)) return;
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(peers) - 1;
  int base = 0;
  if (key >= 0 && lane == leader) base = atomicAdd(&a.qcount_out[key], __popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (key >= 0) {
    const EnsDev& e = a.ens[key >> 3];
    a.queue_out[queue_slot(a, e, key & 7, base + __popc(peers & ((1u << lane) - 1u)))] = i;
  }
}

struct BatchStash {
  Stash s;
  uint16_t ens[kStashCap];
};
static_assert(sizeof(BatchStash) % 16 == 0, "stashes follow each other in shared memory");

// Push the last min(n, 32) stashed particles, one per lane (stash_drain of the
// single-problem kernel, each particle with its ensemble's fields).
template <int P, bool WIDE>
__device__ __forceinline__ void batch_stash_drain(const BatchArgs& a, const BatchStash& S, int k, int& n,
                                                  unsigned long long* sh) {
  const int lane = threadIdx.x & 31;
  const int cnt = n < 32 ? n : 32;
  if (lane < cnt) {
    const int q = n - cnt + lane;
    const EnsDev& e = a.ens[S.ens[q]];
    StepFields<P, true> F;
    ens_fields<P>(a, e, false, F);
    const float4 va = S.s.a[q];
    const float2 vb = S.s.b[q];
    const int32_t i = __float_as_int(vb.y);
    MixedState s = {__float_as_int(va.x), va.y, va.z, va.w, vb.x};
    const bool ok = subcycle_f32<P, true, true>(F, a.wtab, a.mask, e.dt, e.inv_dx, e.qm, e.field_time, NearRule<WIDE>(a.near), a.mono,
                                                k, S.s.kp[q], 0.f, s);
    normalize(s);
    store_state(a, i, s);
    a.status[i] = ok ? (uint8_t)(k | (a.parity_next ? kParity : 0)) : (uint8_t)(k | PIC_STATUS_LOST);
    if (!ok) atomicAdd(&sh[11], 1ull);
  }
  __syncwarp();
  n -= cnt;
}

// Field view of macro step s of ensemble e from its mirrored ring: for a
// deferred particle that runs behind the stream.  With the step's table and
// window where they are kept, else from the slots' window origins.
template <int P>
__device__ __forceinline__ StepFields<P, true> ens_step_fields(const BatchArgs& a, const EnsDev& e,
                                                               int64_t s) {
  StepFields<P, true> F;
  const int64_t R = a.R, T = a.steps_kept, q = &e - a.ens;
  const int64_t start = ((s - P) % R + R) % R;
  F.E.base = e.ringE + start * a.lstride;
  F.B.base = e.ringB + start * a.lstride;
  F.E.lstride = (int32_t)a.lstride;
  F.B.lstride = (int32_t)a.lstride;
  F.coef = nullptr;
  int2 win;
  if (s >= a.oldest_kept) {
    const int64_t at = (s % T + T) % T;
    F.coef = a.coef_all + at * a.coef_stride + q * a.lstride * (2 * (P + 1));
    win = __ldg(a.win_all + at * a.n_ens + q);
  } else {
    win = ens_window<P>(a, e, start);
  }
  F.lo = win.x;
  F.hi = win.y;
  return F;
}

__device__ __forceinline__ void batch_defer_mark(const BatchArgs& a, int64_t i, int k_prev, int k,
                                                 int64_t s, int j = 0) {
  a.status[i] = (uint8_t)(k_prev | (k << 4));
  a.lag_step[i] = (int32_t)(s - a.step0);
  a.lag_j[i] = (uint16_t)j;
}

// Deferred particle i of ensemble ens (the batched form of heavy_particle):
// it is in step step0 + lag_step[i] with lag_j[i] of its sub-steps done.
// Finish that step and, if it ran behind the stream, every step up to the
// previous one (taking each step's criterion), spending at most heavy_budget
// sub-steps of long sub-cycles; then take the current step's criterion:
// pushed at once if k < kDeferMin, else deferred again.  Out of budget: it
// stays deferred where it is and resumes in the next launch.  finalize: bring
// it to the end of the last step only (public status).  key: ens * 8 + k of
// a re-deferral, else -1.
template <int P, bool WIDE>
__device__ __forceinline__ void batch_heavy(const BatchArgs& a, int ens, int64_t i,
                                            const float* wcrit, ThreadCounters& tc,
                                            unsigned long long* sh, int& key) {
  key = -1;
  const EnsDev& e = a.ens[ens];
  StepFields<P, true> Fp, Fc;
  ens_fields<P>(a, e, true, Fp);
  ens_fields<P>(a, e, false, Fc);
  const uint8_t st = a.status[i];
  int k = deferred_k(st);
  int k_prev = st & 7;
  MixedState s = {a.cell[i], a.frac[i], a.px[i], a.py[i], a.pz[i]};
  int64_t si = a.step0 + a.lag_step[i];
  int j0 = a.lag_j[i];
  int budget = !a.finalize && a.heavy_budget > 0 ? a.heavy_budget : INT_MAX;
  float b0 = 0.f;  // the criterion's B_z of step si (used when k = 0)
  auto store = [&]() {
    a.cell[i] = s.cell;
    a.frac[i] = s.frac;
    a.px[i] = s.ux;
    a.py[i] = s.uy;
    a.pz[i] = s.uz;
  };
  auto lose = [&]() {
    store();
    a.status[i] = (uint8_t)(k | PIC_STATUS_LOST);
    atomicAdd(&sh[11], 1ull);
  };
  for (;;) {
    // sub-steps j0+1 .. j1 of step si
    const int m = 1 << (2 * k);
    int j1 = m;
    if (k >= kDeferMin && m - j0 > budget) j1 = j0 + budget;
    bool ok;
    StepFields<P, true> Fs = si == a.step_cur ? Fc : Fp;
    if (si < a.step_cur - 1) Fs = ens_step_fields<P>(a, e, si);
    if (Fs.coef)
      ok = subcycle_f32<P, true, true>(Fs, a.wtab, a.mask, e.dt, e.inv_dx, e.qm, e.field_time, NearRule<WIDE>(a.near), a.mono,
                                       k, k_prev, b0, s, j0, j1);
    else  // further behind than the tables kept
      ok = subcycle_f32<P, true, false>(Fs, a.wtab, a.mask, e.dt, e.inv_dx, e.qm, e.field_time, NearRule<WIDE>(a.near),
                                        a.mono, k, k_prev, b0, s, j0, j1);
    if (k >= kDeferMin) budget -= j1 - j0;
    if (!ok) {
      lose();
      return;
    }
    if (j1 < m) {  // out of budget inside the sub-cycle: resume here next launch
      store();
      batch_defer_mark(a, i, k_prev, k, si, j1);
      key = ens * 8 + k;
      return;
    }
    normalize(s);
    if (si == a.step_cur) {  // the current step's short sub-cycle is done
      store();
      a.status[i] = (uint8_t)(k | (a.parity_next ? kParity : 0));
      return;
    }
    if (si == a.step_cur - 1) {
      if (a.finalize) {
        store();
        a.status[i] = (uint8_t)k;
        return;
      }
      int32_t je, jb;
      float we, wb;
      if (!tent_coords(s.cell, s.frac, Fc.lo, Fc.hi, je, we, jb, wb)) {
        lose();
        return;
      }
      bool capped;
      const int kn = criterion_f32<P>(Fc.B, wcrit, jb, wb, a.mask, s, e.qm_abs, e.dt, e.psi_max,
                                      e.k_max, capped, b0);
      count_step(tc, sh, kn, capped);
      if (kn >= kDeferMin) {
        store();
        batch_defer_mark(a, i, k, kn, a.step_cur);
        key = ens * 8 + kn;
        return;
      }
      // a short sub-cycle of the current step: the next pass of the loop
      k_prev = k;
      k = kn;
      si = a.step_cur;
      j0 = 0;
      continue;
    }
    // behind the stream: the next step's criterion, then its sub-cycle
    si += 1;
    Fs = si == a.step_cur - 1 ? Fp : ens_step_fields<P>(a, e, si);
    int32_t je, jb;
    float we, wb;
    if (!tent_coords(s.cell, s.frac, Fs.lo, Fs.hi, je, we, jb, wb)) {
      lose();
      return;
    }
    bool capped;
    const int kn = criterion_f32<P>(Fs.B, wcrit, jb, wb, a.mask, s, e.qm_abs, e.dt, e.psi_max,
                                    e.k_max, capped, b0);
    count_step(tc, sh, kn, capped);
    k_prev = k;
    k = kn;
    j0 = 0;
    if (k >= kDeferMin && budget <= 0) {
      store();
      batch_defer_mark(a, i, k_prev, k, si);
      key = ens * 8 + k;
      return;
    }
  }
}

// Every ensemble's window nodes at t_n (step_node_f32), every node's monomial
// coefficients of the temporal interpolant (to_monomial, the values the
// sub-cycles would form from the levels), and the step's windows.
template <int P>
__global__ void batch_halfstep_kernel(BatchArgs a) {
  constexpr int stride = 2 * (P + 1);
  const float* wB = a.wtab + a.crit_row * stride + (P + 1);
  const float* wE = a.wtab + wrow(0, 1) * stride;
  const int64_t W = a.lstride;
  const int64_t total = (int64_t)a.n_ens * W;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const EnsDev& e = a.ens[q / W];
    const int32_t c = (int32_t)(q % W);
    StepFields<P, true> F;
    F.E.base = e.ringE + a.start_cur * W;
    F.B.base = e.ringB + a.start_cur * W;
    F.E.lstride = (int32_t)W;
    F.B.lstride = (int32_t)W;
    a.nodes[q] = step_node_f32<P>(F.E, F.B, wE, wB, c, a.mask);
    float e0[P + 1], b0[P + 1];
    to_monomial1<P>(F.E, c, a.mono[0], e0);
    to_monomial1<P>(F.B, c, a.mono[1], b0);
    float* r = a.coef + q * stride;
#pragma unroll
    for (int k = 0; k <= P; ++k) {
      r[k] = e0[k];
      r[P + 1 + k] = b0[k];
    }
    if (c == 0) a.win[q / W] = ens_window<P>(a, e, a.start_cur);
  }
}

// Heavy-item prefix: items of (k, ensemble) in the order k = 7..1, ensemble
// ascending; prefix[q] = first item of entry q, prefix[7 * n_ens] = total.
__global__ void __launch_bounds__(1024) batch_prefix_kernel(const int32_t* qcount_in, int32_t n_ens, int32_t k_lo,
                                                            int64_t* prefix) {
  __shared__ long long part[32];
  const int n = 7 * n_ens, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  long long base = 0;  // items before this pass of 1,024 entries
  for (int q0 = 0; q0 < n; q0 += 1024) {
    const int q = q0 + threadIdx.x;
    const int k = 7 - q / n_ens;
    const long long c = q < n && k >= k_lo ? ((long long)qcount_in[(q % n_ens) * 8 + k] + 31) / 32 : 0;
    long long v = c;  // inclusive scan: in the warp, then over the warps' sums
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    if (lane == 31) part[warp] = v;
    __syncthreads();
    if (warp == 0) {
      long long w = part[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += u;
      }
      part[lane] = w;
    }
    __syncthreads();
    if (q < n) prefix[q] = base + (warp ? part[warp - 1] : 0) + v - c;
    base += part[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) prefix[n] = base;
}

// Block shape of the batched kernel: four blocks of five warps per SM (20
// warps at <= 102 registers, 93 used), measured faster than two of eight
// (16 warps; 104 registers), three of six (18) and three of seven (21, with
// spills) on the 512-ensemble workload: its serial sub-cycle chains want warps.
#ifndef PIC_BATCH_THREADS
#define PIC_BATCH_THREADS 160
#endif
constexpr int kBatchThreads = PIC_BATCH_THREADS;
constexpr int kBatchWarps = kBatchThreads / 32;
#ifndef PIC_BATCH_MIN_BLOCKS
#define PIC_BATCH_MIN_BLOCKS 4
#endif
// Dynamic shared memory: the warps' staged tiles, then their stashes.
constexpr size_t kBatchTileBytes = sizeof(Tile) * 2 * kBatchWarps;
constexpr size_t kBatchSmem = kBatchTileBytes + sizeof(BatchStash) * kBatchWarps * kStashK;
static_assert(kBatchTileBytes % 128 == 0, "stashes start aligned");

// A stream item is a run of whole tiles of kTile particles of one ensemble
// (tiles of the concatenated store: those at an ensemble's ends hold others'
// particles too, which the item leaves alone), staged in shared memory by bulk
// copies one tile ahead and pushed in rounds of 64, two particles per lane, as
// the single-problem kernel's stream (push_mixed.cu).  (One particle per lane
// from plain loads, the ensemble found by a search per chunk, its window from
// the ring per chunk and per parked particle: 17.8 warp instructions per
// particle of the 512-ensemble configuration, 13.8 so; 293 -> 265 us per step
// of 11.9M particles.)
template <int P, bool WIDE>
__global__ void __launch_bounds__(kBatchThreads, PIC_BATCH_MIN_BLOCKS) push_batch_kernel(BatchArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  Tile* tiles = reinterpret_cast<Tile*>(smem);  // [kBatchWarps][2]
  BatchStash* stashes = reinterpret_cast<BatchStash*>(smem + kBatchTileBytes);  // [kBatchWarps][kStashK]
  __shared__ __align__(8) uint64_t bars[kBatchWarps * 2];
  __shared__ unsigned long long sh[12];
  if (threadIdx.x < 12) sh[threadIdx.x] = 0ull;
  __syncthreads();
  constexpr int stride = 2 * (P + 1);
  const float* wcrit = a.wtab + a.crit_row * stride + (P + 1);
  ThreadCounters tc;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  Tile* my_tiles = tiles + 2 * warp;
  uint64_t* my_bars = bars + 2 * warp;
  BatchStash* my_stash = stashes + warp * kStashK;
  if (lane == 0) {
    mbar_init(my_bars);
    mbar_init(my_bars + 1);
    mbar_init_fence();
  }
  __syncwarp();
  uint32_t phase = 0;  // bit s: parity of stage s's next completion
  int stash_n[kStashK];
#pragma unroll
  for (int q = 0; q < kStashK; ++q) stash_n[q] = 0;
  const uint8_t want = a.parity_cur ? kParity : 0;
  const uint8_t done = a.parity_next ? kParity : 0;
  const int64_t n_heavy = a.prefix[7 * a.n_ens];
  const int64_t n_items = n_heavy + (a.finalize ? 0 : a.n_chunks);
  const uint64_t policy = evict_first_policy();

  auto drain = [&](bool all) {
#pragma unroll 1
    for (int q = 0; q < kStashK; ++q) {
      int n = 0;
#pragma unroll
      for (int r = 0; r < kStashK; ++r)
        if (r == q) n = stash_n[r];
      const int keep = all ? 0 : 31;
      if (n <= keep) continue;
#pragma unroll 1
      while (n > keep) batch_stash_drain<P, WIDE>(a, my_stash[q], q + 1, n, sh);
#pragma unroll
      for (int r = 0; r < kStashK; ++r)
        if (r == q) stash_n[r] = n;
    }
  };

  for (;;) {
    int claim = 0;
    if (lane == 0) claim = atomicAdd(a.cursor, 1);
    const int64_t t = __shfl_sync(0xffffffffu, claim, 0);
    if (t >= n_items) break;
    if (t < n_heavy) {
      int lo = 0, hi = 7 * a.n_ens - 1;  // last entry q with prefix[q] <= t
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.prefix[mid] <= t) lo = mid; else hi = mid - 1;
      }
      const int k = 7 - lo / a.n_ens, ens = lo % a.n_ens;
      const int64_t entry = (t - a.prefix[lo]) * 32 + lane;
      int key = -1;
      int32_t i = 0;
      if (entry < a.qcount_in[ens * 8 + k]) {
        i = a.queue_in[queue_slot(a, a.ens[ens], k, entry)];
        batch_heavy<P, WIDE>(a, ens, i, wcrit, tc, sh, key);
      }
      batch_enqueue(a, key, i);
      continue;
    }
    // stream item: which ensemble, which tiles
    const int64_t c = t - n_heavy;
    const int ens = __ldg(a.chunk_ens + c);
    const EnsDev& e = a.ens[ens];
    const int64_t e_first = e.first, e_end = e.first + e.count;
    const int64_t tile0 = e_first / kTile + (c - e.chunk_first) * a.chunk_tiles;
    const int64_t tile_last = (e_end - 1) / kTile;
    const int n_tiles = (int)(tile_last - tile0 + 1 < a.chunk_tiles ? tile_last - tile0 + 1 : a.chunk_tiles);
    const int2 win = __ldg(a.win + ens);
    const float dt = e.dt, qm = e.qm, qm_abs = e.qm_abs, psi_max = e.psi_max;
    const int k_max = e.k_max, k_short = k_max < kDeferMin - 1 ? k_max : kDeferMin - 1;
    const float hx0 = __fmul_rn(dt, e.inv_dx), qm_dt = __fmul_rn(qm_abs, dt);
    const float tp = __fmul_rn(2.0f, psi_max), tp2 = __fmul_rn(tp, tp);
    const float4* nodes = a.nodes + (int64_t)ens * a.lstride;

    auto whole = [&](int64_t tile) { return (tile + 1) * kTile <= a.n_total; };
    auto issue = [&](int stage, int r) {
      if (r < n_tiles && whole(tile0 + r) && lane == 0)
        tile_issue(a, my_tiles + stage, my_bars + stage, (tile0 + r) * kTile, policy);
    };
    issue(0, 0);
    issue(1, 1);
    bool gave_up = false;
#pragma unroll 1
    for (int r = 0; r < n_tiles; ++r) {
      const int stage = r & 1;
      const int64_t first = (tile0 + r) * kTile;
      const bool staged = whole(tile0 + r);
      const Tile& T = my_tiles[stage];
      if (staged) {
        if (!mbar_wait(my_bars + stage, (phase >> stage) & 1u)) {
          // the copies never completed: flag it for the host and leave the
          // stream, after one more bounded wait for each stage in flight
          if (lane == 0) atomicExch(&a.stats->error, 1);
          mbar_wait(my_bars + stage, (phase >> stage) & 1u);
          if (r + 1 < n_tiles && whole(tile0 + r + 1)) mbar_wait(my_bars + (stage ^ 1), (phase >> (stage ^ 1)) & 1u);
          gave_up = true;
          break;
        }
        phase ^= 1u << stage;
      }
#pragma unroll 1
      for (int h = 0; h < kTile / 64; ++h) {
        const int q = h * 32 + lane;
        const int64_t i = first + 2 * q;
        uint8_t st0 = PIC_STATUS_LOST, st1 = PIC_STATUS_LOST;
        MixedState2 s;
        if (staged) {
          const uint32_t st2 = reinterpret_cast<const uint16_t*>(T.st)[q];
          st0 = (uint8_t)st2;
          st1 = (uint8_t)(st2 >> 8);
          s.cell = reinterpret_cast<const int2*>(T.cell)[q];
          s.frac = reinterpret_cast<const float2*>(T.frac)[q];
          s.ux = reinterpret_cast<const float2*>(T.px)[q];
          s.uy = reinterpret_cast<const float2*>(T.py)[q];
          s.uz = reinterpret_cast<const float2*>(T.pz)[q];
        } else {
          MixedState u0 = {0, 0.5f, 0.f, 0.f, 0.f}, u1 = u0;
          if (i < a.n_total) {
            st0 = a.status[i];
            u0 = load_state(a, i);
          }
          if (i + 1 < a.n_total) {
            st1 = a.status[i + 1];
            u1 = load_state(a, i + 1);
          }
          s.cell = make_int2(u0.cell, u1.cell);
          s.frac = make_float2(u0.frac, u1.frac);
          s.ux = make_float2(u0.ux, u1.ux);
          s.uy = make_float2(u0.uy, u1.uy);
          s.uz = make_float2(u0.uz, u1.uz);
        }
        constexpr uint8_t kStreamMask = PIC_STATUS_LOST | kDeferMask | kParity;
        const bool mine0 = (st0 & kStreamMask) == want && i >= e_first && i < e_end;
        const bool mine1 = (st1 & kStreamMask) == want && i + 1 >= e_first && i + 1 < e_end;
        const PairNodes pn = pair_nodes(s, win.x, win.y);
        float2 ey, bz, a2, rhs;
        pair_fields(nodes, a.mask, pn, ey, bz);
        pair_psi(bz, s, qm_dt, tp2, a2, rhs);
        const bool big0 = a2.x > rhs.x, big1 = a2.y > rhs.y;
        bool push0 = mine0 && pn.in0 && !big0, push1 = mine1 && pn.in1 && !big1;
        int k0 = 0, k1 = 0;
        const bool side = !__all_sync(0xffffffffu, (push0 || !mine0) && (push1 || !mine1));
        if (side) {
          const int2 k = pair_short_k(a2, rhs);
          k0 = mine0 && pn.in0 && big0 ? k.x : 0;
          k1 = mine1 && pn.in1 && big1 ? k.y : 0;
          if (__any_sync(0xffffffffu, k0 > k_short || k1 > k_short || (mine0 && !pn.in0) || (mine1 && !pn.in1))) {
#pragma unroll 1
            for (int p = 0; p < 2; ++p) {  // long sub-cycles, caps below that, particles outside the window
              int kk = p ? k1 : k0;
              bool push = false;
              const uint8_t st = p ? st1 : st0;
              int key = -1;
              if ((p ? mine1 : mine0) && !(p ? pn.in1 : pn.in0)) {
                a.status[i + p] = (uint8_t)(st | PIC_STATUS_LOST);
                atomicAdd(&sh[11], 1ull);
              } else if (kk > k_short) {
                bool capped;
                const MixedState one = {0, 0.f, p ? s.ux.y : s.ux.x, p ? s.uy.y : s.uy.x, p ? s.uz.y : s.uz.x};
                kk = psi_to_k(p ? bz.y : bz.x, one, qm_abs, dt, psi_max, k_max, capped);
                tc.capped += capped ? 1u : 0u;
                if (kk == 0) {
                  push = true;  // capped at k_max = 0
                } else if (kk >= kDeferMin) {
                  atomicAdd(&sh[kk], 1ull);
                  batch_defer_mark(a, i + p, st & 7, kk, a.step_cur);
                  key = ens * 8 + kk;
                  kk = 0;
                }
              }
              batch_enqueue(a, key, (int32_t)(i + p));
              k0 = p ? k0 : kk;
              k1 = p ? kk : k1;
              push0 |= !p && push;
              push1 |= p && push;
            }
          }
          tc.k1 += (k0 == 1 ? 1u : 0u) + (k1 == 1 ? 1u : 0u);
          tc.k2 += (k0 == 2 ? 1u : 0u) + (k1 == 2 ? 1u : 0u);
        }
        tc.k0 += (push0 ? 1u : 0u) + (push1 ? 1u : 0u);
        if (push0 || push1) {
          const MixedState2 u = pair_push(s, ey, bz, st0, st1, dt, hx0, qm);
          if (push0 && push1) {  // i even: 8-byte stores
            __stcs(reinterpret_cast<int2*>(a.cell + i), u.cell);
            __stcs(reinterpret_cast<float2*>(a.frac + i), u.frac);
            __stcs(reinterpret_cast<float2*>(a.px + i), u.ux);
            __stcs(reinterpret_cast<float2*>(a.py + i), u.uy);
            __stcs(reinterpret_cast<float2*>(a.pz + i), u.uz);
            *reinterpret_cast<uint16_t*>(a.status + i) = (uint16_t)(done | (done << 8));
          } else if (push0) {
            store_stream(a, (uint32_t)i, MixedState{u.cell.x, u.frac.x, u.ux.x, u.uy.x, u.uz.x});
            a.status[i] = done;
          } else {
            store_stream(a, (uint32_t)i + 1, MixedState{u.cell.y, u.frac.y, u.ux.y, u.uy.y, u.uz.y});
            a.status[i + 1] = done;
          }
        }
        if (side) {  // park k = 1, 2 (push_mixed.cu), with the ensemble
          const unsigned lt = (1u << lane) - 1u;
          int pos0 = 0, pos1 = 0;
          bool full = false;
#pragma unroll
          for (int v = 0; v < kStashK; ++v) {
            const unsigned m0 = __ballot_sync(0xffffffffu, k0 == v + 1), m1 = __ballot_sync(0xffffffffu, k1 == v + 1);
            const int n0 = stash_n[v], n1 = n0 + __popc(m0);
            if (k0 == v + 1) pos0 = n0 + __popc(m0 & lt);
            if (k1 == v + 1) pos1 = n1 + __popc(m1 & lt);
            stash_n[v] = n1 + __popc(m1);
            full |= stash_n[v] >= 32;
          }
          if (k0 > 0) {
            BatchStash& S = my_stash[k0 - 1];
            stash_put(S.s, pos0, (int32_t)i, MixedState{s.cell.x, s.frac.x, s.ux.x, s.uy.x, s.uz.x}, st0 & 7);
            S.ens[pos0] = (uint16_t)ens;
          }
          if (k1 > 0) {
            BatchStash& S = my_stash[k1 - 1];
            stash_put(S.s, pos1, (int32_t)i + 1, MixedState{s.cell.y, s.frac.y, s.ux.y, s.uy.y, s.uz.y}, st1 & 7);
            S.ens[pos1] = (uint16_t)ens;
          }
          __syncwarp();
          if (full) drain(false);
        }
      }
      __syncwarp();  // every lane is done with the stage before it is refilled
      issue(stage, r + 2);
    }
    if (gave_up) break;
  }
  drain(true);
  flush_counters(tc, sh, a.stats);

  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned fin = atomicAdd(a.blocks_done, 1u);
    if (fin == gridDim.x - 1) {
      __threadfence();
      *a.cursor = 0;
      *a.blocks_done = 0;
      for (int q = 0; q < 8 * a.n_ens; ++q) a.qcount_in[q] = 0;
      __threadfence();
    }
  }
}

__global__ void batch_reset_status_kernel(uint8_t* status, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t st = status[i];
    const uint8_t pub = (uint8_t)(st & (PIC_STATUS_LOST | 7));
    if (pub != st) status[i] = pub;
  }
}

// The stream items' ensembles (chunk_first of the table already set).
__global__ void batch_chunk_kernel(const EnsDev* ens, int32_t n_ens, int64_t n_chunks, int32_t* chunk_ens) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n_chunks;
       c += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = n_ens - 1;  // last one that starts at or before c
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (ens[mid].chunk_first <= c) lo = mid; else hi = mid - 1;
    }
    chunk_ens[c] = lo;
  }
}
cudaError_t launch_batch_chunks(const EnsDev* ens, int32_t n_ens, int64_t n_chunks, int32_t* chunk_ens,
                                cudaStream_t s) {
  if (n_chunks <= 0) return cudaSuccess;
  const int64_t want = (n_chunks + 255) / 256;
  batch_chunk_kernel<<<(int)(want < 152 * 8 ? want : 152 * 8), 256, 0, s>>>(ens, n_ens, n_chunks, chunk_ens);
  return cudaGetLastError();
}
int batch_tile() { return kTile; }

template <int P>
static cudaError_t launch_batch_p(const BatchArgs& a, int blocks, cudaStream_t s, int* launches) {
  batch_prefix_kernel<<<1, 1024, 0, s>>>(a.qcount_in, a.n_ens, a.finalize ? 1 : kDeferMin,
                                         const_cast<int64_t*>(a.prefix));
  int n = 2;
  if (!a.finalize) {
    const int64_t total = (int64_t)a.n_ens * a.lstride;
    const int64_t want = (total + 255) / 256;
    batch_halfstep_kernel<P><<<(int)(want < 152 * 16 ? want : 152 * 16), 256, 0, s>>>(a);
    ++n;
  }
  if (a.near.half > 1)  // c dt > dx in an ensemble
    push_batch_kernel<P, true><<<blocks, kBatchThreads, kBatchSmem, s>>>(a);
  else
    push_batch_kernel<P, false><<<blocks, kBatchThreads, kBatchSmem, s>>>(a);
  if (a.finalize) {
    const int64_t want = (a.n_total + 255) / 256;
    batch_reset_status_kernel<<<(int)(want < 152 * 8 ? want : 152 * 8), 256, 0, s>>>(a.status,
                                                                                    a.n_total);
    ++n;
  }
  if (launches) *launches += n;
  return cudaGetLastError();
}

cudaError_t launch_batch_step(const BatchArgs& a, int order, int blocks, cudaStream_t s,
                              int* launches) {
  if (a.n_total <= 0) return cudaSuccess;
  switch (order) {
    case 1: return launch_batch_p<1>(a, blocks, s, launches);
    case 2: return launch_batch_p<2>(a, blocks, s, launches);
    case 3: return launch_batch_p<3>(a, blocks, s, launches);
    case 4: return launch_batch_p<4>(a, blocks, s, launches);
    case 5: return launch_batch_p<5>(a, blocks, s, launches);
    default: return cudaErrorInvalidValue;
  }
}

template <int P, bool WIDE>
static int batch_occupancy_of() {
  int occ = 0;
  if (cudaFuncSetAttribute(push_batch_kernel<P, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kBatchSmem) == cudaSuccess)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, push_batch_kernel<P, WIDE>, kBatchThreads, kBatchSmem);
  return occ;
}
template <int P>
static int batch_occupancy() {
  const int a = batch_occupancy_of<P, false>(), b = batch_occupancy_of<P, true>();
  return a < b ? a : b;
}

// Called at pic_batch_create: also lets the kernel have its shared memory.
int batch_max_blocks_per_sm(int order) {
  int occ = 0;
  switch (order) {
    case 1: occ = batch_occupancy<1>(); break;
    case 2: occ = batch_occupancy<2>(); break;
    case 3: occ = batch_occupancy<3>(); break;
    case 4: occ = batch_occupancy<4>(); break;
    case 5: occ = batch_occupancy<5>(); break;
    default: break;
  }
  return occ > 0 ? occ : 1;
}

// Window of a level for every ensemble: Ey[e][c], Bz[e][c] -> ensemble e's
// mirrored ring, slot and slot + R; the slot's origin recorded on the device.
__global__ void batch_scatter_kernel(const EnsDev* ens, int32_t n_ens, int64_t slot, int64_t R,
                                     int64_t W, const double* Ey, const double* Bz,
                                     const int64_t* i0, int64_t* slot_i0_all) {
  const int64_t total = (int64_t)n_ens * W;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int e = (int)(q / W);
    const int64_t c = q % W;
    const int64_t pos = (i0[e] + c) & (W - 1);
    float* rE = const_cast<float*>(ens[e].ringE);
    float* rB = const_cast<float*>(ens[e].ringB);
    const float ev = (float)Ey[q], bv = (float)Bz[q];
    rE[slot * W + pos] = ev;
    rE[(slot + R) * W + pos] = ev;
    rB[slot * W + pos] = bv;
    rB[(slot + R) * W + pos] = bv;
    if (c == 0) slot_i0_all[(int64_t)e * R + slot] = i0[e];
  }
}

cudaError_t launch_batch_scatter(const EnsDev* ens, int32_t n_ens, int64_t slot, int64_t R,
                                 int64_t W, const double* Ey, const double* Bz, const int64_t* i0,
                                 int64_t* slot_i0_all, cudaStream_t s) {
  const int64_t total = (int64_t)n_ens * W;
  const int64_t want = (total + 255) / 256;
  batch_scatter_kernel<<<(int)(want < 152 * 16 ? want : 152 * 16), 256, 0, s>>>(
      ens, n_ens, slot, R, W, Ey, Bz, i0, slot_i0_all);
  return cudaGetLastError();
}

}  // namespace pic
