// Self-consistent 1D3V PIC loop around the adaptive sub-cycling integrator
// (arXiv 2102.10983): push + deposit, Yee field solve, Gauss check.
//
// Compiled with -fmad=false: every FP64 multiply and add rounds separately in
// the order written, so the loop reproduces a serial FP64 evaluation of the
// same definitions bit for bit.  The current deposit is exact fixed point
// (int64 units of 2^-44 n_c e, two's-complement atomics), so the order in
// which threads add their contributions does not change a bit either.
//
// Per macro step n (state: x at t_n, p at t_n - h_old/2):
//   push and deposit: criterion of Sec. IV (|B_z| at x_n, t_n, gamma of the
//     stored momentum; smallest k with Psi0/4^k <= Psi_max); m = 4^k sub-steps
//     of h = dt/4^k, the first with (h_old + h)/2; each sub-step gathers E_x,
//     E_y, B_z with the order-p weights of Sec. VI (tabulated per (k, j)) and
//     the tent (Eqs. eq:Enp, eq:Bnp), takes the Boris push with E = (E_x, E_y,
//     0) (Eqs. eq:p - eq:gamman) and moves x by h v_x (Eq. eq:x).  It adds
//     (h/dt) v_y S(x_mid) of every sub-step to per-node FP64 sums, and at the
//     end of the macro step one rounded fixed-point value per node to J_y, and
//     the charge flux of its move (start -> end or frozen position) to J_x.
//     As in push_f64.cu: node fields at t_n once per step (nodes_kernel; a grid
//     of more entries than electrons is gathered from instead), the
//     m = 1 electrons in order (push_deposit_kernel), the others in warps of
//     equal k (subcycle_deposit_kernel), and roots, quotients, floors and
//     conversions off the FP64 unit, which bounds the kernels (19 clocks per
//     warp instruction).  1,760,600 electrons, 20,000 cells, a0 = 150: 1.58 ms
//     per step as one kernel on that unit alone, 0.49 ms so (0.25 the m = 1
//     pass at ~48 slots per warp, 0.24 the sub-cycles).
//   field_kernel: E_y^{n+1} (Eq. eq:Ey with -dt J_y; Mur at both ends),
//     E_x^{n+1} = E_x^n - dt J_x, B_z^{n+3/2} (Eq. eq:Bz); also clears the
//     other parity's accumulators for the next step.
//   rho_kernel + gauss_kernel (on request): node charges from the positions
//     and max_k |(E_x_{k+1/2} - E_x_{k-1/2})/dx - rho_k|.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <vector>

#include "fp64_push.cuh"
#include "pic_internal.h"
#include "pic_sc1d.h"

namespace pic {
namespace {

constexpr double kUnit = 0x1p-44;  // fixed-point charge unit

struct Sc1dArgs {
  int64_t n;
  double *x, *px, *py, *pz;
  uint8_t* status;
  const int64_t* Q;
  const double* Ex[kMaxOrder + 1];  // levels n-p .. n
  const double* Ey[kMaxOrder + 1];
  const double* Bz[kMaxOrder + 1];  // levels n+1/2-p .. n+1/2
  unsigned long long* F;            // J_x face fluxes (int64 two's complement)
  unsigned long long* D;            // J_y node sums
  int64_t M;                        // entries of every grid array (n_cells + 5)
  int32_t n_cells;
  double dt, inv_dx, psi_max, qm, qm_abs;
  int k_max;
  const double* wtab;
  int64_t crit_row;
  DevStats* stats;
  float crit_scale;   // criterion_f64_scale
  double2* nodes;     // nullptr, or [M][3]: {f, f_next - f} of E_x, E_y, B_z at t_n (node_fields_pay)
  uint8_t* k_sub;     // as in PushArgsF64
  int32_t* queue;
  int32_t* bin;
  int sms;
};

__device__ __forceinline__ bool inside(double s, int32_t n_cells) {
  return s >= 0.5 && s < (double)n_cells - 0.5;
}

// Tent nodes and offsets of s on both grids; false outside the interior.
__device__ __forceinline__ bool locate(const Sc1dArgs& a, double s, Coords64& c) {
  if (coords64_fast(s, c)) return c.jb < a.n_cells - 1;  // s >= 1; s < N - 1/2
  if (!inside(s, a.n_cells)) return false;
  coords64_any(s, c);
  return true;
}

// a[idx] += v; an index outside [0, M) (only a non-finite position could
// make one) is dropped instead of written
__device__ __forceinline__ void add_i64(unsigned long long* a, int64_t idx, int64_t M, int64_t v) {
  if (idx >= 0 && idx < M) atomicAdd(a + idx, (unsigned long long)v);
}

// The warp's sum of v (two's complement, exact), as three integer reductions
// of 27 + 27 + 10 bits.
__device__ __forceinline__ unsigned long long warp_sum_i64(int64_t v) {
  const uint64_t u = (uint64_t)v;
  const uint64_t lo = __reduce_add_sync(0xffffffffu, (unsigned)u & 0x7ffffffu);
  const uint64_t mid = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 27) & 0x7ffffffu);
  const uint64_t hi = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 54));
  return lo + (mid << 27) + (hi << 54);
}

// a[idx] += v0, a[idx + 1] += v1, summed over the lanes of equal idx first:
// electrons near each other in the store share nodes (a hundred per cell in
// order of position), and atomics on one address are served one at a time
// (rho_kernel on 1,760,600 electrons: 187 us lane by lane, 27 us so).  Three
// sums; a warp spread wider than that adds the rest lane by lane.  All lanes call this; a
// lane without a deposit passes zeros.  The sums are exact, so neither their
// order nor the grouping changes a bit.
__device__ __forceinline__ void add_pair_warp(unsigned long long* a, int64_t idx, int64_t M, int64_t v0,
                                              int64_t v1) {
  const int lane = threadIdx.x & 31;
  const bool some = (v0 | v1) != 0;
  unsigned todo = __ballot_sync(0xffffffffu, some);
#pragma unroll 1
  for (int it = 0; it < 3 && todo; ++it) {
    const int leader = __ffs(todo) - 1;
    const int64_t key = __shfl_sync(0xffffffffu, idx, leader);
    const bool same = some && idx == key;
    const unsigned long long s0 = warp_sum_i64(same ? v0 : 0), s1 = warp_sum_i64(same ? v1 : 0);
    if (lane == leader) {
      if (s0) add_i64(a, key, M, (int64_t)s0);
      if (s1) add_i64(a, key + 1, M, (int64_t)s1);
    }
    todo &= ~__ballot_sync(0xffffffffu, same);
  }
  if ((todo >> lane) & 1u) {
    if (v0) add_i64(a, idx, M, v0);
    if (v1) add_i64(a, idx + 1, M, v1);
  }
}

// Node charges of Q at node i's offset w: r0 at node i, r1 at i + 1, r0 + r1 = Q.
__device__ __forceinline__ void split(int64_t Q, double w, int64_t& r0, int64_t& r1) {
  r1 = double_to_ll(ll_to_double(Q) * w);
  r0 = Q - r1;
}

// J_x of a move from (ia, wa) to (ib, wb): the charge that crosses the faces
// after nodes lo and lo + 1, lo = min(ia, ib) (c dt < dx: at most one node on).
__device__ __forceinline__ void face_flux(int64_t Q, int64_t ia, double wa, int64_t ib, double wb,
                                          int64_t& lo, int64_t& f0, int64_t& f1) {
  int64_t ra0, ra1, rb0, rb1;
  split(Q, wa, ra0, ra1);
  split(Q, wb, rb0, rb1);
  lo = ia < ib ? ia : ib;
  // running sum of the charge -r leaving ia, ia + 1 and arriving at ib, ib + 1
  f0 = ia == ib ? rb0 - ra0 : ia < ib ? -ra0 : rb0;
  f1 = ia == ib ? 0 : ia < ib ? -rb1 : ra1;
}

// Per array index: the temporal sums at theta = 1/2 and the step to the next
// index, of E_x, E_y and B_z: the fields of the criterion and of every m = 1
// push (one multiplication and one addition per grid and electron instead of
// the gather's 17 operations; the same bits).
template <int P>
__global__ void __launch_bounds__(128) nodes_kernel(Sc1dArgs a) {
  constexpr int stride = 2 * (P + 1);
  if (blockIdx.x == 0 && threadIdx.x < kBinF64) a.bin[threadIdx.x] = 0;  // the step's counts
  const double* wE = a.wtab + wrow(0, 1) * stride;
  const double* wB = a.wtab + a.crit_row * stride + (P + 1);
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < 3 * a.M;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int f = (int)(q % 3);
    const int64_t c = q / 3, c1 = c + 1 < a.M ? c + 1 : c;
    const double* const* lv = f == 0 ? a.Ex : f == 1 ? a.Ey : a.Bz;
    const double* w = f == 2 ? wB : wE;
    double f0 = w[0] * __ldg(lv[0] + c), f1 = w[0] * __ldg(lv[0] + c1);
#pragma unroll
    for (int l = 1; l <= P; ++l) {
      f0 = f0 + w[l] * __ldg(lv[l] + c);
      f1 = f1 + w[l] * __ldg(lv[l] + c1);
    }
    a.nodes[q] = make_double2(f0, f1 - f0);
  }
}

// What an electron adds to the grid sums: d0, d1 to D at node jd and the next,
// f0, f1 to F after node jf and the next.
struct Deposit {
  int64_t jd = 0, d0 = 0, d1 = 0, jf = 0, f0 = 0, f1 = 0;
};

// One grid's field at t_n about the array index q, offset w, from the levels.
template <int P>
__device__ __forceinline__ double gather_tn(const double* const* lv, const double* wt, int64_t q, double w) {
  double f0 = wt[0] * __ldg(lv[0] + q), f1 = wt[0] * __ldg(lv[0] + q + 1);
#pragma unroll
  for (int l = 1; l <= P; ++l) {
    f0 = f0 + wt[l] * __ldg(lv[l] + q);
    f1 = f1 + wt[l] * __ldg(lv[l] + q + 1);
  }
  return f0 + w * (f1 - f0);
}

// Electron i's criterion and, with k = 0, its m = 1 push and deposit: its k, or
// -1 if it is lost (or is now).
template <int P, bool UNIT>
__device__ __forceinline__ int criterion_deposit(const Sc1dArgs& a, int64_t i, unsigned long long* sh, Deposit& dep) {
  const uint8_t st = a.status[i];
  if (st & PIC_STATUS_LOST) return -1;
  const double x = a.x[i];
  Mom64 p = mom64(a.px[i], a.py[i], a.pz[i]);
  Coords64 c;
  if (!locate(a, x * a.inv_dx, c)) {
    a.status[i] = (uint8_t)(st | PIC_STATUS_LOST);
    atomicAdd(&sh[11], 1ull);
    return -1;
  }
  double ex, ey, bz;
  if (a.nodes) {
    const double2 nx = __ldg(a.nodes + 3 * (c.jb + 2)), ny = __ldg(a.nodes + 3 * (c.je + 2) + 1),
                  nb = __ldg(a.nodes + 3 * (c.jb + 2) + 2);
    ex = nx.x + c.wb * nx.y;
    ey = ny.x + c.we * ny.y;
    bz = nb.x + c.wb * nb.y;
  } else {
    const double* wE = a.wtab + wrow(0, 1) * (2 * (P + 1));
    ex = gather_tn<P>(a.Ex, wE, c.jb + 2, c.wb);
    ey = gather_tn<P>(a.Ey, wE, c.je + 2, c.we);
    bz = gather_tn<P>(a.Bz, a.wtab + a.crit_row * (2 * (P + 1)) + (P + 1), c.jb + 2, c.wb);
  }
  bool capped;
  const int k = criterion_f64(a.crit_scale, a.qm_abs, a.dt, a.psi_max, a.k_max, bz, p.x, p.y, p.z, capped);
  if (capped) atomicAdd(&sh[10], 1ull);
  if (k > 0) return k;
  const double hp = 0.5 * (pow4_down64(a.dt, st & 0x7f) + a.dt);
  const Push64 r = push64<UNIT, true>(ex, ey, bz, 0.5 * hp, a.qm, p);
  const double hv = a.dt * r.vx;
  const double xn = x + hv;
  a.x[i] = xn;
  a.px[i] = p.x;
  a.py[i] = p.y;
  a.status[i] = 0;
  const int64_t Q = a.Q[i];
  const double Qd = ll_to_double(Q);
  double w;
  floor_frac64((x + half64(hv)) * a.inv_dx, dep.jd, w);
  const double t = r.vy * w;
  dep.d0 = -double_to_ll((r.vy - t) * Qd);
  dep.d1 = -double_to_ll(t * Qd);
  int64_t ib;
  floor_frac64(xn * a.inv_dx, ib, w);
  face_flux(Q, c.je, c.we, ib, w, dep.jf, dep.f0, dep.f1);
  return 0;
}

// The three passes of push_f64.cu with E_x and the deposit: (1) here, every
// electron's criterion, the m = 1 push and its deposit; (2) bin_f64_kernel;
// (3) subcycle_deposit_kernel.
template <int P, bool UNIT>
__global__ void __launch_bounds__(256) push_deposit_kernel(Sc1dArgs a) {
  __shared__ unsigned long long sh[12];
  if (threadIdx.x < 12) sh[threadIdx.x] = 0ull;
  __syncthreads();
  unsigned k0 = 0, k1 = 0;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x; b < a.n; b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = b + threadIdx.x;
    Deposit dep;
    if (i < a.n) {
      const int k = criterion_deposit<P, UNIT>(a, i, sh, dep);
      k0 += k == 0 ? 1u : 0u;
      k1 += k == 1 ? 1u : 0u;
      if (k > 1) atomicAdd(&sh[k], 1ull);
      a.k_sub[i] = (uint8_t)(k > 0 ? k : 0);
    }
    add_pair_warp(a.D, dep.jd + 2, a.M, dep.d0, dep.d1);
    add_pair_warp(a.F, dep.jf + 2, a.M, dep.f0, dep.f1);
  }
  const unsigned k0w = __reduce_add_sync(0xffffffffu, k0), k1w = __reduce_add_sync(0xffffffffu, k1);
  if ((threadIdx.x & 31) == 0 && k0w) atomicAdd(&sh[0], (unsigned long long)k0w);
  if ((threadIdx.x & 31) == 0 && k1w) atomicAdd(&sh[1], (unsigned long long)k1w);
  flush_f64(sh, a.stats);
  if (threadIdx.x > 0 && threadIdx.x < 8 && sh[threadIdx.x])
    atomicAdd(&a.bin[threadIdx.x], (int32_t)sh[threadIdx.x]);
}

// The J_y sums of an electron's sub-steps at nodes base .. base + 4, base =
// floor(s_a) - 2 (a macro step moves an electron less than one cell): the two
// nodes it is between in registers of their own, the five spelled out, since
// an add to each of the five under a predicate costs the FP64 unit five.
struct NodeSums {
  double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  double lo = 0.0, hi = 0.0;  // acc[at], acc[at + 1] while at is current
  int at = 0;
  __device__ __forceinline__ void put() {
#pragma unroll
    for (int q = 0; q < 5; ++q) acc[q] = q == at ? lo : q == at + 1 ? hi : acc[q];
  }
  __device__ __forceinline__ void add(int64_t c, double v0, double v1) {
    if (c < 0 || c > 3) return;
    if ((int)c != at) {
      put();
      at = (int)c;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q == at) {
          lo = acc[q];
          hi = acc[q + 1];
        }
    }
    lo = lo + v0;
    hi = hi + v1;
  }
};

// The sub-cycles, g equal-k electrons per warp, each lane's i (subcycle_f64 of
// push_f64.cu, with E_x and the deposit).
template <int P, bool UNIT>
__device__ __forceinline__ void subcycle_deposit(const Sc1dArgs& a, int64_t i, bool valid, int g, int k,
                                                 unsigned long long* sh) {
  constexpr int stride = 2 * (P + 1);
  const int lane = threadIdx.x & 31, mine = lane & (g - 1), rows = 32 / g;
  const int copy = lane / g;
  const uint8_t st = valid ? a.status[i] : 0;
  double xi = valid ? a.x[i] : 0.0;
  Mom64 p = valid ? mom64(a.px[i], a.py[i], a.pz[i]) : Mom64{0.0, 0.0, 0.0, 0.0, 0.0};
  const int m = 1 << (2 * k);
  const double h = pow4_down64(a.dt, k), h_old = pow4_down64(a.dt, st & 0x7f);
  double half = 0.5 * (0.5 * (h_old + h));
  const double* w = a.wtab + wrow(k, 1) * stride;
  NodePair<P> X, Y, B;
  NodeSums J;
  bool live = valid;
  int64_t ia, ib;
  double wa, wb;
  floor_frac64(xi * a.inv_dx, ia, wa);
  int have = 0, at = 0;  // the warp holds the sums of sub-steps at .. at + have - 1
  double v[6];           // sub-step j's
  auto take = [&](int r) {  // they are with copy r
    const double mineof[6] = {X.f, X.d, Y.f, Y.d, B.f, B.d};
    const int src = mine + (r & (rows - 1)) * g;
#pragma unroll
    for (int q = 0; q < 6; ++q) v[q] = rows > 1 ? __shfl_sync(0xffffffffu, mineof[q], src) : mineof[q];
  };
#pragma unroll 1
  for (int j = 0; j < m; ++j) {
    Coords64 c;
    const bool in = live && locate(a, xi * a.inv_dx, c);
    const int32_t ny = in ? (int32_t)c.je + 2 : Y.at, nb = in ? (int32_t)c.jb + 2 : B.at;
    live = in;
    const bool moved = ny != Y.at || nb != B.at;
    if (__any_sync(0xffffffffu, moved || j >= at + have)) {
      if (!__any_sync(0xffffffffu, live)) break;
      if (moved) {
        X.load(a.Ex, nb, 0x7fffffff);
        Y.load(a.Ey, ny, 0x7fffffff);
        B.load(a.Bz, nb, 0x7fffffff);
      }
      at = j;
      have = rows;
      const double* wr = w + (int64_t)(j + copy < m ? j + copy : m - 1) * stride;
      X.sums(wr);
      Y.sums(wr);
      B.sums(wr + (P + 1));
      take(0);
    }
    const double ex = v[0] + c.wb * v[1], ey = v[2] + c.we * v[3], bz = v[4] + c.wb * v[5];
    take(j + 1 - at);  // the next sub-step's, unless an electron changes node
    if (live) {
      const Push64 r = push64<UNIT, true>(ex, ey, bz, half, a.qm, p);
      half = 0.5 * h;
      const double hv = h * r.vx;
      int64_t jm;
      double wm;
      floor_frac64((xi + half64(hv)) * a.inv_dx, jm, wm);
      xi = xi + hv;
      const double cw = scale_down64(r.vy, k);  // (h/dt) v_y
      const double t = cw * wm;
      J.add(jm - (ia - 2), cw - t, t);
    }
  }
  if (valid && copy == 0) {
    a.x[i] = xi;
    a.px[i] = p.x;
    a.py[i] = p.y;
    a.status[i] = (uint8_t)(live ? k : k | PIC_STATUS_LOST);
    if (!live) atomicAdd(&sh[11], 1ull);
    J.put();
    const int64_t Q = a.Q[i];
#pragma unroll
    for (int q = 0; q < 5; ++q)
      if (J.acc[q] != 0.0) add_i64(a.D, ia + q, a.M, -__double2ll_rn(J.acc[q] * (double)Q));
    floor_frac64(xi * a.inv_dx, ib, wb);
    int64_t lo, f0, f1;
    face_flux(Q, ia, wa, ib, wb, lo, f0, f1);
    if (f0) add_i64(a.F, lo + 2, a.M, f0);
    if (f1) add_i64(a.F, lo + 3, a.M, f1);
  }
}

template <int P, bool UNIT>
__global__ void __launch_bounds__(32) subcycle_deposit_kernel(Sc1dArgs a) {
  __shared__ unsigned long long sh[12];
  if (threadIdx.x < 12) sh[threadIdx.x] = 0ull;
  __syncwarp();
  int64_t t = blockIdx.x;
  for (;;) {
    int64_t first, end;
    int k, g;
    if (!item_f64(a.bin, a.sms, t, first, end, k, g)) break;
    const int64_t q = first + (threadIdx.x & (g - 1));
    subcycle_deposit<P, UNIT>(a, q < end ? a.queue[q] : 0, q < end, g, k, sh);
    int next = 0;
    if (threadIdx.x == 0) next = atomicAdd(&a.bin[16], 1);
    t = (int64_t)gridDim.x + __shfl_sync(0xffffffffu, next, 0);
  }
  __syncwarp();
  if (threadIdx.x == 0 && sh[11]) atomicAdd(&a.stats->lost, sh[11]);
}

// A small ensemble's step in one launch, a warp per electron (each_f64_kernel of
// push_f64.cu).  us per step by the passes and so: 100 electrons on 20,000 cells,
// m = 1, 32 and 18 (28 once, as one thread per electron); every electron k = 5, 456
// 2,569 and 2,434, 608 2,566 and 2,613, 1,216 2,780 and 4,013.
constexpr int kEachSc1d = 3;  // electrons per SM
template <int P, bool UNIT>
__global__ void __launch_bounds__(32) each_deposit_kernel(Sc1dArgs a) {
  __shared__ unsigned long long sh[12];
  if (threadIdx.x < 12) sh[threadIdx.x] = 0ull;
  __syncwarp();
  const int64_t i = blockIdx.x;
  int k = 0;
  if (threadIdx.x == 0) {
    Deposit dep;
    k = criterion_deposit<P, UNIT>(a, i, sh, dep);
    if (k >= 0) atomicAdd(&sh[k], 1ull);
    if (dep.d0) add_i64(a.D, dep.jd + 2, a.M, dep.d0);
    if (dep.d1) add_i64(a.D, dep.jd + 3, a.M, dep.d1);
    if (dep.f0) add_i64(a.F, dep.jf + 2, a.M, dep.f0);
    if (dep.f1) add_i64(a.F, dep.jf + 3, a.M, dep.f1);
  }
  k = __shfl_sync(0xffffffffu, k, 0);
  if (k > 0) subcycle_deposit<P, UNIT>(a, i, true, 1, k, sh);
  flush_f64(sh, a.stats);
}

struct FieldArgs {
  const double *Ex0, *Ey0, *Bz0;
  double *Ex1, *Ey1, *Bz1;
  unsigned long long* F;  // this step's accumulators (read)
  unsigned long long* D;
  unsigned long long* F_next;  // the next step's (cleared)
  unsigned long long* D_next;
  int64_t N;
  double dt, dx, r, kappa;
};

// E_y^{n+1} at array index q (node q - 2): interior Yee update with -dt J_y,
// Mur at the two ends, zero in the padding.
__device__ __forceinline__ double ey_next(const FieldArgs& a, int64_t q) {
  auto interior = [&](int64_t u) {
    return (a.Ey0[u] - a.r * (a.Bz0[u] - a.Bz0[u - 1])) - a.dt * ((double)(long long)a.D[u] * kUnit);
  };
  const int64_t k = q - 2;
  if (k >= 1 && k <= a.N - 1) return interior(q);
  if (k == 0) return a.Ey0[3] + a.kappa * (interior(3) - a.Ey0[2]);
  if (k == a.N) return a.Ey0[a.N + 1] + a.kappa * (interior(a.N + 1) - a.Ey0[a.N + 2]);
  return 0.0;
}

__global__ void field_kernel(FieldArgs a) {
  const int64_t M = a.N + 5;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < M;
       q += (int64_t)gridDim.x * blockDim.x) {
    a.Ex1[q] = a.Ex0[q] - ((double)(long long)a.F[q] * kUnit) * a.dx;
    const double e = ey_next(a, q);
    a.Ey1[q] = e;
    const int64_t k = q - 2;
    a.Bz1[q] = (k >= 0 && k <= a.N - 1) ? a.Bz0[q] - a.r * (ey_next(a, q + 1) - e) : 0.0;
    a.F_next[q] = 0ull;
    a.D_next[q] = 0ull;
  }
}

// C += the node charges of every electron (negate: minus them).
__global__ void __launch_bounds__(256) rho_kernel(const double* x, const int64_t* Q, int64_t n, double inv_dx,
                                                  unsigned long long* C, int64_t M, int negate) {
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x; b < n; b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = b + threadIdx.x;
    int64_t j = 0, r0 = 0, r1 = 0;
    if (i < n) {
      double w;
      floor_frac64(x[i] * inv_dx, j, w);
      split(Q[i], w, r0, r1);
    }
    add_pair_warp(C, j + 2, M, negate ? r0 : -r0, negate ? r1 : -r1);
  }
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
    v = u > v ? u : v;
  }
  return v;
}

// max over nodes k = -1 .. N+1 of |(E_x_{k+1/2} - E_x_{k-1/2})/dx - rho_k| and
// of |rho^e_k| (non-negative doubles compare like their bit patterns)
__global__ void __launch_bounds__(256) gauss_kernel(const double* Ex, const unsigned long long* C,
                                                    const unsigned long long* C_ion, int64_t N, double inv_dx,
                                                    unsigned long long* out) {
  unsigned long long mg = 0, mr = 0;
  for (int64_t k = -1 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k <= N + 1;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q = k + 2;
    const double rho = (double)((long long)C[q] + (long long)C_ion[q]) * kUnit;
    const unsigned long long g =
        (unsigned long long)__double_as_longlong(fabs((Ex[q] - Ex[q - 1]) * inv_dx - rho));
    const unsigned long long re =
        (unsigned long long)__double_as_longlong(fabs((double)(long long)C[q] * kUnit));
    mg = g > mg ? g : mg;
    mr = re > mr ? re : mr;
  }
  mg = warp_max_u64(mg);
  mr = warp_max_u64(mr);
  if ((threadIdx.x & 31) == 0) {
    if (mg) atomicMax(&out[0], mg);
    if (mr) atomicMax(&out[1], mr);
  }
}

__global__ void charge_units_kernel(const double* w, int64_t* Q, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    Q[i] = __double2ll_rn(w[i] * 0x1p44);
}

}  // namespace
}  // namespace pic

using namespace pic;

struct pic_sc1d {
  pic_sc1d_params prm;
  int64_t capacity = 0, n = 0, M = 0;
  int R = 0;  // ring slots (order + 1)
  cudaStream_t stream = nullptr;
  int sm_count = 0;
  double *x = nullptr, *px = nullptr, *py = nullptr, *pz = nullptr, *w_stage = nullptr;
  uint8_t* status = nullptr;
  int64_t* Q = nullptr;
  double* ring = nullptr;  // R slots x 3 fields x M
  std::vector<int64_t> slot_level;
  unsigned long long* acc = nullptr;  // [2 parities][F, D][M], then C, C_ion [M] each, gauss [2]
  double* wtab = nullptr;
  double2* nodes = nullptr;  // [M][3] fields at t_n
  int32_t* queue = nullptr;  // the electrons of a step that sub-cycle (push_deposit_kernel)
  uint8_t* k_sub = nullptr;  // in queue's allocation
  int64_t slice = 0;
  int32_t* bin = nullptr;
  DevStats* dstats = nullptr;
  int64_t launches = 0;
  double gauss_res = 0.0, rho_max = 0.0;
  int32_t checks = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  bool timing = false, timed = false;
  double timed_ms = 0.0;
  int64_t timed_steps = 0;
  char err[256] = {0};
};

static thread_local char g_sc_err[256];

static int sc_fail(pic_sc1d* c, int code, const char* msg, const char* detail = "") {
  char* dst = c ? c->err : g_sc_err;
  snprintf(dst, 256, "%s%s", msg, detail);
  return code;
}

#define SC_TRY(c, call)                                                           \
  do {                                                                            \
    cudaError_t e_ = (call);                                                      \
    if (e_ != cudaSuccess) return sc_fail((c), PIC_ECUDA, #call ": ", cudaGetErrorString(e_)); \
  } while (0)

// The queue's entries and counts are 32-bit numbers: electrons beyond this (or
// than there is room for, alloc_bin_f64) are pushed in further rounds of the
// passes.
constexpr int64_t kSlice = (int64_t)1 << 30;

static double* slot_field(pic_sc1d* c, int slot, int f) {
  return c->ring + ((int64_t)slot * 3 + f) * c->M;
}
static unsigned long long* accF(pic_sc1d* c, int par) { return c->acc + (int64_t)(2 * par) * c->M; }
static unsigned long long* accD(pic_sc1d* c, int par) { return c->acc + (int64_t)(2 * par + 1) * c->M; }
static unsigned long long* accC(pic_sc1d* c) { return c->acc + 4 * c->M; }
static unsigned long long* accCion(pic_sc1d* c) { return c->acc + 5 * c->M; }
static unsigned long long* accGauss(pic_sc1d* c) { return c->acc + 6 * c->M; }
static int grid_for(const pic_sc1d* c, int64_t n) {
  const int64_t want = (n + 255) / 256;
  const int64_t cap = (int64_t)(c->sm_count > 0 ? c->sm_count : 152) * 8;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

extern "C" int pic_sc1d_create(const pic_sc1d_params* prm, int64_t capacity, void* stream,
                               pic_sc1d** out) {
  if (!prm || !out) return sc_fail(nullptr, PIC_EINVAL, "pic_sc1d_create: NULL argument");
  *out = nullptr;
  if (!(prm->dt > 0) || !(prm->dx > 0) || !(prm->psi_max > 0) || !isfinite(prm->qm) || prm->qm == 0.0)
    return sc_fail(nullptr, PIC_EINVAL, "pic_sc1d_create: dt, dx, psi_max must be > 0, qm != 0");
  if (!(prm->dt < prm->dx))
    return sc_fail(nullptr, PIC_EINVAL, "pic_sc1d_create: the Yee scheme needs c dt < dx");
  if (prm->order < 1 || prm->order > kMaxOrder || prm->k_max < 0 || prm->k_max > kMaxK ||
      (prm->field_time != 0 && prm->field_time != 1) || prm->n_cells < 16 ||
      prm->n_cells > (1 << 26) || prm->gauss_every < 0 || capacity < 0)
    return sc_fail(nullptr, PIC_EINVAL, "pic_sc1d_create: parameter out of range");
  pic_sc1d* c = new pic_sc1d();
  c->prm = *prm;
  c->capacity = capacity;
  c->M = (int64_t)prm->n_cells + 5;
  c->R = prm->order + 1;
  c->stream = (cudaStream_t)stream;
  c->slot_level.assign(c->R, INT64_MIN);
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, dev);
  const int64_t cap = capacity > 0 ? capacity : 1;
  bool ok = true;
  ok &= cudaMalloc(&c->x, cap * 8) == cudaSuccess;
  ok &= cudaMalloc(&c->px, cap * 8) == cudaSuccess;
  ok &= cudaMalloc(&c->py, cap * 8) == cudaSuccess;
  ok &= cudaMalloc(&c->pz, cap * 8) == cudaSuccess;
  ok &= cudaMalloc(&c->w_stage, cap * 8) == cudaSuccess;
  ok &= cudaMalloc(&c->status, cap) == cudaSuccess;
  ok &= cudaMalloc(&c->Q, cap * 8) == cudaSuccess;
  ok &= cudaMalloc(&c->ring, (int64_t)c->R * 3 * c->M * 8) == cudaSuccess;
  ok &= cudaMalloc(&c->acc, (6 * c->M + 2) * 8) == cudaSuccess;
  const int64_t wcount = wrows_total(prm->k_max) * 2 * (prm->order + 1);
  ok &= cudaMalloc(&c->wtab, wcount * 8) == cudaSuccess;
  ok &= cudaMalloc(&c->dstats, sizeof(DevStats)) == cudaSuccess;
  ok &= cudaMalloc(&c->bin, kBinF64 * 4) == cudaSuccess;
  ok = ok && alloc_bin_f64(cap, kSlice, &c->queue, &c->k_sub, &c->slice) == cudaSuccess;
  // without node fields (a grid that no ensemble of this capacity pays for, no
  // room) the push gathers the levels
  if (ok && node_fields_pay(cap, c->M) && cudaMalloc(&c->nodes, 3 * c->M * sizeof(double2)) != cudaSuccess) {
    c->nodes = nullptr;
    cudaGetLastError();
  }
  if (!ok) {
    pic_sc1d_destroy(c);
    return sc_fail(nullptr, PIC_ENOMEM, "pic_sc1d_create: device allocation failed");
  }
  cudaError_t e = cudaMemsetAsync(c->ring, 0, (int64_t)c->R * 3 * c->M * 8, c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->acc, 0, (6 * c->M + 2) * 8, c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->dstats, 0, sizeof(DevStats), c->stream);
  if (e == cudaSuccess) e = build_wtab_f64(c->wtab, prm->order, prm->k_max, prm->field_time, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) {
    pic_sc1d_destroy(c);
    return sc_fail(nullptr, PIC_ECUDA, "pic_sc1d_create: ", cudaGetErrorString(e));
  }
  c->launches = 1;
  *out = c;
  return PIC_OK;
}

extern "C" int pic_sc1d_destroy(pic_sc1d* c) {
  if (!c) return PIC_OK;
  cudaFree(c->x); cudaFree(c->px); cudaFree(c->py); cudaFree(c->pz); cudaFree(c->w_stage);
  cudaFree(c->status); cudaFree(c->Q); cudaFree(c->ring); cudaFree(c->acc); cudaFree(c->wtab);
  cudaFree(c->dstats);
  cudaFree(c->nodes); cudaFree(c->queue); cudaFree(c->bin);
  if (c->ev0) cudaEventDestroy(c->ev0);
  if (c->ev1) cudaEventDestroy(c->ev1);
  delete c;
  return PIC_OK;
}

static cudaMemcpyKind kind_to_dev(int where) {
  return where == PIC_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
}
static cudaMemcpyKind kind_from_dev(int where) {
  return where == PIC_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
}

extern "C" int pic_sc1d_particles_write(pic_sc1d* c, const double* x, const double* px,
                                        const double* py, const double* pz, const double* w,
                                        int64_t n, int32_t where) {
  if (!c) return PIC_EINVAL;
  if (n < 0 || n > c->capacity) return sc_fail(c, PIC_EINVAL, "pic_sc1d_particles_write: n out of range");
  if (where != PIC_HOST && where != PIC_DEVICE) return sc_fail(c, PIC_EINVAL, "bad where");
  if (n > 0 && (!x || !px || !py || !pz || !w)) return sc_fail(c, PIC_EINVAL, "NULL particle array");
  const cudaMemcpyKind k = kind_to_dev(where);
  if (n > 0) {
    SC_TRY(c, cudaMemcpyAsync(c->x, x, n * 8, k, c->stream));
    SC_TRY(c, cudaMemcpyAsync(c->px, px, n * 8, k, c->stream));
    SC_TRY(c, cudaMemcpyAsync(c->py, py, n * 8, k, c->stream));
    SC_TRY(c, cudaMemcpyAsync(c->pz, pz, n * 8, k, c->stream));
    SC_TRY(c, cudaMemcpyAsync(c->w_stage, w, n * 8, k, c->stream));
  }
  SC_TRY(c, cudaMemsetAsync(c->status, 0, n > 0 ? n : 1, c->stream));
  c->n = n;
  // fixed-point charges, then the ion background: minus the electrons' charge
  SC_TRY(c, cudaMemsetAsync(accCion(c), 0, c->M * 8, c->stream));
  if (n > 0) {
    charge_units_kernel<<<grid_for(c, n), 256, 0, c->stream>>>(c->w_stage, c->Q, n);
    rho_kernel<<<grid_for(c, n), 256, 0, c->stream>>>(c->x, c->Q, n, 1.0 / c->prm.dx, accCion(c), c->M, 1);
    c->launches += 2;
  }
  SC_TRY(c, cudaGetLastError());
  if (where == PIC_HOST) SC_TRY(c, cudaStreamSynchronize(c->stream));
  return PIC_OK;
}

extern "C" int pic_sc1d_particles_read(pic_sc1d* c, double* x, double* px, double* py, double* pz,
                                       uint8_t* status, int64_t n, int32_t where) {
  if (!c) return PIC_EINVAL;
  if (n < 0 || n > c->n) return sc_fail(c, PIC_EINVAL, "pic_sc1d_particles_read: n out of range");
  if (where != PIC_HOST && where != PIC_DEVICE) return sc_fail(c, PIC_EINVAL, "bad where");
  const cudaMemcpyKind k = kind_from_dev(where);
  if (n > 0) {
    if (x) SC_TRY(c, cudaMemcpyAsync(x, c->x, n * 8, k, c->stream));
    if (px) SC_TRY(c, cudaMemcpyAsync(px, c->px, n * 8, k, c->stream));
    if (py) SC_TRY(c, cudaMemcpyAsync(py, c->py, n * 8, k, c->stream));
    if (pz) SC_TRY(c, cudaMemcpyAsync(pz, c->pz, n * 8, k, c->stream));
    if (status) SC_TRY(c, cudaMemcpyAsync(status, c->status, n, k, c->stream));
  }
  if (where == PIC_HOST) SC_TRY(c, cudaStreamSynchronize(c->stream));
  return PIC_OK;
}

static int slot_of(const pic_sc1d* c, int64_t level) {
  return (int)(((level % c->R) + c->R) % c->R);
}

extern "C" int pic_sc1d_fields_write(pic_sc1d* c, int64_t level, const double* Ex, const double* Ey,
                                     const double* Bz, int32_t where) {
  if (!c) return PIC_EINVAL;
  if (!Ex || !Ey || !Bz) return sc_fail(c, PIC_EINVAL, "pic_sc1d_fields_write: NULL field");
  if (where != PIC_HOST && where != PIC_DEVICE) return sc_fail(c, PIC_EINVAL, "bad where");
  const int s = slot_of(c, level);
  const cudaMemcpyKind k = kind_to_dev(where);
  SC_TRY(c, cudaMemcpyAsync(slot_field(c, s, 0), Ex, c->M * 8, k, c->stream));
  SC_TRY(c, cudaMemcpyAsync(slot_field(c, s, 1), Ey, c->M * 8, k, c->stream));
  SC_TRY(c, cudaMemcpyAsync(slot_field(c, s, 2), Bz, c->M * 8, k, c->stream));
  if (where == PIC_HOST) SC_TRY(c, cudaStreamSynchronize(c->stream));
  c->slot_level[s] = level;
  return PIC_OK;
}

extern "C" int pic_sc1d_fields_read(pic_sc1d* c, int64_t level, double* Ex, double* Ey, double* Bz,
                                    int32_t where) {
  if (!c) return PIC_EINVAL;
  if (where != PIC_HOST && where != PIC_DEVICE) return sc_fail(c, PIC_EINVAL, "bad where");
  const int s = slot_of(c, level);
  if (c->slot_level[s] != level) return sc_fail(c, PIC_EINVAL, "pic_sc1d_fields_read: level not stored");
  const cudaMemcpyKind k = kind_from_dev(where);
  if (Ex) SC_TRY(c, cudaMemcpyAsync(Ex, slot_field(c, s, 0), c->M * 8, k, c->stream));
  if (Ey) SC_TRY(c, cudaMemcpyAsync(Ey, slot_field(c, s, 1), c->M * 8, k, c->stream));
  if (Bz) SC_TRY(c, cudaMemcpyAsync(Bz, slot_field(c, s, 2), c->M * 8, k, c->stream));
  if (where == PIC_HOST) SC_TRY(c, cudaStreamSynchronize(c->stream));
  return PIC_OK;
}

static int sc_gauss(pic_sc1d* c) {
  SC_TRY(c, cudaMemsetAsync(accC(c), 0, c->M * 8, c->stream));
  if (c->n > 0) {
    rho_kernel<<<grid_for(c, c->n), 256, 0, c->stream>>>(c->x, c->Q, c->n, 1.0 / c->prm.dx, accC(c), c->M, 0);
    ++c->launches;
  }
  return PIC_OK;
}

template <int P>
static void launch_push(pic_sc1d* c, const Sc1dArgs& all, int64_t off = 0) {
  const cudaStream_t s = c->stream;
  Sc1dArgs a = all;
  a.x += off; a.px += off; a.py += off; a.pz += off; a.status += off; a.Q += off;
  a.n = all.n - off < c->slice ? all.n - off : c->slice;
  const bool unit = a.qm_abs == 1.0;
  if (all.n <= (int64_t)a.sms * kEachSc1d) {
    a.nodes = nullptr;
    if (unit)
      each_deposit_kernel<P, true><<<(int)a.n, 32, 0, s>>>(a);
    else
      each_deposit_kernel<P, false><<<(int)a.n, 32, 0, s>>>(a);
    ++c->launches;
    return;
  }
  const bool fill = off == 0 && a.nodes;
  if (fill)
    nodes_kernel<P><<<grid_for(c, 2 * 3 * c->M), 128, 0, s>>>(a);
  else
    cudaMemsetAsync(a.bin, 0, kBinF64 * sizeof(int32_t), s);
  // small ensembles in small blocks: every SM's FP64 unit takes part
  const int threads = a.n >= (int64_t)a.sms * 256 ? 256 : a.n >= (int64_t)a.sms * 64 ? 64 : 32;
  const int64_t want = (a.n + threads - 1) / threads, cap = (int64_t)a.sms * 8;
  const int blocks = (int)(want < cap ? want : cap);
  if (unit)
    push_deposit_kernel<P, true><<<blocks, threads, 0, s>>>(a);
  else
    push_deposit_kernel<P, false><<<blocks, threads, 0, s>>>(a);
  launch_bin_f64(BinF64{a.n, a.k_sub, a.queue, a.bin}, a.sms, s);
  const int64_t most = (int64_t)a.sms * 12;
  const int warps = (int)(a.n < most ? a.n : most);
  if (unit)
    subcycle_deposit_kernel<P, true><<<warps, 32, 0, s>>>(a);
  else
    subcycle_deposit_kernel<P, false><<<warps, 32, 0, s>>>(a);
  c->launches += fill ? 4 : 3;
  if (off + a.n < all.n) launch_push<P>(c, all, off + a.n);
}

extern "C" int pic_sc1d_step(pic_sc1d* c, int64_t n0, int64_t n_steps, pic_sc1d_stats* stats) {
  if (!c) return PIC_EINVAL;
  if (n_steps < 1) return sc_fail(c, PIC_EINVAL, "pic_sc1d_step: n_steps must be >= 1");
  const int p = c->prm.order;
  for (int l = 0; l <= p; ++l)
    if (c->slot_level[slot_of(c, n0 - p + l)] != n0 - p + l)
      return sc_fail(c, PIC_EINVAL, "pic_sc1d_step: levels n0-p .. n0 must be stored");
  if (c->timing && !c->ev0) {
    SC_TRY(c, cudaEventCreate(&c->ev0));
    SC_TRY(c, cudaEventCreate(&c->ev1));
  }
  if (c->timing) SC_TRY(c, cudaEventRecord(c->ev0, c->stream));
  const double r = c->prm.dt / c->prm.dx;
  for (int64_t j = 0; j < n_steps; ++j) {
    const int64_t s = n0 + j;
    const int par = (int)(s & 1);
    Sc1dArgs a;
    memset(&a, 0, sizeof(a));
    a.n = c->n;
    a.x = c->x; a.px = c->px; a.py = c->py; a.pz = c->pz;
    a.status = c->status;
    a.Q = c->Q;
    for (int l = 0; l <= p; ++l) {
      const int se = slot_of(c, s - p + l);
      a.Ex[l] = slot_field(c, se, 0);
      a.Ey[l] = slot_field(c, se, 1);
      a.Bz[l] = slot_field(c, se, 2);
    }
    a.F = accF(c, par);
    a.D = accD(c, par);
    a.M = c->M;
    a.n_cells = c->prm.n_cells;
    a.dt = c->prm.dt;
    a.inv_dx = 1.0 / c->prm.dx;
    a.psi_max = c->prm.psi_max;
    a.qm = c->prm.qm;
    a.qm_abs = fabs(c->prm.qm);
    a.k_max = c->prm.k_max;
    a.wtab = c->wtab;
    a.crit_row = wrows_total(c->prm.k_max) - 1;
    a.stats = c->dstats;
    if (c->n > 0) {
      a.crit_scale = criterion_f64_scale(a.qm_abs, a.dt, a.psi_max);
      a.nodes = node_fields_pay(c->n, c->M) ? c->nodes : nullptr;
      a.k_sub = c->k_sub;
      a.queue = c->queue;
      a.bin = c->bin;
      a.sms = c->sm_count > 0 ? c->sm_count : 152;
      switch (p) {
        case 1: launch_push<1>(c, a); break;
        case 2: launch_push<2>(c, a); break;
        case 3: launch_push<3>(c, a); break;
        case 4: launch_push<4>(c, a); break;
        case 5: launch_push<5>(c, a); break;
      }
    }
    FieldArgs f;
    const int s0 = slot_of(c, s), s1 = slot_of(c, s + 1);
    f.Ex0 = slot_field(c, s0, 0); f.Ey0 = slot_field(c, s0, 1); f.Bz0 = slot_field(c, s0, 2);
    f.Ex1 = slot_field(c, s1, 0); f.Ey1 = slot_field(c, s1, 1); f.Bz1 = slot_field(c, s1, 2);
    f.F = accF(c, par); f.D = accD(c, par);
    f.F_next = accF(c, par ^ 1); f.D_next = accD(c, par ^ 1);
    f.N = c->prm.n_cells;
    f.dt = c->prm.dt;
    f.dx = c->prm.dx;
    f.r = r;
    f.kappa = (r - 1.0) / (r + 1.0);
    field_kernel<<<grid_for(c, c->M), 256, 0, c->stream>>>(f);
    ++c->launches;
    SC_TRY(c, cudaGetLastError());
    c->slot_level[s1] = s + 1;
    const int ge = c->prm.gauss_every;
    if (ge > 0 && (((s + 1) % ge) + ge) % ge == 0) {  // after steps s + 1 = multiples of ge
      int rc = sc_gauss(c);
      if (rc != PIC_OK) return rc;
      gauss_kernel<<<grid_for(c, c->M), 256, 0, c->stream>>>(slot_field(c, s1, 0), accC(c), accCion(c),
                                                             c->prm.n_cells, 1.0 / c->prm.dx,
                                                             accGauss(c));
      ++c->launches;
      ++c->checks;  // the maxima accumulate on the device until stats are read
    }
  }
  if (c->timing) {
    SC_TRY(c, cudaEventRecord(c->ev1, c->stream));
    SC_TRY(c, cudaEventSynchronize(c->ev1));
    float ms = 0.f;
    SC_TRY(c, cudaEventElapsedTime(&ms, c->ev0, c->ev1));
    c->timed_ms += ms;
    c->timed_steps += n_steps;
  }
  if (!stats) return PIC_OK;
  DevStats h;
  unsigned long long g[2];
  SC_TRY(c, cudaMemcpyAsync(&h, c->dstats, sizeof(DevStats), cudaMemcpyDeviceToHost, c->stream));
  SC_TRY(c, cudaMemcpyAsync(g, accGauss(c), 16, cudaMemcpyDeviceToHost, c->stream));
  SC_TRY(c, cudaMemsetAsync(c->dstats, 0, sizeof(DevStats), c->stream));
  SC_TRY(c, cudaMemsetAsync(accGauss(c), 0, 16, c->stream));
  SC_TRY(c, cudaStreamSynchronize(c->stream));
  memcpy(&c->gauss_res, &g[0], 8);
  memcpy(&c->rho_max, &g[1], 8);
  memset(stats, 0, sizeof(*stats));
  for (int k = 0; k < 8; ++k) stats->k_hist[k] = (int64_t)h.k_hist[k];
  stats->substeps = (int64_t)h.substeps;
  stats->n_star = (int64_t)h.n_star;
  stats->clamped = (int64_t)h.clamped;
  stats->frozen = (int64_t)h.lost;
  stats->gauss_residual = c->gauss_res;
  stats->rho_max = c->rho_max;
  stats->checks = c->checks;
  c->gauss_res = 0.0;
  c->checks = 0;
  if (stats->clamped) return sc_fail(c, PIC_EKMAX, "criterion capped at k_max");
  return PIC_OK;
}

extern "C" int pic_sc1d_timing(pic_sc1d* c, double* total_ms, int64_t* steps) {
  if (!c) return PIC_EINVAL;
  c->timing = true;
  if (total_ms) *total_ms = c->timed_ms;
  if (steps) *steps = c->timed_steps;
  c->timed_ms = 0.0;
  c->timed_steps = 0;
  return PIC_OK;
}

extern "C" int64_t pic_sc1d_launch_count(const pic_sc1d* c) { return c ? c->launches : 0; }

extern "C" const char* pic_sc1d_last_error(const pic_sc1d* c) { return c ? c->err : g_sc_err; }
