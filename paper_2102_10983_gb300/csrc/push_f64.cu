// FP64 form of the adaptive sub-cycling push (arXiv 2102.10983).
//
// This translation unit is compiled with -fmad=false: every multiply and add
// below rounds separately, in exactly the order written, so that the result
// matches a serial FP64 evaluation of the same formulas bit for bit.  sqrt and
// division are the IEEE correctly rounded double operations.
//
// Per particle and macro step (Algorithm 1, Sec. IV):
//   criterion: Psi0 = |q/m| |B(x_n, t_n)| dt / (2 gamma), gamma of the stored
//              momentum, B interpolated with the order-p weights at t_n;
//              k = smallest k with Psi0/4^k <= Psi_max (capped at k_max);
//   m = 4^k sub-steps of h = dt/4^k; the first uses (h_old + h)/2 (the
//   transitional step), each: order-p Lagrange in time (Sec. VI), tent in space
//   (Eqs. eq:Enp, eq:Bnp), Boris (Eqs. eq:p - eq:gamman), x += h v_x (Eq. eq:x).
#include <math.h>

#include "fp64_push.cuh"
#include "pic_internal.h"

namespace pic {

// Weights of Eqs. eq:lagrange2-2 (B) and eq:lagrange2-3 (E):
//   L_j(theta) = prod_{k != j} (c_k + theta) / (j - k),
// c_k = p-k-1 (B) or p-k-1/2 (E); numerator over ascending k, times the
// correctly rounded reciprocal of the integer denominator.
__device__ void lagrange_f64(int p, bool is_e, double theta, double* w) {
  const double c_off = is_e ? -0.5 : -1.0;
  for (int j = 0; j <= p; ++j) {
    double num = 1.0;
    bool first = true;
    long long den = 1;
    for (int k = 0; k <= p; ++k) {
      if (k == j) continue;
      double factor = ((double)(p - k) + c_off) + theta;
      if (first) {
        num = factor;
        first = false;
      } else {
        num = num * factor;
      }
      den *= (long long)(j - k);
    }
    w[j] = num * (1.0 / (double)den);
  }
}

// One row per (k, j) sub-step plus a last row for the criterion (theta = 1/2).
__global__ void wtab_f64_kernel(double* wtab, int p, int k_max, int field_time, int64_t rows) {
  const int stride = 2 * (p + 1);
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x) {
    double theta;
    if (r == rows - 1) {
      theta = 0.5;
    } else {
      int k = 0;
      while (k < k_max && wrow(k + 1, 1) <= r) ++k;
      int64_t j = r - wrow(k, 1) + 1;
      double inv_m = ldexp(1.0, -2 * k);
      theta = (field_time == 0) ? 0.5 + (double)(j - 1) * inv_m : ((double)(j - 1) + 0.5) * inv_m;
    }
    lagrange_f64(p, true, theta, wtab + r * stride);
    lagrange_f64(p, false, theta, wtab + r * stride + (p + 1));
  }
}

cudaError_t build_wtab_f64(double* wtab, int order, int k_max, int field_time, cudaStream_t s) {
  int64_t rows = wrows_total(k_max);
  int blocks = (int)((rows + 255) / 256);
  wtab_f64_kernel<<<blocks, 256, 0, s>>>(wtab, order, k_max, field_time, rows);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- node sums at t_n

// Per window node (position i & (W-1)): the temporal sums f_i of E_y and B_z at
// theta = 1/2 and the steps f_{i+1} - f_i to the next node, as {E, dE, B, dB}.
// The criterion's B_z and an m = 1 push's fields at a particle are then one
// multiplication and one addition per grid, the bits of the full gather.
template <int P>
__device__ __forceinline__ double tsum64(const double* const* lv, const double* w, int64_t c) {
  double f = w[0] * __ldg(lv[0] + c);
#pragma unroll
  for (int l = 1; l <= P; ++l) f = f + w[l] * __ldg(lv[l] + c);
  return f;
}

template <int P>
__global__ void __launch_bounds__(128) nodes_f64_kernel(PushArgsF64 a) {
  if (blockIdx.x == 0 && threadIdx.x < kBinF64) a.bin[threadIdx.x] = 0;  // the step's counts
  const double* wE = a.wtab + wrow(0, 1) * (2 * (P + 1));
  const double* wB = a.wtab + a.crit_row * (2 * (P + 1)) + (P + 1);
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c <= a.mask;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c1 = (c + 1) & a.mask;
    const double e0 = tsum64<P>(a.E, wE, c), e1 = tsum64<P>(a.E, wE, c1);
    const double b0 = tsum64<P>(a.B, wB, c), b1 = tsum64<P>(a.B, wB, c1);
    reinterpret_cast<double2*>(a.nodes)[2 * c] = make_double2(e0, e1 - e0);
    reinterpret_cast<double2*>(a.nodes)[2 * c + 1] = make_double2(b0, b1 - b0);
  }
}

// ---------------------------------------------------------------- one sub-cycle

// Node indices and offsets of s, and whether both grids' tents lie in the
// window (lo <= s, s - 1/2 < hi; lo and hi are integers).
__device__ __forceinline__ bool locate(const PushArgsF64& a, double s, Coords64& c) {
  if (coords64_fast(s, c)) return c.jb >= a.lo_i && c.je < a.hi_i;  // jb <= je
  const double sb = s - 0.5;
  if (!(s >= a.lo && s < a.hi) || !(sb >= a.lo && sb < a.hi)) return false;
  coords64_any(s, c);
  return true;
}

// All 4^k sub-steps of one macro step of g electrons (g a power of two; lane l
// has electron i of index l mod g, if `valid`).  Each is worked on in 32 / g
// equal copies: every copy takes the electron's serial chain (about 21
// dependent FP64 operations of 64 clocks and five divisions and roots per
// sub-step), which costs the FP64 unit nothing, its time being per warp
// instruction.  What does not depend on where the electron goes while it
// keeps its nodes -- the temporal sums at its nodes, 28 operations at order 3
// -- the copies share: copy r forms those of the r-th sub-step to come, so a
// warp pays for them once in 32 / g sub-steps, or when one of its electrons
// changes node.
template <int P, bool UNIT>
__device__ __forceinline__ void subcycle_f64(const PushArgsF64& a, int64_t i, bool valid, int g, int k,
                                             unsigned long long* sh) {
  constexpr int stride = 2 * (P + 1);
  const int lane = threadIdx.x & 31, mine = lane & (g - 1), rows = 32 / g;
  const int copy = lane / g;
  const uint8_t st = valid ? a.status[i] : 0;
  double xi = valid ? a.x[i] : 0.0;
  Mom64 p = valid ? mom64(a.px[i], a.py[i], a.pz[i]) : Mom64{0.0, 0.0, 0.0, 0.0, 0.0};
  const int m = 1 << (2 * k);
  const int32_t mask = (int32_t)a.mask;
  const double h = pow4_down64(a.dt, k), h_old = pow4_down64(a.dt, st & 0x7f);
  double hp = 0.5 * (h_old + h);
  double half = 0.5 * hp;
  const double* w = a.wtab + wrow(k, 1) * stride;
  const bool diag = a.work != nullptr;
  double work = diag && valid ? a.work[i] : 0.0;
  double vy = diag ? div_rn(p.y, sqrt_rn(1.0 + (p.x2 + p.y * p.y + p.z2))) : 0.0;
  NodePair<P> E, B;
  bool live = valid;
  int have = 0, at = 0;  // the warp holds the sums of sub-steps at .. at + have - 1
  double ef = 0.0, ed = 0.0, bf = 0.0, bd = 0.0;  // sub-step j's
  auto take = [&](int r) {  // they are with copy r
    if (rows > 1) {
      const int src = mine + (r & (rows - 1)) * g;
      ef = __shfl_sync(0xffffffffu, E.f, src);
      ed = __shfl_sync(0xffffffffu, E.d, src);
      bf = __shfl_sync(0xffffffffu, B.f, src);
      bd = __shfl_sync(0xffffffffu, B.d, src);
    } else {
      ef = E.f;
      ed = E.d;
      bf = B.f;
      bd = B.d;
    }
  };
  // No branch on the chain but the vote, which the gather's first two
  // operations overlap: they are taken with the nodes as they were, and again
  // in the rare case.  An electron that is lost is written out there; its
  // lanes' later values are not used.
#pragma unroll 1
  for (int j = 0; j < m; ++j) {
    const double s = xi * a.inv_dx;
    Coords64 c;
    const bool in = coords64_fast(s, c) & live & (c.jb >= a.lo_i) & (c.je < a.hi_i);  // as locate
    double ey = ef + c.we * ed, bz = bf + c.wb * bd;
    bool moved = in & (((int32_t)(c.je & a.mask) != E.at) | ((int32_t)(c.jb & a.mask) != B.at));
    if (__any_sync(0xffffffffu, moved | (in != live) | (j >= at + have))) {
      if (in != live) {
        live = locate(a, s, c);
        moved = live && ((int32_t)(c.je & a.mask) != E.at || (int32_t)(c.jb & a.mask) != B.at);
        if (!live && copy == 0) {
          if (diag) a.work[i] = work;
          a.x[i] = xi;
          a.px[i] = p.x;
          a.py[i] = p.y;
          a.status[i] = (uint8_t)(k | PIC_STATUS_LOST);
          atomicAdd(&sh[11], 1ull);
        }
      }
      if (!__any_sync(0xffffffffu, live)) break;
      if (moved) {
        E.load(a.E, (int32_t)(c.je & a.mask), mask);
        B.load(a.B, (int32_t)(c.jb & a.mask), mask);
      }
      at = j;
      have = rows;
      const double* wr = w + (int64_t)(j + copy < m ? j + copy : m - 1) * stride;
      E.sums(wr);
      B.sums(wr + (P + 1));
      take(0);
      ey = ef + c.we * ed;
      bz = bf + c.wb * bd;
    }
    take(j + 1 - at);  // the next sub-step's, unless the electron changes node
    Mom64 q;
    Push64 r;
    const bool ok = push64_try<UNIT, false>(0.0, ey, bz, half, a.qm, p, q, r);
    double xn = xi + h * r.vx;
    if (live && !ok) {
      q = p;
      r = push64_any<UNIT, false>(0.0, ey, bz, half, a.qm, &q);
      xn = xi + h * r.vx;
    }
    p = q;
    xi = xn;
    if (diag) {  // (q hp / 2) E . (v_before + v_after) (App. B)
      const double v = div_rn(p.y, r.gam);
      work = work + ((a.qm * hp) * 0.5) * (ey * (vy + v));
      vy = v;
      hp = h;
    }
    half = 0.5 * h;
  }
  if (live && copy == 0) {
    if (diag) a.work[i] = work;
    a.x[i] = xi;
    a.px[i] = p.x;
    a.py[i] = p.y;
    a.status[i] = (uint8_t)k;
  }
}

// ---------------------------------------------------------------- the three passes of a step
//
// A warp runs as long as its largest 4^k, and the FP64 unit takes an
// instruction's 19 clocks however few lanes are active (one thread per
// particle left 4.75 of 32 active on the a0 = 150 ensemble).  So:
//  1. criterion_push_f64_kernel, one thread per particle in order: the
//     criterion; m = 1 electrons are pushed at once, the others' k is noted;
//  2. bin_f64_kernel: the noted electrons, grouped by k, largest first;
//  3. subcycle_f64_kernel: warps take up to 32 of one k at a time, longest first.
// Measured per step (order 3): 1,048,576 electrons of the a0 = 150 ensemble 6.2
// ms as one thread per particle, 1.9 ms so (pass 1 0.09 ms = 25 FP64 slots per
// warp, pass 2 6 us, the rest the longest chain: 1,024 sub-steps of 1.7 us,
// 2.6 us before); 2,432 electrons at the a0 = 100 front 4.24 -> 1.54 ms, the chain
// likewise.  Small ensembles go without the passes (each_f64_kernel).

// Electron i's criterion and, with k = 0, its m = 1 push: its k, or -1 if it is
// lost (or is now).
template <int P, bool UNIT>
__device__ __forceinline__ int criterion_push_f64(const PushArgsF64& a, int64_t i, unsigned long long* sh) {
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
  double ey, bz;
  if (a.nodes) {
    const double2 e = __ldg(reinterpret_cast<const double2*>(a.nodes) + 2 * (c.je & a.mask));
    const double2 b = __ldg(reinterpret_cast<const double2*>(a.nodes) + 2 * (c.jb & a.mask) + 1);
    ey = e.x + c.we * e.y;
    bz = b.x + c.wb * b.y;
  } else {
    const double* wE = a.wtab + wrow(0, 1) * (2 * (P + 1));
    const double* wB = a.wtab + a.crit_row * (2 * (P + 1)) + (P + 1);
    const int64_t e0 = c.je & a.mask, b0 = c.jb & a.mask;
    const double fe = tsum64<P>(a.E, wE, e0), fb = tsum64<P>(a.B, wB, b0);
    ey = fe + c.we * (tsum64<P>(a.E, wE, (e0 + 1) & a.mask) - fe);
    bz = fb + c.wb * (tsum64<P>(a.B, wB, (b0 + 1) & a.mask) - fb);
  }
  bool capped;
  const int k = criterion_f64(a.crit_scale, a.qm_abs, a.dt, a.psi_max, a.k_max, bz, p.x, p.y, p.z, capped);
  if (capped) atomicAdd(&sh[10], 1ull);
  if (k > 0) return k;
  const double hp = 0.5 * (pow4_down64(a.dt, st & 0x7f) + a.dt);
  double vy = 0.0;
  if (a.work) vy = div_rn(p.y, sqrt_rn(1.0 + (p.x2 + p.y * p.y + p.z2)));
  const Push64 r = push64<UNIT, false>(0.0, ey, bz, 0.5 * hp, a.qm, p);
  a.x[i] = x + a.dt * r.vx;
  if (a.work) a.work[i] = a.work[i] + ((a.qm * hp) * 0.5) * (ey * (vy + div_rn(p.y, r.gam)));
  a.px[i] = p.x;
  a.py[i] = p.y;
  a.status[i] = 0;
  return 0;
}

template <int P, bool UNIT>
__global__ void __launch_bounds__(256) criterion_push_f64_kernel(PushArgsF64 a) {
  __shared__ unsigned long long sh[12];
  if (threadIdx.x < 12) sh[threadIdx.x] = 0ull;
  __syncthreads();
  unsigned k0 = 0, k1 = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int k = criterion_push_f64<P, UNIT>(a, i, sh);
    k0 += k == 0 ? 1u : 0u;
    k1 += k == 1 ? 1u : 0u;
    if (k > 1) atomicAdd(&sh[k], 1ull);
    a.k_sub[i] = (uint8_t)(k > 0 ? k : 0);
  }
  const unsigned k0w = __reduce_add_sync(0xffffffffu, k0), k1w = __reduce_add_sync(0xffffffffu, k1);
  if ((threadIdx.x & 31) == 0 && k0w) atomicAdd(&sh[0], (unsigned long long)k0w);
  if ((threadIdx.x & 31) == 0 && k1w) atomicAdd(&sh[1], (unsigned long long)k1w);
  flush_f64(sh, a.stats);
  if (threadIdx.x > 0 && threadIdx.x < 8 && sh[threadIdx.x])
    atomicAdd(&a.bin[threadIdx.x], (int32_t)sh[threadIdx.x]);
}

// The whole step of a small ensemble in one launch, a warp (and a block) per
// electron: its criterion and m = 1 push by one lane, a sub-cycle by all.  The
// four launches of the three passes are most of such a step, and four warps per
// SM leave the FP64 unit idle between their chains' operations (more do not: the
// passes put several electrons into a warp).  us per step by the passes and so:
// m = 1, 1 electron 17 and 8.4 (12.5 once, as one thread per electron), 608 17 and
// 8.5; every electron k = 5, 152 1,613 and 1,555, 608 1,743 and 1,685, 1,216 1,907
// and 2,603.
constexpr int kEachF64 = 4;  // electrons per SM
template <int P, bool UNIT>
__global__ void __launch_bounds__(32) each_f64_kernel(PushArgsF64 a) {
  __shared__ unsigned long long sh[12];
  if (threadIdx.x < 12) sh[threadIdx.x] = 0ull;
  __syncwarp();
  const int64_t i = blockIdx.x;
  int k = 0;
  if (threadIdx.x == 0) {
    k = criterion_push_f64<P, UNIT>(a, i, sh);
    if (k >= 0) atomicAdd(&sh[k], 1ull);
  }
  k = __shfl_sync(0xffffffffu, k, 0);
  if (k > 0) subcycle_f64<P, UNIT>(a, i, true, 1, k, sh);
  flush_f64(sh, a.stats);
}

// Every step starts from counts of zero, so that a captured step can be replayed.
// bin[1..7]: the step's counts per k; bin[8 + k]: entries of k placed so far;
// bin[16]: the sub-cycle kernel's item cursor.  Queue order: k = 7 first.
__global__ void __launch_bounds__(256) bin_f64_kernel(BinF64 a) {
  __shared__ int cnt[8], base[8];
  const int64_t n16 = (a.n + 15) / 16;
  int64_t start[8];
  start[7] = 0;
#pragma unroll
  for (int k = 6; k >= 1; --k) start[k] = start[k + 1] + a.bin[k + 1];
  if (start[1] + a.bin[1] == 0) return;
  for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x; v0 < n16; v0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i0 = 16 * (v0 + threadIdx.x);
    uint32_t w[4] = {0, 0, 0, 0};
    if (i0 + 16 <= a.n) {
      const uint4 q = *reinterpret_cast<const uint4*>(a.k_sub + i0);
      w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
    } else {
      for (int q = 0; q < 16 && i0 + q < a.n; ++q) w[q >> 2] |= (uint32_t)a.k_sub[i0 + q] << (8 * (q & 3));
    }
    if (!__syncthreads_or((w[0] | w[1] | w[2] | w[3]) != 0)) continue;
    if (threadIdx.x < 8) cnt[threadIdx.x] = 0;
    __syncthreads();
    int off[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int k = (w[q >> 2] >> (8 * (q & 3))) & 7;
      off[q] = k ? atomicAdd(&cnt[k], 1) : 0;
    }
    __syncthreads();
    if (threadIdx.x > 0 && threadIdx.x < 8 && cnt[threadIdx.x])
      base[threadIdx.x] = atomicAdd(&a.bin[8 + threadIdx.x], cnt[threadIdx.x]);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int k = (w[q >> 2] >> (8 * (q & 3))) & 7;
      if (k) {
        int64_t s = 0;
#pragma unroll
        for (int r = 1; r < 8; ++r)
          if (r == k) s = start[r];
        a.queue[s + base[k] + off[q]] = (int32_t)(i0 + q);
      }
    }
    __syncthreads();
  }
}

cudaError_t launch_bin_f64(const BinF64& a, int sms, cudaStream_t s) {
  const int64_t vecs = (a.n + 4095) / 4096;
  bin_f64_kernel<<<(int)(vecs < sms * 8 ? vecs : sms * 8), 256, 0, s>>>(a);
  return cudaGetLastError();
}

// One warp per block: the few long chains of a step spread over the SMs.
template <int P, bool UNIT>
__global__ void __launch_bounds__(32) subcycle_f64_kernel(PushArgsF64 a) {
  __shared__ unsigned long long sh[12];
  if (threadIdx.x < 12) sh[threadIdx.x] = 0ull;
  __syncwarp();
  int64_t t = blockIdx.x;
  for (;;) {
    int64_t first, end;
    int k, g;
    if (!item_f64(a.bin, a.sms, t, first, end, k, g)) break;
    const int64_t q = first + (threadIdx.x & (g - 1));
    subcycle_f64<P, UNIT>(a, q < end ? a.queue[q] : 0, q < end, g, k, sh);
    int next = 0;
    if (threadIdx.x == 0) next = atomicAdd(&a.bin[16], 1);
    t = (int64_t)gridDim.x + __shfl_sync(0xffffffffu, next, 0);
  }
  __syncwarp();
  if (threadIdx.x == 0 && sh[11]) atomicAdd(&a.stats->lost, sh[11]);
}

template <int P, bool UNIT>
static void launch_f64_p(PushArgsF64 a, int sms, cudaStream_t s, int* launches) {
  a.sms = sms;
  if (a.n <= (int64_t)sms * kEachF64) {
    a.nodes = nullptr;
    each_f64_kernel<P, UNIT><<<(int)a.n, 32, 0, s>>>(a);
    if (launches) ++*launches;
    return;
  }
  const int64_t all = a.n;
  for (int64_t off = 0; off < all; off += a.slice) {
    a.n = all - off < a.slice ? all - off : a.slice;
    if (off == 0 && a.nodes) {
      const int64_t want = (a.mask + 128) / 128;
      nodes_f64_kernel<P><<<(int)(want < sms * 8 ? want : sms * 8), 128, 0, s>>>(a);
      if (launches) ++*launches;
    } else {
      cudaMemsetAsync(a.bin, 0, kBinF64 * sizeof(int32_t), s);
    }
    // small ensembles in small blocks: every SM's FP64 unit takes part
    const int threads = a.n >= (int64_t)sms * 256 ? 256 : a.n >= (int64_t)sms * 64 ? 64 : 32;
    const int64_t want = (a.n + threads - 1) / threads, cap = (int64_t)sms * 8;
    criterion_push_f64_kernel<P, UNIT><<<(int)(want < cap ? want : cap), threads, 0, s>>>(a);
    launch_bin_f64(BinF64{a.n, a.k_sub, a.queue, a.bin}, sms, s);
    const int64_t most = (int64_t)sms * 12;
    subcycle_f64_kernel<P, UNIT><<<(int)(a.n < most ? a.n : most), 32, 0, s>>>(a);
    if (launches) *launches += 3;
    a.x += a.n; a.px += a.n; a.py += a.n; a.pz += a.n; a.status += a.n;
    if (a.work) a.work += a.n;
  }
}

cudaError_t launch_push_f64(const PushArgsF64& a, int order, cudaStream_t s, int* launches) {
  if (a.n <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool unit = a.qm_abs == 1.0;
  switch (order) {
    case 1: unit ? launch_f64_p<1, true>(a, sms, s, launches) : launch_f64_p<1, false>(a, sms, s, launches); break;
    case 2: unit ? launch_f64_p<2, true>(a, sms, s, launches) : launch_f64_p<2, false>(a, sms, s, launches); break;
    case 3: unit ? launch_f64_p<3, true>(a, sms, s, launches) : launch_f64_p<3, false>(a, sms, s, launches); break;
    case 4: unit ? launch_f64_p<4, true>(a, sms, s, launches) : launch_f64_p<4, false>(a, sms, s, launches); break;
    case 5: unit ? launch_f64_p<5, true>(a, sms, s, launches) : launch_f64_p<5, false>(a, sms, s, launches); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace pic
