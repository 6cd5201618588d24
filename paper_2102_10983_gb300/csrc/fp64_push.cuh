// Per-electron FP64 pieces shared by the FP64 kernels (push_f64.cu,
// pic_sc1d.cu, study.cu): every result has the bits of the plain FP64
// expression it replaces, but the FP64 unit (one per SM, 19 clocks per warp
// instruction) only sees the multiplications and additions of the method.
// Division and square root run on the integer pipes (fp64_int.cuh); so do the
// floors, offsets, window tests and powers of two below, each of which would
// take one to three of the unit's slots.
#pragma once

#include <math.h>

#include "fp64_int.cuh"
#include "pic_internal.h"

namespace pic {

// dt / 4^k: the exponent field lowered by 2k (ldexp's bits) while it stays
// normal.
__device__ __forceinline__ double pow4_down64(double dt, int k) {
  const long long u = __double_as_longlong(dt);
  if (((u >> 52) & 0x7ff) > 2 * k) return __longlong_as_double(u - ((long long)k << 53));
  return ldexp(dt, -2 * k);
}

// G / 2^52 for 0 <= G < 2^52, exact.
__device__ __forceinline__ double fix52(uint64_t G) {
  const int lz = __clzll((long long)G);
  const uint64_t bits = (G << (lz - 11)) + ((uint64_t)(uint32_t)(1033 - lz) << 52);
  return G ? __longlong_as_double((long long)bits) : 0.0;
}

// A position in node units on both grids (E nodes at i, B nodes at i + 1/2):
// the tent's lower nodes and the offsets from them.
struct Coords64 {
  int64_t je, jb;
  double we, wb;
};

// floor(s), s - floor(s) and the same of s - 1/2.  For 1 <= s < 2^21 all four
// are exact and read off the significand: the fraction as a 52-bit fixed-point
// number, half a node being its top bit.  False outside that range (the caller
// takes coords64_any).
__device__ __forceinline__ bool coords64_fast(double s, Coords64& c) {
  const uint64_t u = (uint64_t)__double_as_longlong(s);
  const uint32_t h = (uint32_t)(u >> 32);
  const int sh = (int)(h >> 20) - 1023;
  const uint64_t G = (u << (sh & 31)) & 0xfffffffffffffull;
  const int32_t j = (int32_t)(((h & 0xfffffu) | 0x100000u) >> ((20 - sh) & 31));
  c.je = j;
  c.we = fix52(G);
  c.jb = j - ((G >> 51) ? 0 : 1);
  c.wb = fix52(G ^ 0x8000000000000ull);
  return h - 0x3ff00000u < 0x01500000u;
}
__device__ __forceinline__ void coords64_any(double s, Coords64& c) {
  const double fe = floor(s), sb = s - 0.5, fb = floor(sb);
  c.je = (int64_t)fe;
  c.we = s - fe;
  c.jb = (int64_t)fb;
  c.wb = sb - fb;
}

// floor(s) and s - floor(s) on one grid, the same way.
__device__ __forceinline__ void floor_frac64(double s, int64_t& j, double& w) {
  const uint64_t u = (uint64_t)__double_as_longlong(s);
  const uint32_t h = (uint32_t)(u >> 32);
  const int sh = (int)(h >> 20) - 1023;
  j = (int32_t)(((h & 0xfffffu) | 0x100000u) >> ((20 - sh) & 31));
  w = fix52((u << (sh & 31)) & 0xfffffffffffffull);
  if (h - 0x3ff00000u >= 0x01500000u) {
    const double fl = floor(s);
    j = (int64_t)fl;
    w = s - fl;
  }
}

// v 4^-k (ldexp's bits, which a multiplication by that power has too).
__device__ __forceinline__ double scale_down64(double v, int k) {
  return v == 0.0 ? v : pow4_down64(v, k);
}
__device__ __forceinline__ double half64(double v) {
  const long long u = __double_as_longlong(v);
  return ((u >> 52) & 0x7ff) > 1 ? __longlong_as_double(u - (1ll << 52)) : 0.5 * v;
}

// (double)q and __double2ll_rn(v) on the integer pipes.
__device__ __forceinline__ double ll_to_double(int64_t q) {
  if ((uint64_t)q >> 52) return (double)q;
  const int lz = __clzll(q);
  const uint64_t bits = ((uint64_t)q << (lz - 11)) + ((uint64_t)(uint32_t)(1085 - lz) << 52);
  return q ? __longlong_as_double((long long)bits) : 0.0;
}
__device__ __forceinline__ int64_t double_to_ll(double v) {
  const uint64_t u = (uint64_t)__double_as_longlong(v);
  const int sh = 1075 - (int)((u >> 52) & 0x7ff);  // |v| = M 2^-sh
  if (sh < 1) return __double2ll_rn(v);
  const uint64_t M = fp64i_sig(u);
  const int r = sh & 63;
  // nearest, ties to even: half a unit less one, plus the quotient's last bit
  const uint64_t q = sh > 53 ? 0ull : (M + (1ull << (r - 1)) - 1 + ((M >> r) & 1)) >> r;
  return (int64_t)u < 0 ? -(int64_t)q : (int64_t)q;
}

// The criterion of Sec. IV decided in FP32 where that is safe.  c = |q/m| dt /
// (2 Psi_max) (a normal FP32 number in [2^-60, 2^60], Psi_max not tiny; else
// the host passes 0 and every electron takes the exact test): r = c |B| /
// gamma carries a relative error below 2^-20, so away from the powers of four
// by 2^-18 the comparisons of r are those of Psi / Psi_max.  Returns -1 where
// it cannot tell (near a threshold, or anything not finite).
__device__ __forceinline__ int criterion_f64_guess(float c, double b0, double px, double py, double pz,
                                                   int k_max, bool& capped) {
  const float b = fabsf((float)b0), x = (float)px, y = (float)py, z = (float)pz;
  const float g2 = fmaf(x, x, fmaf(y, y, fmaf(z, z, 1.0f)));
  float r = c * b * fp64i_rsqrt(g2);
  if (!(g2 < 0x1p100f && r < 0x1p60f && c > 0.f)) return -1;
  int k = 0;
  while (r > 0x1.00004p0f && k < k_max) {
    r *= 0.25f;
    ++k;
  }
  capped = r > 1.0f;
  // r <= 1 + 2^-18 here, or k = k_max; the last threshold not passed was 1,
  // and a passed one left r > (1 + 2^-18) / 4
  return fabsf(r - 1.0f) <= 0x1p-18f ? -1 : k;
}

// The exact test: Psi as the oracle forms it, k the smallest with
// Psi / 4^k <= Psi_max.
__device__ __forceinline__ int criterion_f64_exact(double qm_abs, double dt, double psi_max, int k_max,
                                                   double b0, double px, double py, double pz,
                                                   bool& capped) {
  const double g0 = sqrt_rn(1.0 + (px * px + py * py + pz * pz));
  double psi = div_rn(qm_abs * fabs(b0) * dt, 2.0 * g0);
  int k = 0;
  while (psi > psi_max && k < k_max) {
    psi = psi * 0.25;
    ++k;
  }
  capped = psi > psi_max;
  return k;
}

__device__ __forceinline__ int criterion_f64(float c, double qm_abs, double dt, double psi_max,
                                             int k_max, double b0, double px, double py, double pz,
                                             bool& capped) {
  int k = criterion_f64_guess(c, b0, px, py, pz, k_max, capped);
  if (k < 0) k = criterion_f64_exact(qm_abs, dt, psi_max, k_max, b0, px, py, pz, capped);
  return k;
}

// One grid's levels at the current node pair, and their temporal sums for the
// next sub-step.
template <int P>
struct NodePair {
  double v0[P + 1], v1[P + 1];
  int32_t at = -1;  // masked index of the lower node
  double f, d;      // f_i, f_{i+1} - f_i
  __device__ __forceinline__ void load(const double* const* lv, int32_t node, int32_t mask) {
    const int32_t next = (node + 1) & mask;
#pragma unroll
    for (int l = 0; l <= P; ++l) {
      v0[l] = __ldg(lv[l] + node);
      v1[l] = __ldg(lv[l] + next);
    }
    at = node;
  }
  __device__ __forceinline__ void sums(const double* w) {
    double f0 = w[0] * v0[0], f1 = w[0] * v1[0];
#pragma unroll
    for (int l = 1; l <= P; ++l) {
      f0 = f0 + w[l] * v0[l];
      f1 = f1 + w[l] * v1[l];
    }
    f = f0;
    d = f1 - f0;
  }
};

// Electrons per warp for a k with `count` of them: few enough that every SM
// gets a warp of them before any warp holds a second electron (a sub-cycle is
// a latency-bound chain, so fewer electrons per warp cost nothing while units
// are idle and save the temporal sums), at most 32.
__device__ __forceinline__ int group_f64(int count, int sms) {
  int g = 1;
  while (g < 32 && count > g * sms) g *= 2;
  return g;
}

// Work item t of the binned electrons (bin[1..7]: their counts, k = 7 first in
// the queue): entries first .. of the queue (those from `end` on absent), g of
// them, all of one k.  False past the last item.
__device__ __forceinline__ bool item_f64(const int32_t* bin, int sms, int64_t t, int64_t& first,
                                         int64_t& end, int& k, int& g) {
  int64_t items = 0, entries = 0;
  first = -1;
#pragma unroll
  for (int q = 7; q >= 1; --q) {
    const int c = bin[q];
    const int gq = group_f64(c, sms);
    const int64_t n = (c + gq - 1) / gq;
    if (first < 0 && t < items + n) {
      k = q;
      g = gq;
      first = entries + (t - items) * gq;
      end = entries + c;
    }
    items += n;
    entries += c;
  }
  return first >= 0;
}

// Block counters -> context counters: sh[0..7] the k histogram, sh[10] caps,
// sh[11] lost.  Sub-step sums follow from the histogram (m = 4^k).
__device__ __forceinline__ void flush_f64(unsigned long long* sh, DevStats* st) {
  __syncthreads();
  if (threadIdx.x < 12) {
    unsigned long long v = sh[threadIdx.x];
    if (threadIdx.x == 8 || threadIdx.x == 9) {
      v = 0;
      for (int k = threadIdx.x == 8 ? 0 : 1; k < 8; ++k) v += sh[k] << (2 * k);
    }
    if (v) {
      unsigned long long* dst = threadIdx.x < 8 ? &st->k_hist[threadIdx.x]
                                : threadIdx.x == 8 ? &st->substeps
                                : threadIdx.x == 9 ? &st->n_star
                                : threadIdx.x == 10 ? &st->clamped
                                                    : &st->lost;
      atomicAdd(dst, v);
    }
  }
}

// q/m times v: a sign for the electron (UNIT: |q/m| = 1).
template <bool UNIT>
__device__ __forceinline__ double times_qm(double qm, double v) {
  if constexpr (UNIT)
    return __longlong_as_double(__double_as_longlong(v) ^
                                (__double_as_longlong(qm) & (long long)0x8000000000000000ull));
  else
    return qm * v;
}

// Momentum, with p_x^2 (which the next push of the sub-cycle needs again) and
// p_z^2 (which no push changes: B is along z, E in the plane).
struct Mom64 {
  double x, y, z, x2, z2;
};
__device__ __forceinline__ Mom64 mom64(double x, double y, double z) {
  return Mom64{x, y, z, x * x, z * z};
}

// Boris push in E = (ex, ey, 0), B = (0, 0, bz) (Eqs. eq:p - eq:gamman) with
// half = hp / 2, and the velocity after it.  EX: with E_x (and v_y wanted).
struct Push64 {
  double vx, vy, gam;
};
template <bool UNIT, bool EX>
static __device__ __noinline__ Push64 push64_any(double ex, double ey, double bz, double half, double qm,
                                                 Mom64* p) {
  const double dpx = EX ? times_qm<UNIT>(qm, ex) * half : 0.0;
  const double dpy = times_qm<UNIT>(qm, ey) * half;
  const double mx = EX ? p->x + dpx : p->x, my = p->y + dpy;
  const double gn = sqrt(1.0 + (mx * mx + my * my + p->z2));
  const double tz = (times_qm<UNIT>(qm, bz) * half) / gn;
  const double ppx = mx + my * tz;
  const double ppy = my - mx * tz;
  const double sz = (2.0 * tz) / (1.0 + tz * tz);
  p->x = EX ? (mx + ppy * sz) + dpx : mx + ppy * sz;
  p->y = (my - ppx * sz) + dpy;
  p->x2 = p->x * p->x;
  Push64 r;
  r.gam = sqrt(1.0 + (p->x2 + p->y * p->y + p->z2));
  r.vx = p->x / r.gam;
  r.vy = EX ? p->y / r.gam : 0.0;
  return r;
}
// The same bits with the integer roots and quotients, in one straight line (no
// branch between the FP64 operations, so their latencies overlap what is
// independent); q: the momentum after it.  False: operands outside those
// routines' domain, the push is to be taken again by push64_any.  A serial
// chain forms its next position before it looks at that.
template <bool UNIT, bool EX>
__device__ __forceinline__ bool push64_try(double ex, double ey, double bz, double half, double qm,
                                           const Mom64& p, Mom64& q, Push64& r) {
  const double dpx = EX ? times_qm<UNIT>(qm, ex) * half : 0.0;
  const double dpy = times_qm<UNIT>(qm, ey) * half;
  const double mx = EX ? p.x + dpx : p.x, mx2 = EX ? mx * mx : p.x2;
  const double my = p.y + dpy;
  const double num = times_qm<UNIT>(qm, bz) * half;
  double tz, sz, none;
  bool ok = div_sqrt_try<false>(num, 0.0, 1.0 + (mx2 + my * my + p.z2), tz, none, none);
  const double ppx = mx + my * tz;
  const double ppy = my - mx * tz;
  ok &= div2_try(tz, 1.0 + tz * tz, sz);
  q.x = EX ? (mx + ppy * sz) + dpx : mx + ppy * sz;
  q.y = (my - ppx * sz) + dpy;
  q.z = p.z;
  q.z2 = p.z2;
  q.x2 = q.x * q.x;
  r.vy = 0.0;
  ok &= div_sqrt_try<EX>(q.x, q.y, 1.0 + (q.x2 + q.y * q.y + q.z2), r.vx, r.vy, r.gam);
  return ok;
}
template <bool UNIT, bool EX>
__device__ __forceinline__ Push64 push64(double ex, double ey, double bz, double half, double qm, Mom64& p) {
  Mom64 q;
  Push64 r;
  if (!push64_try<UNIT, EX>(ex, ey, bz, half, qm, p, q, r))
    return push64_any<UNIT, EX>(ex, ey, bz, half, qm, &p);
  p = q;
  return r;
}

}  // namespace pic
