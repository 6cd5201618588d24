// Per-particle device arithmetic of the mixed-precision push, shared by the
// single-problem kernels (push_mixed.cu), the batched kernel (push_batch.cu)
// and the fused predictor kernel (mlp_bf16.cu).
#pragma once

#include <limits.h>
#include <math.h>

#include "pic_internal.h"

namespace pic {

// ---------------------------------------------------------------- per-particle math

// The p+1 levels of one grid used by one macro step (level 0 = oldest).
// Ring form: consecutive slots of the mirrored ring, level l at base + l*W.
// Pointer form: one pointer per level (levels owned by the caller).
template <int P, bool RING>
struct Levels;
template <int P>
struct Levels<P, true> {
  const float* base;
  int32_t lstride;  // l * lstride + node stays below 2^31 (window <= 2^28 nodes)
  __device__ __forceinline__ const float* at(int l) const { return base + (uint32_t)(l * lstride); }
};
template <int P>
struct Levels<P, false> {
  const float* ptr[P + 1];
  __device__ __forceinline__ const float* at(int l) const { return ptr[l]; }
};

// Temporal sums at the two tent nodes jn, jn+1, then the tent weight wt.
template <int P, class LV>
__device__ __forceinline__ float gather_f32(const LV& lv, const float* w, int32_t jn, float wt,
                                            int32_t mask) {
  const int32_t a0 = jn & mask, a1 = (jn + 1) & mask;
  float f0 = __fmul_rn(w[0], __ldg(lv.at(0) + a0));
  float f1 = __fmul_rn(w[0], __ldg(lv.at(0) + a1));
#pragma unroll
  for (int l = 1; l <= P; ++l) {
    f0 = __fmaf_rn(w[l], __ldg(lv.at(l) + a0), f0);
    f1 = __fmaf_rn(w[l], __ldg(lv.at(l) + a1), f1);
  }
  return __fmaf_rn(wt, __fsub_rn(f1, f0), f0);
}

struct MixedState {
  int32_t cell;
  float frac, ux, uy, uz;
};

// Tent coordinates of offset f from node `cell`: E grid nodes at i dx, B grid
// nodes at (i + 1/2) dx.  False if a node is outside [lo, hi].
__device__ __forceinline__ bool tent_coords(int32_t cell, float f, int32_t lo, int32_t hi,
                                            int32_t& je, float& we, int32_t& jb, float& wb) {
  const float fe = floorf(f);
  const float fbm = __fsub_rn(f, 0.5f);
  const float fb = floorf(fbm);
  je = cell + (int32_t)fe;
  we = __fsub_rn(f, fe);
  jb = cell + (int32_t)fb;
  wb = __fsub_rn(fbm, fb);
  return jb >= lo && je < hi;  // jb <= je: both nodes of both grids in [lo, hi)
}

__device__ __forceinline__ float norm2(float a, float b, float c) {
  return __fmaf_rn(c, c, __fmaf_rn(b, b, __fmul_rn(a, a)));
}

// Criterion (Sec. IV) in FP32: Psi0 = |q/m| |B| dt / (2 gamma); smallest k with
// Psi0 / 4^k <= Psi_max, capped at k_max.  Taken in squared form, with no
// square root and no division: Psi0 <= Psi_max 4^k  <=>
// (|q/m| dt B)^2 <= (2 Psi_max)^2 (1 + |p|^2) 16^k, and the right side is
// scaled by 16 (exactly) per step of k.
// The two sides of the k = 0 test: a2 = (|q/m| dt B)^2, rhs = (2 Psi_max)^2 (1 + |p|^2).
__device__ __forceinline__ void psi_terms(float b0, const MixedState& s, float qm_abs, float dt,
                                          float psi_max, float& a2, float& rhs) {
  const float a = __fmul_rn(__fmul_rn(qm_abs, dt), b0);
  a2 = __fmul_rn(a, a);
  const float tp = __fmul_rn(2.0f, psi_max);
  rhs = __fmul_rn(__fmul_rn(tp, tp), __fadd_rn(1.0f, norm2(s.ux, s.uy, s.uz)));
}

__device__ __forceinline__ int psi_to_k(float b0, const MixedState& s, float qm_abs, float dt,
                                        float psi_max, int k_max, bool& capped) {
  float a2, rhs;
  psi_terms(b0, s, qm_abs, dt, psi_max, a2, rhs);
  int k = 0;
  while (a2 > rhs && k < k_max) {
    rhs = __fmul_rn(rhs, 16.0f);
    ++k;
  }
  capped = a2 > rhs;
  return k;
}

// dt / 4^k for a normal dt whose quotient stays normal (checked by the host):
// the exponent field lowered by 2k, the same bits as ldexpf(dt, -2k).
__device__ __forceinline__ float pow4_down(float dt, int k) {
  return __int_as_float(__float_as_int(dt) - (k << 24));
}

// b0 is B_z at the particle and t_n: with m = 1 it is also the first (and only)
// sub-step's B_z, since both use the theta = 1/2 weights at the same nodes.
template <int P, class LV>
__device__ __forceinline__ int criterion_f32(const LV& B, const float* wcrit, int32_t jb,
                                             float wb, int32_t mask, const MixedState& s,
                                             float qm_abs, float dt, float psi_max, int k_max,
                                             bool& capped, float& b0) {
  b0 = gather_f32<P>(B, wcrit, jb, wb, mask);
  return psi_to_k(b0, s, qm_abs, dt, psi_max, k_max, capped);
}

// Field view of one macro step.  coef (optional): per window node, the
// monomial coefficients (to_monomial) of the temporal interpolant of E_y (P+1)
// then of B_z (P+1), written once per step by the half-step kernel, so a node
// change costs two contiguous loads per grid instead of 2(P+1) scattered ones.
template <int P, bool RING>
struct StepFields {
  Levels<P, RING> E, B;
  const float* coef;
  int32_t lo, hi;
};

// Single-instruction reciprocal and reciprocal square root (the SFU's
// approximations, ~2 ulp, subnormals flushed): every schedule of the mixed form
// calls these same two, so they agree bit for bit.  Their arguments here are
// 1 + |p|^2 >= 1 and 1 + t^2 >= 1.
__device__ __forceinline__ float rsqrt_sfu(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_sfu(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One Boris sub-step (Eqs. eq:p - eq:gamman) and the position update (Eq. eq:x)
// in the fields ey, bz, with momentum step hp and offset step hx (cells per
// unit velocity).  The operations are ordered for the serial chain of a long
// sub-cycle: the terms of 1 + |p|^2 known early are summed first, so the
// component that arrives last costs a single FMA before each square root.
__device__ __forceinline__ void boris_f32(float ey, float bz, float hp, float hx, float qm,
                                          MixedState& s) {
  const float qmh = __fmul_rn(qm, __fmul_rn(0.5f, hp));  // q/m hp/2
  const float dpy = __fmul_rn(qmh, ey);
  const float mx = s.ux, mz = s.uz;
  const float g2xz = __fadd_rn(1.0f, __fmaf_rn(mz, mz, __fmul_rn(mx, mx)));
  const float my = __fadd_rn(s.uy, dpy);
  const float inv_gn = rsqrt_sfu(__fmaf_rn(my, my, g2xz));
  const float tz = __fmul_rn(__fmul_rn(qmh, bz), inv_gn);
  const float ppx = __fmaf_rn(my, tz, mx);
  const float ppy = __fmaf_rn(-mx, tz, my);
  const float sz = __fmul_rn(__fmul_rn(2.0f, tz), rcp_sfu(__fmaf_rn(tz, tz, 1.0f)));
  const float ux = __fmaf_rn(ppy, sz, mx);
  const float uy = __fadd_rn(__fmaf_rn(-ppx, sz, my), dpy);
  s.ux = ux;
  s.uy = uy;
  s.uz = mz;
  const float g2n = __fadd_rn(1.0f, __fmaf_rn(mz, mz, __fmul_rn(ux, ux)));
  const float inv_g = rsqrt_sfu(__fmaf_rn(uy, uy, g2n));
  s.frac = __fmaf_rn(hx, __fmul_rn(ux, inv_g), s.frac);
}

// ---------------------------------------------------------------- two particles per lane
//
// The same arithmetic on two particles at once with GB300's paired FP32
// instructions (mul/add/fma.rn.f32x2, written as PTX): each half rounds
// exactly as the scalar operation it replaces.  a - b is fma(b, -1, a).  A
// paired product that only paired sums consume can still be merged into them
// by the compiler, so such a product is kept scalar (see boris_f32x2).
__device__ __forceinline__ float2 bc2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
      " mul.rn.f32x2 rd, ra, rb;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
      " add.rn.f32x2 rd, ra, rb;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n .reg .b64 ra, rb, rc, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
      " mov.b64 rc, {%6, %7};\n fma.rn.f32x2 rd, ra, rb, rc;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, bc2(-1.0f), a); }
__device__ __forceinline__ float2 floor2(float2 a) { return make_float2(floorf(a.x), floorf(a.y)); }

struct MixedState2 {
  int2 cell;
  float2 frac, ux, uy, uz;
};

// boris_f32 on two particles (same operation order, same bits).
__device__ __forceinline__ void boris_f32x2(float2 ey, float2 bz, float2 hp, float hx, float qm,
                                            MixedState2& s) {
  const float2 qmh = mul2(bc2(qm), mul2(bc2(0.5f), hp));
  const float2 dpy = make_float2(__fmul_rn(qmh.x, ey.x), __fmul_rn(qmh.y, ey.y));
  const float2 mx = s.ux, mz = s.uz;
  const float2 g2xz = add2(bc2(1.0f), fma2(mz, mz, mul2(mx, mx)));
  const float2 my = add2(s.uy, dpy);
  const float2 gn = fma2(my, my, g2xz);
  const float2 inv_gn = make_float2(rsqrt_sfu(gn.x), rsqrt_sfu(gn.y));
  const float2 tz = mul2(mul2(qmh, bz), inv_gn);
  const float2 ppx = fma2(my, tz, mx);
  const float2 ppy = fma2(make_float2(-mx.x, -mx.y), tz, my);
  const float2 tt = fma2(tz, tz, bc2(1.0f));
  const float2 sz = mul2(mul2(bc2(2.0f), tz), make_float2(rcp_sfu(tt.x), rcp_sfu(tt.y)));
  const float2 ux = fma2(ppy, sz, mx);
  const float2 uy = add2(fma2(make_float2(-ppx.x, -ppx.y), sz, my), dpy);
  s.ux = ux;
  s.uy = uy;
  s.uz = mz;
  const float2 g2n = add2(bc2(1.0f), fma2(mz, mz, mul2(ux, ux)));
  const float2 g = fma2(uy, uy, g2n);
  const float2 inv_g = make_float2(rsqrt_sfu(g.x), rsqrt_sfu(g.y));
  s.frac = fma2(bc2(hx), mul2(ux, inv_g), s.frac);
}

// ---------------------------------------------------------------- m = 1 pushes from the step's node fields

// Every node's E_y and B_z at t_n and the steps to the next node, {E, dE, B,
// dB}: the FMA chains gather_f32 takes at the two nodes over the same levels
// and their difference, so an m = 1 push (and the criterion) that reads them
// and applies the tent weight gets exactly the bits of the full gather, from
// one 8-byte load per grid instead of 2(p+1) scattered ones.
template <int P, class LV>
__device__ __forceinline__ float4 step_node_f32(const LV& E, const LV& B, const float* wE, const float* wB,
                                                int32_t c, int32_t mask) {
  const int32_t c1 = (c + 1) & mask;
  float e0 = __fmul_rn(wE[0], __ldg(E.at(0) + c)), e1 = __fmul_rn(wE[0], __ldg(E.at(0) + c1));
  float b0 = __fmul_rn(wB[0], __ldg(B.at(0) + c)), b1 = __fmul_rn(wB[0], __ldg(B.at(0) + c1));
#pragma unroll
  for (int l = 1; l <= P; ++l) {
    e0 = __fmaf_rn(wE[l], __ldg(E.at(l) + c), e0);
    e1 = __fmaf_rn(wE[l], __ldg(E.at(l) + c1), e1);
    b0 = __fmaf_rn(wB[l], __ldg(B.at(l) + c), b0);
    b1 = __fmaf_rn(wB[l], __ldg(B.at(l) + c1), b1);
  }
  return make_float4(e0, __fsub_rn(e1, e0), b0, __fsub_rn(b1, b0));
}
__device__ __forceinline__ float2 node_e(const float4* nodes, int32_t j) {
  return __ldg(reinterpret_cast<const float2*>(nodes + j));
}
__device__ __forceinline__ float2 node_b(const float4* nodes, int32_t j) {
  return __ldg(reinterpret_cast<const float2*>(nodes + j) + 1);
}
__device__ __forceinline__ float node_lerp_e(const float4* nodes, int32_t j, float w) {
  const float2 v = node_e(nodes, j);
  return __fmaf_rn(w, v.y, v.x);
}
__device__ __forceinline__ float node_lerp_b(const float4* nodes, int32_t j, float w) {
  const float2 v = node_b(nodes, j);
  return __fmaf_rn(w, v.y, v.x);
}

// tent_coords of two particles.
struct PairNodes {
  int2 je, jb;
  float2 we, wb;
  bool in0, in1;
};
__device__ __forceinline__ PairNodes pair_nodes(const MixedState2& s, int32_t lo, int32_t hi) {
  PairNodes n;
  const float2 fe = floor2(s.frac);
  const float2 fbm = add2(s.frac, bc2(-0.5f));
  const float2 fb = floor2(fbm);
  n.we = sub2(s.frac, fe);
  n.wb = sub2(fbm, fb);
  n.je = make_int2(s.cell.x + (int32_t)fe.x, s.cell.y + (int32_t)fe.y);
  n.jb = make_int2(s.cell.x + (int32_t)fb.x, s.cell.y + (int32_t)fb.y);
  n.in0 = n.jb.x >= lo && n.je.x < hi;
  n.in1 = n.jb.y >= lo && n.je.y < hi;
  return n;
}
__device__ __forceinline__ void pair_fields(const float4* nodes, int32_t mask, const PairNodes& n, float2& ey,
                                            float2& bz) {
  const float2 e0 = node_e(nodes, n.je.x & mask), e1 = node_e(nodes, n.je.y & mask);
  const float2 b0 = node_b(nodes, n.jb.x & mask), b1 = node_b(nodes, n.jb.y & mask);
  ey = fma2(n.we, make_float2(e0.y, e1.y), make_float2(e0.x, e1.x));
  bz = fma2(n.wb, make_float2(b0.y, b1.y), make_float2(b0.x, b1.x));
}
// psi_terms of each; qm_dt = |q/m| dt, tp2 = (2 Psi_max)^2.
__device__ __forceinline__ void pair_psi(float2 bz, const MixedState2& s, float qm_dt, float tp2, float2& a2,
                                         float2& rhs) {
  const float2 av = mul2(bc2(qm_dt), bz);
  a2 = mul2(av, av);
  rhs = mul2(bc2(tp2), add2(bc2(1.0f), fma2(s.uz, s.uz, fma2(s.uy, s.uy, mul2(s.ux, s.ux)))));
}
// psi_to_k of particles with k >= 1, uncapped, as far as 3 (= 3 or more).
__device__ __forceinline__ int2 pair_short_k(float2 a2, float2 rhs) {
  const float2 r16 = mul2(rhs, bc2(16.0f)), r256 = mul2(r16, bc2(16.0f));
  return make_int2(1 + (a2.x > r16.x ? 1 : 0) + (a2.x > r256.x ? 1 : 0),
                   1 + (a2.y > r16.y ? 1 : 0) + (a2.y > r256.y ? 1 : 0));
}
// The m = 1 push of two particles, k_prev in bits 0-2 of their status.
__device__ __forceinline__ MixedState2 pair_push(const MixedState2& s, float2 ey, float2 bz, uint8_t st0,
                                                 uint8_t st1, float dt, float hx0, float qm) {
  const float2 h_old = make_float2(pow4_down(dt, st0 & 7), pow4_down(dt, st1 & 7));
  const float2 hp = mul2(bc2(0.5f), add2(h_old, bc2(dt)));
  MixedState2 u = s;
  boris_f32x2(ey, bz, hp, hx0, qm, u);
  const float2 fl = floor2(u.frac);  // normalize each
  u.cell.x += (int32_t)fl.x;
  u.cell.y += (int32_t)fl.y;
  u.frac = sub2(u.frac, fl);
  return u;
}

// Reciprocal of prod_{k != j} (j - k), the denominator of L_{p,j} (Sec. VI).
__host__ __device__ constexpr float lagrange_inv_den(int p, int j) {
  float d = 1.f;
  for (int k = 0; k <= p; ++k)
    if (k != j) d *= (float)(j - k);
  return 1.f / d;
}

// Weights of Eqs. eq:lagrange2-3 (E) and eq:lagrange2-2 (B) at theta, in FP32:
// prod_{k != j} (c_k + theta) times the reciprocal denominator, c_k = p-k-1/2
// (E) or p-k-1 (B).  Depends on the sub-step index only, so these FP32 ops run
// alongside the serial chain of the push instead of on it.
template <int P>
__device__ __forceinline__ void lagrange_f32(float theta, float* w) {
#pragma unroll
  for (int j = 0; j <= P; ++j) {
    float ne = 1.f, nb = 1.f;
#pragma unroll
    for (int k = 0; k <= P; ++k) {
      if (k == j) continue;
      ne = __fmul_rn(ne, __fadd_rn((float)(P - k) - 0.5f, theta));
      nb = __fmul_rn(nb, __fadd_rn((float)(P - k) - 1.0f, theta));
    }
    w[j] = __fmul_rn(ne, lagrange_inv_den(P, j));
    w[P + 1 + j] = __fmul_rn(nb, lagrange_inv_den(P, j));
  }
}

// Temporal sum over the levels' values v at one node, then nothing else: the
// same operation order as gather_f32.
template <int P>
__device__ __forceinline__ float tsum(const float* w, const float* v) {
  float f = __fmul_rn(w[0], v[0]);
#pragma unroll
  for (int l = 1; l <= P; ++l) f = __fmaf_rn(w[l], v[l], f);
  return f;
}

// The m = 4^k sub-steps of one macro step (Algorithm 1).  False if the particle
// left the window (state kept as reached).
//
// Coefficients of the interpolating polynomial in u at two nodes a0, a1 of the
// given levels: c_q = sum_l v_l M[l][q].
template <int P, class LV>
__device__ __forceinline__ void to_monomial(const LV& lv, int32_t a0, int32_t a1,
                                            const float (&M)[kMaxOrder + 1][kMaxOrder + 1],
                                            float* c0, float* c1) {
  float v0[P + 1], v1[P + 1];
#pragma unroll
  for (int l = 0; l <= P; ++l) {
    v0[l] = __ldg(lv.at(l) + a0);
    v1[l] = __ldg(lv.at(l) + a1);
  }
#pragma unroll
  for (int q = 0; q <= P; ++q) {
    float x0 = __fmul_rn(v0[0], M[0][q]), x1 = __fmul_rn(v1[0], M[0][q]);
#pragma unroll
    for (int l = 1; l <= P; ++l) {
      x0 = __fmaf_rn(v0[l], M[l][q], x0);
      x1 = __fmaf_rn(v1[l], M[l][q], x1);
    }
    c0[q] = x0;
    c1[q] = x1;
  }
}

// Coefficients of nodes a0, a1 of one grid (g = 0: E, 1: B) from the step's
// table; the same values to_monomial computes from the levels.
template <int P>
__device__ __forceinline__ void table_coefs(const float* coef, int g, int32_t a0, int32_t a1,
                                            float* c0, float* c1) {
  constexpr int S = 2 * (P + 1);
  const float* r0 = coef + (int64_t)a0 * S + g * (P + 1);
  const float* r1 = coef + (int64_t)a1 * S + g * (P + 1);
  if constexpr (P == 3) {  // rows of 8 floats: each half is one aligned 16-byte load
    const float4 v0 = __ldg(reinterpret_cast<const float4*>(r0));
    const float4 v1 = __ldg(reinterpret_cast<const float4*>(r1));
    c0[0] = v0.x; c0[1] = v0.y; c0[2] = v0.z; c0[3] = v0.w;
    c1[0] = v1.x; c1[1] = v1.y; c1[2] = v1.z; c1[3] = v1.w;
  } else {
#pragma unroll
    for (int q = 0; q <= P; ++q) {
      c0[q] = __ldg(r0 + q);
      c1[q] = __ldg(r1 + q);
    }
  }
}

// One node of table_coefs / to_monomial (the same values).
template <int P>
__device__ __forceinline__ void table_coef(const float* coef, int g, int32_t a0, float* c0) {
  const float* r0 = coef + (int64_t)a0 * (2 * (P + 1)) + g * (P + 1);
  if constexpr (P == 3) {
    const float4 v0 = __ldg(reinterpret_cast<const float4*>(r0));
    c0[0] = v0.x; c0[1] = v0.y; c0[2] = v0.z; c0[3] = v0.w;
  } else {
#pragma unroll
    for (int q = 0; q <= P; ++q) c0[q] = __ldg(r0 + q);
  }
}
template <int P, class LV>
__device__ __forceinline__ void to_monomial1(const LV& lv, int32_t a0,
                                             const float (&M)[kMaxOrder + 1][kMaxOrder + 1], float* c0) {
  float v0[P + 1];
#pragma unroll
  for (int l = 0; l <= P; ++l) v0[l] = __ldg(lv.at(l) + a0);
#pragma unroll
  for (int q = 0; q <= P; ++q) {
    float x0 = __fmul_rn(v0[0], M[0][q]);
#pragma unroll
    for (int l = 1; l <= P; ++l) x0 = __fmaf_rn(v0[l], M[l][q], x0);
    c0[q] = x0;
  }
}

template <int P>
__device__ __forceinline__ float horner(const float* c, float u) {
  float f = c[P];
#pragma unroll
  for (int q = P - 1; q >= 0; --q) f = __fmaf_rn(f, u, c[q]);
  return f;
}

// The m = 1 push: tabulated weights, the criterion's B_z (b0: same weights,
// same nodes).
template <int P, bool RING>
__device__ __forceinline__ bool push_once_f32(const StepFields<P, RING>& F, const float* wtab, int32_t mask,
                                              float dt, float inv_dx, float qm, int k_prev, float b0,
                                              MixedState& s) {
  const float* wr = wtab + wrow(0, 1) * (2 * (P + 1));
  int32_t je, jb;
  float we, wb;
  if (!tent_coords(s.cell, s.frac, F.lo, F.hi, je, we, jb, wb)) return false;
  const float ey = gather_f32<P>(F.E, wr, je, we, mask);
  const float hp = __fmul_rn(0.5f, __fadd_rn(pow4_down(dt, k_prev), dt));
  boris_f32(ey, b0, hp, __fmul_rn(dt, inv_dx), qm, s);
  return true;
}

// One Boris sub-step as boris_f32 takes it (same operations, same bits) with
// what the sub-steps of a cycle share carried along: qmh = q/m hp/2 and g2 = 1 +
// p_x^2 + p_z^2 (the last sub-step's g2n is the next one's g2xz).
__device__ __forceinline__ void boris_chain_f32(float ey, float bz, float qmh, float hx, MixedState& s,
                                                float& g2) {
  const float dpy = __fmul_rn(qmh, ey);
  const float mx = s.ux, mz = s.uz;
  const float my = __fadd_rn(s.uy, dpy);
  const float inv_gn = rsqrt_sfu(__fmaf_rn(my, my, g2));
  const float tz = __fmul_rn(__fmul_rn(qmh, bz), inv_gn);
  const float ppx = __fmaf_rn(my, tz, mx);
  const float ppy = __fmaf_rn(-mx, tz, my);
  const float sz = __fmul_rn(__fmul_rn(2.0f, tz), rcp_sfu(__fmaf_rn(tz, tz, 1.0f)));
  s.ux = __fmaf_rn(ppy, sz, mx);
  s.uy = __fadd_rn(__fmaf_rn(-ppx, sz, my), dpy);
  g2 = __fadd_rn(1.0f, __fmaf_rn(mz, mz, __fmul_rn(s.ux, s.ux)));
  const float inv_g = rsqrt_sfu(__fmaf_rn(s.uy, s.uy, g2));
  s.frac = __fmaf_rn(hx, __fmul_rn(s.ux, inv_g), s.frac);
}

// Three consecutive nodes' coefficients on one grid (g = 0: E, 1: B), lowest
// node a: from the step's node table (TABLE) or formed from the levels.
template <int P, bool RING, bool TABLE>
__device__ __forceinline__ void three_nodes(const StepFields<P, RING>& F, int g, int32_t a, int32_t mask,
                                            const float (&mono)[2][kMaxOrder + 1][kMaxOrder + 1],
                                            float (&c)[3][P + 1]) {
  if constexpr (TABLE) {
    table_coefs<P>(F.coef, g, a & mask, (a + 1) & mask, c[0], c[1]);
    table_coef<P>(F.coef, g, (a + 2) & mask, c[2]);
  } else {
    const Levels<P, RING>& lv = g ? F.B : F.E;
    to_monomial<P>(lv, a & mask, (a + 1) & mask, mono[g], c[0], c[1]);
    to_monomial1<P>(lv, (a + 2) & mask, mono[g], c[2]);
  }
}
// Both rounded weights in [+0, 1): then the offsets' differences from their
// nodes are exact and those nodes are the floors (a NaN or a negative weight
// fails the unsigned test).
__device__ __forceinline__ bool in_cell(float we, float wb) {
  return __float_as_uint(we) < 0x3f800000u && __float_as_uint(wb) < 0x3f800000u;
}

// What the sub-steps of a cycle carry: the state, qmh = q/m hp/2, g2 = 1 + p_x^2
// + p_z^2 and the sub-step's u = theta - 1.
struct CycleState {
  MixedState s;
  float qmh, g2, u;
};

// n sub-steps, the electron's nodes looked at in each: any way it moves.  False
// if it left the window.
template <int P, bool RING, bool TABLE>
__device__ __forceinline__ bool cycle_any(const StepFields<P, RING>& F, int32_t mask,
                                          const float (&mono)[2][kMaxOrder + 1][kMaxOrder + 1], int n,
                                          float hx, float qmh_next, float inv_m, CycleState& c) {
  float ce[3][P + 1], cb[3][P + 1];  // monomial coefficients per node
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int q = 0; q <= P; ++q) ce[a][q] = cb[a][q] = 0.f;
  // floors of the offset on the two grids at the lowest kept nodes (NaN: none
  // yet), and the offset from which E's upper pair would leave the window
  float fe = __int_as_float(0x7fc00000), fb = fe, fe_end = fe;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const float f = c.s.frac;
    const float fbm = __fsub_rn(f, 0.5f);
    // floors: the kept node's or the next one's (whole numbers: exact)
    const float fe1 = __fadd_rn(fe, 1.0f), fb1 = __fadd_rn(fb, 1.0f);
    bool up_e = f >= fe1, up_b = fbm >= fb1;
    float we = __fsub_rn(f, up_e ? fe1 : fe), wb = __fsub_rn(fbm, up_b ? fb1 : fb);
    if (!(in_cell(we, wb) && f < fe_end)) {
      int32_t je, jb;
      if (!tent_coords(c.s.cell, f, F.lo, F.hi, je, we, jb, wb)) return false;
      fe = floorf(f);
      fb = floorf(fbm);
      up_e = up_b = false;
      // (past 2^22 cells a floor plus one may not be exact)
      fe_end = je + 1 < F.hi && fabsf(f) < 0x1p22f ? __int_as_float(0x7f800000) : __fadd_rn(fe, 1.0f);
      three_nodes<P, RING, TABLE>(F, 0, je, mask, mono, ce);
      three_nodes<P, RING, TABLE>(F, 1, jb, mask, mono, cb);
    }
    const float e0 = horner<P>(ce[0], c.u), e1 = horner<P>(ce[1], c.u), e2 = horner<P>(ce[2], c.u);
    const float b1 = horner<P>(cb[0], c.u), b2 = horner<P>(cb[1], c.u), b3 = horner<P>(cb[2], c.u);
    const float el = up_e ? e1 : e0, eh = up_e ? e2 : e1;
    const float bl = up_b ? b2 : b1, bh = up_b ? b3 : b2;
    boris_chain_f32(__fmaf_rn(we, __fsub_rn(eh, el), el), __fmaf_rn(wb, __fsub_rn(bh, bl), bl), c.qmh, hx,
                    c.s, c.g2);
    c.qmh = qmh_next;
    c.u = __fadd_rn(c.u, inv_m);
  }
  return true;
}

// n sub-steps without a branch among them, for an electron that stays within
// two cells: the kept nodes are base .. base + 2 with base the floor of its
// offset less `back` on each grid.  False (c to be ignored) if a weight left
// its range, or near the window's ends.
template <int P, bool RING, bool TABLE>
__device__ __forceinline__ bool cycle_near(const StepFields<P, RING>& F, int32_t mask,
                                           const float (&mono)[2][kMaxOrder + 1][kMaxOrder + 1], int n, float back,
                                           float hx, float qmh_next, float inv_m, CycleState& c) {
  const float f0 = c.s.frac;
  const float fe = floorf(__fsub_rn(f0, back)), fb = floorf(__fsub_rn(__fsub_rn(f0, 0.5f), back));
  const float fe1 = __fadd_rn(fe, 1.0f), fb1 = __fadd_rn(fb, 1.0f);
  if (!(fabsf(f0) < 0x1p22f)) return false;
  const int32_t je = c.s.cell + (int32_t)fe, jb = c.s.cell + (int32_t)fb;
  if (jb < F.lo || je + 1 >= F.hi) return false;  // (jb <= je)
  float ce[3][P + 1], cb[3][P + 1];
  three_nodes<P, RING, TABLE>(F, 0, je, mask, mono, ce);
  three_nodes<P, RING, TABLE>(F, 1, jb, mask, mono, cb);
  float e0, e1, de0, de1, b0, b1, db0, db1;  // lower and upper pair: value, step to the next node
  auto values = [&](float u) {
    e0 = horner<P>(ce[0], u);
    e1 = horner<P>(ce[1], u);
    de0 = __fsub_rn(e1, e0);
    de1 = __fsub_rn(horner<P>(ce[2], u), e1);
    b0 = horner<P>(cb[0], u);
    b1 = horner<P>(cb[1], u);
    db0 = __fsub_rn(b1, b0);
    db1 = __fsub_rn(horner<P>(cb[2], u), b1);
  };
  values(c.u);
  bool held = true;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const float f = c.s.frac;
    const float fbm = __fsub_rn(f, 0.5f);
    const bool up_e = f >= fe1, up_b = fbm >= fb1;
    const float we = __fsub_rn(f, up_e ? fe1 : fe), wb = __fsub_rn(fbm, up_b ? fb1 : fb);
    const float ey = __fmaf_rn(we, up_e ? de1 : de0, up_e ? e1 : e0);
    const float bz = __fmaf_rn(wb, up_b ? db1 : db0, up_b ? b1 : b0);
    held = held && in_cell(we, wb);
    c.u = __fadd_rn(c.u, inv_m);
    values(c.u);
    boris_chain_f32(ey, bz, c.qmh, hx, c.s, c.g2);
    c.qmh = qmh_next;
  }
  return held;
}

// Sub-steps j0+1 .. j1 of the m = 4^k of one macro step (j1 = -1: all of them;
// k >= 1 unless a whole m = 1 step): a sub-cycle can stop after any sub-step
// and resume from the state it left (offset not yet normalised) with the same
// bits as an uninterrupted one.
//
// The temporal interpolant at each tent node is a polynomial of degree p in u =
// theta - 1, evaluated by Horner's rule (p FMAs per node).  Each grid keeps
// three nodes' coefficients: an electron moves less than a cell per macro step
// (c dt < dx), so the nodes it needs change at most once within a sub-cycle,
// and then it takes the other pair of the three: a select instead of a load.
// (With two nodes kept, every lane's crossing made its warp wait about 600
// clocks for L2 at a sub-step of its own.)
//
// A long sub-cycle is a serial chain, and the longest one of a call bounds it
// whatever else the GPU does (1,024 sub-steps at k = 5).  Its dependent
// operations take 120 clocks per sub-step; a branch that looks at the nodes in
// each, and the nodes' values formed after it, made that 200.  So k >= kNearMin
// runs without a branch (cycle_near), the next sub-step's values formed in the
// shadow of this one's push: 153.  k >= kHalfMin goes in stretches of at most
// half a cell (half a macro step where c dt <= dx), from the middle of the kept
// nodes, which an electron cannot leave either way; k = 2 in one stretch, the
// nodes ahead of the electron kept (its 16 sub-steps would not pay for a second
// load).  What does not fit (a turn back, the window's ends) takes cycle_any, as
// does k = 1, whose four sub-steps gain nothing.  near: the rule for the grid
// (stretches), fixed at compile time where c dt <= dx: as a value of its own it
// cost the kernels 1 to 5 % (16.8M electrons over steps 2405 to 4404, binned, push
// kernel 0.254 and 0.263 ms).  Per step, two nodes ->
// three -> with stretches: 300 electrons at the front 119 -> 117 -> 95 us,
// 16.8M electrons 249 -> 219 -> 199 us, 1,000,003 at fifth order 120 -> 118 ->
// 90 us.
template <bool WIDE, int K_MIN = kNearMin>
struct NearRule {
  static constexpr int k_min = K_MIN, half = 1;
  __device__ __forceinline__ explicit NearRule(const Stretches&) {}
};
template <int K_MIN>
struct NearRule<true, K_MIN> {
  int k_min, half;
  __device__ __forceinline__ explicit NearRule(const Stretches& s) : k_min(s.k_min), half(s.half) {}
};
template <int P, bool RING, bool TABLE = false, class NEAR>
__device__ __forceinline__ bool subcycle_f32(const StepFields<P, RING>& F, const float* wtab,
                                             int32_t mask, float dt, float inv_dx, float qm,
                                             int field_time, const NEAR& near,
                                             const float (&mono)[2][kMaxOrder + 1][kMaxOrder + 1],
                                             int k, int k_prev, float b0, MixedState& s,
                                             int j0 = 0, int j1 = -1) {
  if (k == 0) return push_once_f32<P, RING>(F, wtab, mask, dt, inv_dx, qm, k_prev, b0, s);
  const float h = pow4_down(dt, k);
  const float hx = __fmul_rn(h, inv_dx);
  const float qmh_next = __fmul_rn(qm, __fmul_rn(0.5f, h));
  const int m = 1 << (2 * k);
  const float inv_m = pow4_down(1.0f, k);
  const int j_end = j1 < 0 ? m : j1;
  // u_j = theta_j - 1 = u_1 + (j-1)/m: every partial sum is a multiple of 1/m
  // in [-1, 1], exact in FP32 (m <= 4^7), so the running sum has the bits of
  // the direct formula
  const float u1 = field_time == 0 ? -0.5f : __fsub_rn(__fmul_rn(0.5f, inv_m), 1.0f);
  const float hp = j0 == 0 ? __fmul_rn(0.5f, __fadd_rn(pow4_down(dt, k_prev), h)) : h;
  CycleState c{s, __fmul_rn(qm, __fmul_rn(0.5f, hp)),
               __fadd_rn(1.0f, __fmaf_rn(s.uz, s.uz, __fmul_rn(s.ux, s.ux))), __fmaf_rn((float)j0, inv_m, u1)};
  bool ok = true;
#pragma unroll 1
  for (int j = j0; j < j_end && ok;) {
    int n = j_end - j;
    bool done = false;
    if (k >= near.k_min) {
      float back = c.s.ux < 0.f ? 1.0f : 0.0f;
      if (k >= kHalfMin) {
        n = min(n, m >> near.half);
        back = 0.5f;
      }
      const CycleState before = c;
      done = cycle_near<P, RING, TABLE>(F, mask, mono, n, back, hx, qmh_next, inv_m, c);
      if (!done) c = before;
    }
    if (!done) ok = cycle_any<P, RING, TABLE>(F, mask, mono, n, hx, qmh_next, inv_m, c);
    j += n;
  }
  s = c.s;
  return ok;
}

// The node-table form of subcycle_f32 behind one call site.  With
// PIC_SUBCYCLE_NOINLINE defined, every caller in a kernel shares one copy of
// its code (a call per sub-cycle instead of a copy per caller: less for the
// instruction cache to hold); otherwise it is inlined at each caller.
struct SubOut {
  MixedState s;
  bool ok;
};
template <int P, class NEAR>
__device__ __noinline__ SubOut subcycle_table_call(StepFields<P, true> F, const float* wtab,
                                                   int32_t mask, float dt, float inv_dx, float qm,
                                                   int field_time, NEAR near, int k, int k_prev, float b0,
                                                   MixedState s, int j0, int j1) {
  float no_mono[2][kMaxOrder + 1][kMaxOrder + 1];  // the table form never reads it
  SubOut o;
  o.s = s;
  o.ok = subcycle_f32<P, true, true>(F, wtab, mask, dt, inv_dx, qm, field_time, near, no_mono, k, k_prev,
                                     b0, o.s, j0, j1);
  return o;
}
template <int P, bool RING, bool TABLE, class NEAR>
__device__ __forceinline__ bool subcycle_site(const StepFields<P, RING>& F, const float* wtab,
                                              int32_t mask, float dt, float inv_dx, float qm,
                                              int field_time, const NEAR& near,
                                              const float (&mono)[2][kMaxOrder + 1][kMaxOrder + 1],
                                              int k, int k_prev, float b0, MixedState& s,
                                              int j0 = 0, int j1 = -1) {
#ifdef PIC_SUBCYCLE_NOINLINE
  if constexpr (RING && TABLE) {
    const SubOut o = subcycle_table_call<P>(F, wtab, mask, dt, inv_dx, qm, field_time, near, k, k_prev, b0,
                                            s, j0, j1);
    s = o.s;
    return o.ok;
  }
#endif
  return subcycle_f32<P, RING, TABLE>(F, wtab, mask, dt, inv_dx, qm, field_time, near, mono, k, k_prev,
                                      b0, s, j0, j1);
}

__device__ __forceinline__ void normalize(MixedState& s) {
  const float fl = floorf(s.frac);
  s.cell += (int32_t)fl;
  s.frac = __fsub_rn(s.frac, fl);
}

// ---------------------------------------------------------------- counters

// Per-thread counters in registers: steps with k = 0, 1, 2 (the common ones)
// and caps.  Steps with k >= 3 are rare and go straight into the block's
// shared counters.  (Shared-memory atomics on one address for every
// sub-cycled particle serialised the warps at a front.)  The sub-step sums are
// not counted per particle: every counted step takes m = 4^k sub-steps, so
// they follow from the k histogram when the block flushes.
struct ThreadCounters {
  unsigned k0 = 0, k1 = 0, k2 = 0, capped = 0;
};

__device__ __forceinline__ void count_step(ThreadCounters& tc, unsigned long long* sh, int k,
                                           bool capped) {
  if (k == 0)
    ++tc.k0;
  else if (k == 1)
    ++tc.k1;
  else if (k == 2)
    ++tc.k2;
  else
    atomicAdd(&sh[k], 1ull);
  tc.capped += capped ? 1u : 0u;
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// All threads of the block must call this.  Block counters: sh[0..7] the k
// histogram, sh[10] caps, sh[11] particles lost; sh[8], sh[9] unused.
__device__ __forceinline__ void flush_counters(const ThreadCounters& tc, unsigned long long* sh,
                                               DevStats* st) {
  const unsigned long long k0 = warp_sum(tc.k0), k1 = warp_sum(tc.k1), k2 = warp_sum(tc.k2);
  const unsigned long long cap = warp_sum(tc.capped);
  if ((threadIdx.x & 31) == 0) {
    if (k0) atomicAdd(&sh[0], k0);
    if (k1) atomicAdd(&sh[1], k1);
    if (k2) atomicAdd(&sh[2], k2);
    if (cap) atomicAdd(&sh[10], cap);
  }
  __syncthreads();
  if (threadIdx.x < 12) {
    unsigned long long v = 0;
    if (threadIdx.x == 8 || threadIdx.x == 9) {  // sum of m = 4^k over the counted steps
#pragma unroll
      for (int k = threadIdx.x == 8 ? 0 : 1; k < 8; ++k) v += sh[k] << (2 * k);
    } else {
      v = sh[threadIdx.x];
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

template <class ARGS>
__device__ __forceinline__ MixedState load_state(const ARGS& a, int64_t i) {
  MixedState s;
  s.cell = a.cell[i];
  s.frac = a.frac[i];
  s.ux = a.px[i];
  s.uy = a.py[i];
  s.uz = a.pz[i];
  return s;
}

template <class ARGS>
__device__ __forceinline__ void store_state(const ARGS& a, int64_t i, const MixedState& s) {
  a.cell[i] = s.cell;
  a.frac[i] = s.frac;
  a.px[i] = s.ux;
  a.py[i] = s.uy;
  a.pz[i] = s.uz;
}

// The stream's loads and stores: each state word is touched once per step and
// the whole state is larger than L2, so these are marked evict-first to leave
// L2 to the field levels, half-step fields and queues.
// (Particle indices are below 2^31: 32-bit offsets address every array.)
__device__ __forceinline__ void fetch_stream(const PushArgsMixed& a, uint32_t i, uint8_t& st,
                                             MixedState& s) {
  st = PIC_STATUS_LOST;
  s = {0, 0.5f, 0.f, 0.f, 0.f};
  if ((int64_t)i < a.n) {
    st = __ldcs(a.status + i);
    s.cell = __ldcs(a.cell + i);
    s.frac = __ldcs(a.frac + i);
    s.ux = __ldcs(a.px + i);
    s.uy = __ldcs(a.py + i);
    s.uz = __ldcs(a.pz + i);
  }
}

template <class ARGS>
__device__ __forceinline__ void store_stream(const ARGS& a, uint32_t i, const MixedState& s) {
  __stcs(a.cell + i, s.cell);
  __stcs(a.frac + i, s.frac);
  __stcs(a.px + i, s.ux);
  __stcs(a.py + i, s.uy);
  __stcs(a.pz + i, s.uz);
}

// ---------------------------------------------------------------- bulk-copy staging of particle tiles

// A tile of kTile consecutive particles' state as the stream reads it from
// shared memory; filled by six bulk copies (cp.async.bulk, the TMA engine's
// linear mode) that complete on one mbarrier.  Every member starts on a
// 128-byte boundary and the size is a multiple of 16 bytes.
#ifndef PIC_TILE
#define PIC_TILE 128
#endif
constexpr int kTile = PIC_TILE;
struct Tile {
  int32_t cell[kTile];
  float frac[kTile], px[kTile], py[kTile], pz[kTile];
  uint8_t st[kTile];
};
constexpr uint32_t kTileBytes = (uint32_t)sizeof(Tile);
static_assert(sizeof(Tile) % 16 == 0, "bulk copies move multiples of 16 bytes");

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
// Make the initialised barriers visible to the bulk-copy (async) proxy.
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for phase `parity` of the barrier to complete, giving up after a bound
// (each try_wait itself blocks for a while): false = the copies never landed.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 24); ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
// L2 policy for the particle stream: each word is used once per step and the
// whole state is larger than L2.
__device__ __forceinline__ uint64_t evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void bulk_to_smem(void* dst, const void* src, uint32_t bytes,
                                             uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1], %2, [%3], %4;" ::"r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
      : "memory");
}
// One lane: stage particles [first, first + kTile) into t (all of them exist,
// the arrays are 16-byte aligned and first is a multiple of kTile).
template <class ARGS>
__device__ __forceinline__ void tile_issue(const ARGS& a, Tile* t, uint64_t* bar,
                                           int64_t first, uint64_t policy) {
  mbar_expect(bar, kTileBytes);
  bulk_to_smem(t->cell, a.cell + first, kTile * 4, bar, policy);
  bulk_to_smem(t->frac, a.frac + first, kTile * 4, bar, policy);
  bulk_to_smem(t->px, a.px + first, kTile * 4, bar, policy);
  bulk_to_smem(t->py, a.py + first, kTile * 4, bar, policy);
  bulk_to_smem(t->pz, a.pz + first, kTile * 4, bar, policy);
  bulk_to_smem(t->st, a.status + first, kTile, bar, policy);
}

// The current (prev = false) or previous step's field view from the launch
// arguments: ring form from the mirrored ring's start slot, pointer form from
// the per-level pointers.
template <int P, bool RING>
__device__ __forceinline__ void load_fields(StepFields<P, RING>& F, const PushArgsMixed& a,
                                            bool prev) {
  if constexpr (RING) {
    const int64_t start = prev ? a.start_prev : a.start_cur;
    F.E.base = a.ringE + start * a.lstride;
    F.B.base = a.ringB + start * a.lstride;
    F.E.lstride = a.lstride;
    F.B.lstride = a.lstride;
  } else {
#pragma unroll
    for (int l = 0; l <= P; ++l) {
      F.E.ptr[l] = prev ? a.Ep[l] : a.E[l];
      F.B.ptr[l] = prev ? a.Bp[l] : a.B[l];
    }
  }
  F.coef = prev ? a.coef_p : a.coef;
  F.lo = prev ? a.lo_p : a.lo;
  F.hi = prev ? a.hi_p : a.hi;
}

// ---------------------------------------------------------------- predictor features

// phi = (asinh|E|, asinh|B|, asinh p_x, asinh p_y, asinh p_z, log gamma) of
// particle i after macro step n, with E and B at its position extrapolated to
// t_{n+1} (theta = 3/2) from step n's levels: everything known before level
// n+1 arrives.  The temporal extrapolation of every window node is done once
// (feature_nodes_kernel: nodeE, nodeB, W + 1 nodes each, node W repeating
// node 0), so a particle reads two nodes per grid and applies its tent weight:
// the same operations, in the same order, as gathering the levels at the
// particle.  lo, hi: step n's window.  Lost particles and i >= n get zeros;
// E and B are zero outside the window.
// The stored state particle_features reads (status LOST for i >= n), loaded
// apart from the arithmetic so that a caller can issue the loads of its next
// particle before working on the current one.
struct FeatureInput {
  uint8_t st;
  MixedState s;
};
__device__ __forceinline__ FeatureInput feature_input(const PushArgsMixed& a, int64_t i) {
  FeatureInput r;
  r.st = PIC_STATUS_LOST;
  r.s = {0, 0.f, 0.f, 0.f, 0.f};
  if (i < a.n) {
    r.st = a.status[i];
    r.s = load_state(a, i);
  }
  return r;
}

// asinh x = sign(x) ln(|x| + sqrt(x^2 + 1)), with the special-function unit's
// approximate reciprocal square root and logarithm (a few 1e-7 absolute, far
// below the BF16 resolution of the network's input); exactly 0 at 0 (a
// particle without field has zero field features).
__device__ __forceinline__ float asinh_sfu(float x) {
  const float a = fabsf(x);
  const float t = __fmaf_rn(a, a, 1.0f);
  const float r = copysignf(__logf(__fadd_rn(a, __fmul_rn(t, rsqrt_sfu(t)))), x);
  return x == 0.f ? x : r;
}

__device__ __forceinline__ void features_of(const PushArgsMixed& a, const float* nodeE,
                                            const float* nodeB, int32_t lo, int32_t hi,
                                            const FeatureInput& in, float (&f)[6]) {
#pragma unroll
  for (int q = 0; q < 6; ++q) f[q] = 0.f;
  if (in.st & PIC_STATUS_LOST) return;
  const MixedState& s = in.s;
  int32_t je, jb;
  float we, wb;
  if (tent_coords(s.cell, s.frac, lo, hi, je, we, jb, wb)) {
    const float* e = nodeE + (je & a.mask);
    const float* b = nodeB + (jb & a.mask);
    const float e0 = __ldg(e), e1 = __ldg(e + 1), b0 = __ldg(b), b1 = __ldg(b + 1);
    f[0] = asinh_sfu(fabsf(__fmaf_rn(we, __fsub_rn(e1, e0), e0)));
    f[1] = asinh_sfu(fabsf(__fmaf_rn(wb, __fsub_rn(b1, b0), b0)));
  }
  f[2] = asinh_sfu(s.ux);
  f[3] = asinh_sfu(s.uy);
  f[4] = asinh_sfu(s.uz);
  f[5] = 0.5f * __logf(__fadd_rn(1.0f, norm2(s.ux, s.uy, s.uz)));  // log gamma
}

__device__ __forceinline__ void particle_features(const PushArgsMixed& a, const float* nodeE,
                                                  const float* nodeB, int32_t lo, int32_t hi,
                                                  int64_t i, float (&f)[6]) {
  features_of(a, nodeE, nodeB, lo, hi, feature_input(a, i), f);
}

// Field view of macro step s from the mirrored ring and the device copy of
// the slots' window origins (the host's step_slots / fill_mixed, on the GPU):
// for a deferred particle that runs behind the stream.
template <int P>
__device__ __forceinline__ StepFields<P, true> ring_step_fields(const PushArgsMixed& a, int64_t s) {
  StepFields<P, true> F;
  const int64_t R = a.ring_R;
  const int64_t start = ((s - P) % R + R) % R;
  F.E.base = a.ringE + start * a.lstride;
  F.B.base = a.ringB + start * a.lstride;
  F.E.lstride = (int32_t)a.lstride;
  F.B.lstride = (int32_t)a.lstride;
  const int64_t T = a.coef_steps;
  F.coef = s >= a.coef_oldest ? a.coef_all + ((s % T + T) % T) * a.coef_stride : nullptr;
  int64_t lo = INT64_MIN, hi = INT64_MAX;
#pragma unroll
  for (int l = 0; l <= P; ++l) {
    const int64_t o = a.slot_i0[(start + l) % R];
    lo = o > lo ? o : lo;
    hi = o + a.lstride - 1 < hi ? o + a.lstride - 1 : hi;
  }
  F.lo = (int32_t)lo;
  F.hi = (int32_t)hi;
  return F;
}

// Marks particle i as deferred in step s with k (a long sub-cycle pending),
// j of its sub-steps done.
__device__ __forceinline__ void defer_mark(const PushArgsMixed& a, int64_t i, int k_prev, int k,
                                           int64_t s, int j = 0) {
  a.status[i] = (uint8_t)(k_prev | (k << 4));
  if (a.lag_step) {
    a.lag_step[i] = (int32_t)(s - a.step0);
    a.lag_j[i] = (uint16_t)j;
  }
}

// ---------------------------------------------------------------- binned schedule pieces

// Threads per block of the binned kernel: ten warps, two blocks per SM (20
// warps at <= 102 registers, 96 used); measured faster than eight (16 warps at
// <= 128) and twelve (24 at <= 85) on the 16.8M workload.
#ifndef PIC_THREADS
#define PIC_THREADS 320
#endif
constexpr int kThreads = PIC_THREADS;
constexpr int kWarps = kThreads / 32;
#ifndef PIC_STAGES
#define PIC_STAGES 2
#endif
constexpr int kStages = PIC_STAGES;  // staged tiles per warp (one in flight while one is pushed)
static_assert(kTile % 64 == 0, "a tile is whole rounds");
constexpr int kStashK = kDeferMin - 1;
constexpr int kStashCap = 96;  // up to 31 left over and a round's 64
constexpr uint8_t kParity = 0x08;
constexpr uint8_t kDeferMask = 0x70;
// Deferred-k field value 1 (a k no sub-cycle is deferred with): the particle
// belongs to the predicted queue, which pushes it every step until the next
// refresh of the predictions; the stream leaves it alone.
constexpr uint8_t kOwned = 0x10;
static_assert(kDeferMin > 1, "deferred-k value 1 marks predicted-queue particles");

__device__ __forceinline__ int deferred_k(uint8_t st) { return (st >> 4) & 7; }

// Enqueue particle i into the queue of its k; warp-aggregated: one atomic per
// distinct k in the warp.  All 32 lanes call this; key 0 = nothing.
__device__ __forceinline__ void enqueue(const PushArgsMixed& a, int key, int32_t i) {
  if (!__any_sync(0xffffffffu, key != 0)) return;
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(peers) - 1;
  int base = 0;
  if (key != 0 && lane == leader) base = atomicAdd(&a.qcount_out[key], __popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (key != 0) {
    const int rank = __popc(peers & ((1u << lane) - 1u));
    a.queue_out[(int64_t)(key - 1) * a.qcap + base + rank] = i;
  }
}

// A warp's stash of particles waiting for a short sub-cycle of one k: two wide
// words and a byte per entry, so that parking a particle is three stores.
struct Stash {
  float4 a[kStashCap];  // cell (bits), frac, ux, uy
  float2 b[kStashCap];  // uz, particle index (bits)
  uint8_t kp[kStashCap];
};
static_assert(sizeof(Stash) % 16 == 0, "stashes follow each other in shared memory");

__device__ __forceinline__ void stash_put(Stash& S, int pos, int32_t i, const MixedState& s, uint8_t kp) {
  S.a[pos] = make_float4(__int_as_float(s.cell), s.frac, s.ux, s.uy);
  S.b[pos] = make_float2(s.uz, __int_as_float(i));
  S.kp[pos] = kp;
}

// Push the last min(n, 32) stashed particles, one per lane, with 4^k sub-steps
// each.  Warp-collective.  Stash entry kp: k_prev in bits 0-2, bit 3 set for a
// predicted-queue particle (which stays in that queue).
template <int P, bool RING, bool WIDE>
__device__ __forceinline__ void stash_drain(const PushArgsMixed& a, const StepFields<P, RING>& F,
                                            const Stash& S, int k, int& n, unsigned long long* sh) {
  const int lane = threadIdx.x & 31;
  const int cnt = n < 32 ? n : 32;
  if (lane < cnt) {
    const int q = n - cnt + lane;
    const float4 va = S.a[q];
    const float2 vb = S.b[q];
    const uint8_t kp = S.kp[q];
    const int32_t i = __float_as_int(vb.y);
    MixedState s = {__float_as_int(va.x), va.y, va.z, va.w, vb.x};
    const bool ok = subcycle_site<P, RING, RING>(F, a.wtab, a.mask, a.dt, a.inv_dx, a.qm,
                                                 a.field_time, NearRule<WIDE>(a.near), a.mono, k, kp & 7, 0.f, s);
    normalize(s);
    store_state(a, i, s);
    a.status[i] = ok ? (uint8_t)(k | (kp & 8 ? kOwned : 0) | (a.parity_next ? kParity : 0))
                     : (uint8_t)(k | PIC_STATUS_LOST);
    if (!ok) atomicAdd(&sh[11], 1ull);
  }
  __syncwarp();
  n -= cnt;
}

// Deferred item: particle i is in a step before this launch's (a long
// sub-cycle, possibly partly done), or -- a predicted particle -- starts the
// long sub-cycle of this launch's step.  Finish it -- and, if it ran behind the
// stream, every step up to the previous one, taking each step's criterion --
// spending at most heavy_budget sub-steps of long sub-cycles; then take the
// criterion of the current step: pushed at once if k < kDeferMin, else
// deferred again.  Out of budget: the particle stays deferred where it is
// (offset not normalised) and resumes in the next launch -- but not in a step
// before keep_step (the last launch of a call that carries its deferred work
// into the next call: the steps whose levels the ring must keep), which it
// finishes regardless of the budget.  finalize: bring it
// to the end of the last step only (public status).
template <int P, bool RING, bool WIDE>
__device__ __forceinline__ void heavy_particle(const PushArgsMixed& a, const StepFields<P, RING>& Fp,
                                            const StepFields<P, RING>& Fc, const float* wcrit,
                                            int64_t i, ThreadCounters& tc,
                                            unsigned long long* sh, int& defer_key) {
  defer_key = 0;
  const uint8_t st = a.status[i];
  int k = deferred_k(st);
  int k_prev = st & 7;
  MixedState s = load_state(a, i);
  int64_t si = a.step_cur - 1;  // the step the particle is in
  int j0 = 0;                    // its sub-steps already done
  bool lag = false;
  if constexpr (RING) {
    if (a.lag_step) {
      si = a.step0 + a.lag_step[i];
      j0 = a.lag_j[i];
      lag = true;
    }
  }
  int budget = lag && !a.finalize && a.heavy_budget > 0 ? a.heavy_budget : INT_MAX;
  float b0 = 0.f;  // the criterion's B_z of step si (used when k = 0)
  for (;;) {
    // sub-steps j0+1 .. j1 of step si
    const int m = 1 << (2 * k);
    int j1 = m;
    if (k >= kDeferMin && m - j0 > budget && si >= a.keep_step) j1 = j0 + budget;
    bool ok = false;
    // the particle's own step's fields, so that a warp whose particles are in
    // different steps still runs their sub-steps together
    StepFields<P, RING> Fs = si == a.step_cur ? Fc : Fp;
    if constexpr (RING) {
      if (si < a.step_cur - 1) Fs = ring_step_fields<P>(a, si);
    }
    if (!RING || Fs.coef) {
      ok = subcycle_site<P, RING, RING>(Fs, a.wtab, a.mask, a.dt, a.inv_dx, a.qm, a.field_time, NearRule<WIDE>(a.near),
                                        a.mono, k, k_prev, b0, s, j0, j1);
    } else {  // further behind than the tables kept
      if constexpr (RING)
        ok = subcycle_f32<P, true, false>(Fs, a.wtab, a.mask, a.dt, a.inv_dx, a.qm, a.field_time, NearRule<WIDE>(a.near),
                                          a.mono, k, k_prev, b0, s, j0, j1);
    }
    if (k >= kDeferMin) budget -= j1 - j0;
    if (!ok) {
      store_state(a, i, s);
      a.status[i] = (uint8_t)(k | PIC_STATUS_LOST);
      atomicAdd(&sh[11], 1ull);
      return;
    }
    if (j1 < m) {  // out of budget inside the sub-cycle: resume here next launch
      store_state(a, i, s);
      defer_mark(a, i, k_prev, k, si, j1);
      defer_key = k;
      return;
    }
    normalize(s);
    if (si == a.step_cur) {  // the current step's short sub-cycle is done
      store_state(a, i, s);
      a.status[i] = (uint8_t)(k | (a.parity_next ? kParity : 0));
      return;
    }
    if (si == a.step_cur - 1) {
      if (a.finalize) {
        store_state(a, i, s);
        a.status[i] = (uint8_t)k;
        return;
      }
      int32_t je, jb;
      float we, wb;
      if (!tent_coords(s.cell, s.frac, Fc.lo, Fc.hi, je, we, jb, wb)) {
        store_state(a, i, s);
        a.status[i] = (uint8_t)(k | PIC_STATUS_LOST);
        atomicAdd(&sh[11], 1ull);
        return;
      }
      bool capped;
      const int kn = criterion_f32<P>(Fc.B, wcrit, jb, wb, a.mask, s, a.qm_abs, a.dt, a.psi_max,
                                      a.k_max, capped, b0);
      count_step(tc, sh, kn, capped);
      if (kn >= kDeferMin) {
        store_state(a, i, s);
        defer_mark(a, i, k, kn, a.step_cur);
        defer_key = kn;
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
    if constexpr (RING) {
      si += 1;
      const StepFields<P, true> Fs = si == a.step_cur - 1 ? Fp : ring_step_fields<P>(a, si);
      int32_t je, jb;
      float we, wb;
      if (!tent_coords(s.cell, s.frac, Fs.lo, Fs.hi, je, we, jb, wb)) {
        store_state(a, i, s);
        a.status[i] = (uint8_t)(k | PIC_STATUS_LOST);
        atomicAdd(&sh[11], 1ull);
        return;
      }
      bool capped;
      const int kn = criterion_f32<P>(Fs.B, wcrit, jb, wb, a.mask, s, a.qm_abs, a.dt, a.psi_max,
                                      a.k_max, capped, b0);
      count_step(tc, sh, kn, capped);
      k_prev = k;
      k = kn;
      j0 = 0;
      if (k >= kDeferMin && budget <= 0 && si >= a.keep_step) {
        store_state(a, i, s);
        defer_mark(a, i, k_prev, k, si);
        defer_key = k;
        return;
      }
    }
  }
}

// Predicted item: particle i was binned at the last refresh of the
// predictions as likely to take k_pred.  Skipped unless it still belongs to
// the predicted queue (a particle deferred since then is the deferred items'
// and then the stream's).  Takes its exact criterion: k = 0, and a short k
// equal to the predicted one, are pushed at once (a warp of right predictions
// runs dense); another short k goes to the caller's stash (sk, with its state
// s and stash byte kp); both stay in the queue.  A long sub-cycle leaves the
// queue and, with
// resumable sub-cycles (run_heavy), starts at once in the caller's deferred-
// particle code, at most heavy_budget sub-steps in this launch -- so a warp of
// right predictions runs dense from the start of the launch -- else it is
// deferred to the next launch (key), as the stream would.
template <int P, bool RING, bool WIDE>
__device__ __forceinline__ void predicted_particle(const PushArgsMixed& a, const StepFields<P, RING>& Fc,
                                                   const float* wcrit, int64_t i, int k_pred,
                                                   ThreadCounters& tc, unsigned long long* sh,
                                                   int& key, int& sk, MixedState& s, uint8_t& kp,
                                                   bool& run_heavy) {
  const uint8_t st = a.status[i];
  if ((st & (PIC_STATUS_LOST | kDeferMask)) != kOwned) return;
  const int k_prev = st & 7;
  kp = (uint8_t)(k_prev | 8);
  s = load_state(a, i);
  int32_t je, jb;
  float we, wb;
  if (!tent_coords(s.cell, s.frac, Fc.lo, Fc.hi, je, we, jb, wb)) {
    a.status[i] = (uint8_t)(k_prev | PIC_STATUS_LOST);
    atomicAdd(&sh[11], 1ull);
    return;
  }
  bool capped;
  float b0;
  const int k = criterion_f32<P>(Fc.B, wcrit, jb, wb, a.mask, s, a.qm_abs, a.dt, a.psi_max,
                                 a.k_max, capped, b0);
  count_step(tc, sh, k, capped);
  if (k == 0 || (k == k_pred && k < kDeferMin)) {
    const bool ok = subcycle_site<P, RING, RING>(Fc, a.wtab, a.mask, a.dt, a.inv_dx, a.qm,
                                                 a.field_time, NearRule<WIDE>(a.near), a.mono, k, k_prev, b0, s);
    normalize(s);
    store_state(a, i, s);
    a.status[i] = ok ? (uint8_t)(k | kOwned | (a.parity_next ? kParity : 0))
                     : (uint8_t)(k | PIC_STATUS_LOST);
    if (!ok) atomicAdd(&sh[11], 1ull);
  } else if (k < kDeferMin) {
    sk = k;
  } else {
    defer_mark(a, i, k_prev, k, a.step_cur);  // in this step, none of its sub-steps done
    if (RING && a.lag_step)
      run_heavy = true;
    else
      key = k;
  }
}

}  // namespace pic
