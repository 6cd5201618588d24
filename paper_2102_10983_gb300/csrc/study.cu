// Single-electron studies of Secs. IV-VII on the GPU: electrons from rest
// through the Gaussian-enveloped plane wave of Eqs. laser5 - laser3
// (a = a0 exp(-(xi - xi0)^2 / (2 sigma^2)) sin xi, E_y = B_z = -da/dxi) with
// the field sampled on the grid (the "perfectly propagating PIC" of Sec. III):
// E_y at nodes i dx and times n dt, B_z at (i + 1/2) dx and (n + 1/2) dt.
//
// Each electron integrates its whole trajectory with the method (Algorithm 1 of
// Sec. IV, order-p Lagrange in time of Sec. VI, tent in space, Boris), in FP64
// compiled with -fmad=false in the order of a serial evaluation.  A trajectory
// is one serial chain, and the FP64 unit takes 19 clocks for a warp instruction
// with one active lane as with 32.  So there are two forms of the same bits:
//  study_kernel, one warp per electron: the chain is taken by every lane alike
//    and the work beside it is dealt to the lanes: the field at the nodes about
//    the electron (the formula's exp, sin, cos: one evaluation of the warp per
//    macro step serves all levels, grids and nodes, and the diagnostic's a), the
//    Lagrange weights and the temporal sums of 32 sub-steps at a time (orders 1,
//    3 and 5, a0 = 5, lambda/75, 64 electrons each, 2,000 macro steps: 25 ms, 264
//    as one thread per electron);
//  study_many_kernel, one thread per electron: 32 chains for the unit's time of
//    one, where there are more electrons than the unit has time for.
// pic_study_run chooses by the cases' steps and electrons (study_by_warp).
//
// Per electron and macro step (Sec. IV, Eqs. R error, gamma error): R = gamma
// - p_x, the energy error |gamma - gamma_th| / gamma_th with gamma_th = 1 +
// a(xi_p)^2 / 2 at the momentum's phase xi_p = t_p - x_p (t_p = t_{n+1} - h/2,
// x_p = x - (h/2) v_x); per case the maxima over steps and electrons, electron
// 0's own values, N and N* (Sec. VII).
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <vector>

#include "fp64_push.cuh"
#include "pic_internal.h"

namespace pic {
namespace {

// prod_{k != j} (c_k + theta) times the rounded reciprocal of the integer
// denominator, c_k = p-k-1/2 (E) or p-k-1 (B).
template <int P>
__device__ __forceinline__ void lagrange(bool is_e, double theta, double* w) {
  const double c_off = is_e ? -0.5 : -1.0;
#pragma unroll
  for (int j = 0; j <= P; ++j) {
    double num = 1.0;
    bool first = true;
    int den = 1;
#pragma unroll
    for (int k = 0; k <= P; ++k) {
      if (k == j) continue;
      const double factor = ((double)(P - k) + c_off) + theta;
      num = first ? factor : num * factor;
      first = false;
      den *= j - k;
    }
    w[j] = num * (1.0 / (double)den);
  }
}

// theta of the j-th (0-based) of 4^k sub-steps.
__device__ __forceinline__ double theta_of(int field_time, int j, int k) {
  const double inv_m = scale_down64(1.0, k);
  return field_time == 0 ? 0.5 + (double)j * inv_m : ((double)j + 0.5) * inv_m;
}

__device__ __forceinline__ int mod_pos(int64_t a, int m) {
  const int r = (int)(a % m);
  return r < 0 ? r + m : r;
}

// The field about the electron: per grid (E: times n dt, nodes i dx; B: both
// half a step on) the values at three nodes base .. base + 2 and levels n-P ..
// n, one per lane (two at order 5), node i and level l in the slot (i mod 3, l
// mod (P + 1)), so that a step on replaces the oldest level only and a node on
// the hindmost node; and a copy in shared memory for the lanes to read.
template <int P>
struct FieldTile {
  static constexpr int kPerGrid = 3 * (P + 1), kSlots = 2 * kPerGrid;
  static constexpr int kPer = (kSlots + 31) / 32;  // slots per lane; lane 31's last is free
  int64_t node[kPer], level[kPer];

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int t = 0; t < kPer; ++t) node[t] = level[t] = INT64_MIN;
  }
  // Bring the tile to nodes je .. je + 2 (E), jb .. jb + 2 (B) and levels n-P
  // .. n.  The free slot evaluates a(xi_diag), returned to every lane.
  __device__ __forceinline__ double fill(const pic_study_case& q, double* sm, int64_t je, int64_t jb, int64_t n,
                                         double xi_diag) {
    const int lane = threadIdx.x;
    const double ss = q.sigma * q.sigma, s2 = 2.0 * q.sigma * q.sigma;
    double a = 0.0;
    __syncwarp();
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int slot = lane + 32 * t;
      const bool used = slot < kSlots, is_b = slot >= kPerGrid;
      const int r = is_b ? slot - kPerGrid : slot;
      const int64_t j = is_b ? jb : je;
      const int64_t i = j + (r / (P + 1) + 3 - mod_pos(j, 3)) % 3;
      const int64_t l = n - (mod_pos(n, P + 1) + (P + 1) - r % (P + 1)) % (P + 1);
      const bool stale = used && (node[t] != i || level[t] != l);
      const bool diag = t == kPer - 1 && lane == 31;
      if (stale || diag) {
        const double off = is_b ? 0.5 : 0.0;
        const double xi = diag ? xi_diag
                               : (ll_to_double(l) + off) * q.dt - (ll_to_double(i) + off) * q.dx;
        const double d = xi - q.xi0;
        const double env = q.a0 * exp(div_rn(-(d * d), s2));
        double sn, cs;
        sincos(xi, &sn, &cs);  // one argument reduction for both
        if (stale) {
          sm[slot] = -(env * (cs - div_rn(d, ss) * sn));  // E_y = B_z = -da/dxi (Eq. laser5)
          node[t] = i;
          level[t] = l;
        } else {
          a = env * sn;
        }
      }
    }
    __syncwarp();
    return __shfl_sync(0xffffffffu, a, 31);
  }
  // The values at nodes j, j + 1 of one grid, levels ascending.
  __device__ __forceinline__ void read(const double* sm, bool is_b, int64_t j, int64_t n, double* v0,
                                       double* v1) const {
    const double* g = sm + (is_b ? kPerGrid : 0);
    const int a = mod_pos(j, 3);
    const double* r0 = g + a * (P + 1);
    const double* r1 = g + (a == 2 ? 0 : a + 1) * (P + 1);
    int l = mod_pos(n - P, P + 1);
#pragma unroll
    for (int q = 0; q <= P; ++q) {
      v0[q] = r0[l];
      v1[q] = r1[l];
      l = l == P ? 0 : l + 1;
    }
  }
};

template <int P, bool UNIT>
__device__ __forceinline__ void study_electron(const pic_study_case& q, double x0, double* sm,
                                               double* out_eps_r, double* out_eps_e, double* out_gmax,
                                               int64_t* n_star, int64_t* substeps, int64_t* k_count) {
  const int lane = threadIdx.x;
  const double dt = q.dt, inv_dx = 1.0 / q.dx;
  const double qm_abs = fabs(q.qm);
  const float scale = criterion_f64_scale(qm_abs, dt, q.psi_max);
  // the lane's weights for k <= 2: lanes 0 .. 15 the rows of k = 2, 16 .. 19
  // those of k = 1, the rest theta = 1/2 (k = 0 and the criterion)
  double wE0[P + 1], wB0[P + 1];
  {
    const double th = lane < 16 ? theta_of(q.field_time, lane, 2)
                      : lane < 20 ? theta_of(q.field_time, lane - 16, 1) : 0.5;
    lagrange<P>(true, th, wE0);
    lagrange<P>(false, th, wB0);
  }
  FieldTile<P> tile;
  tile.init();
  NodePair<P> E, B;
  Mom64 p = mom64(0.0, 0.0, 0.0);
  double xi = x0;
  int k_prev = 0;
  double eps_r = 0.0, eps_e = 0.0, gmax = 1.0;
  int64_t ns = 0, sub = 0, count = 0;
  double xi_diag = q.xi0, g_diag = 1.0;  // the last step's momentum phase and gamma
  auto locate = [&](Coords64& c) {
    const double s = xi * inv_dx;
    if (!coords64_fast(s, c)) coords64_any(s, c);
  };
  auto diagnose = [&](double a) {  // |gamma - gamma_th| / gamma_th of the step before
    const double g_th = 1.0 + 0.5 * a * a;
    const double de = div_rn(fabs(g_diag - g_th), g_th);
    if (de > eps_e) eps_e = de;
  };
  for (int64_t n = 0; n < q.n_steps; ++n) {
    Coords64 c;
    locate(c);
    const double a = tile.fill(q, sm, c.je, c.jb, n, xi_diag);
    if (n > 0) diagnose(a);
    int64_t je = c.je, jb = c.jb, te = je, tb = jb;  // the electron's nodes and the tile's
    tile.read(sm, false, je, n, E.v0, E.v1);
    tile.read(sm, true, jb, n, B.v0, B.v1);
    E.sums(wE0);
    B.sums(wB0);
    const double b0 = __shfl_sync(0xffffffffu, B.f, 31) + c.wb * __shfl_sync(0xffffffffu, B.d, 31);
    bool capped;
    const int k = criterion_f64(scale, qm_abs, dt, q.psi_max, q.k_max, b0, p.x, p.y, p.z, capped);
    const int m = 1 << (2 * k);
    const double h = pow4_down64(dt, k), h_old = pow4_down64(dt, k_prev);
    if (lane == k) ++count;
    sub += m;
    if (k > 0) ns += m;
    double half = 0.5 * (0.5 * (h_old + h));
    double wE[P + 1], wB[P + 1];
#pragma unroll
    for (int l = 0; l <= P; ++l) {
      wE[l] = wE0[l];
      wB[l] = wB0[l];
    }
    const int first = k == 0 ? 31 : k == 1 ? 16 : 0;  // the lane with the first sub-step's sums
    Push64 r;
    double ef, ed, bf, bd;  // sub-step j's sums
    auto take = [&](int j) {
      const int src = (first + (j & 31)) & 31;
      ef = __shfl_sync(0xffffffffu, E.f, src);
      ed = __shfl_sync(0xffffffffu, E.d, src);
      bf = __shfl_sync(0xffffffffu, B.f, src);
      bd = __shfl_sync(0xffffffffu, B.d, src);
    };
    take(0);
    for (int j = 0; j < m; ++j) {
      if (j > 0) locate(c);
      // the gather overlaps the tests: taken again where they find new sums
      double ey = ef + c.we * ed, bz = bf + c.wb * bd;
      const bool moved = c.je != je || c.jb != jb, more = k > 2 && (j & 31) == 0;
      if (moved || more) {
        if (more) {  // the next 32 sub-steps' weights
          const double th = theta_of(q.field_time, j + lane, k);
          lagrange<P>(true, th, wE);
          lagrange<P>(false, th, wB);
        }
        if (moved) {
          // one node on is in the tile; anything else (a step of more than a
          // node, c dt > dx, or a turn back) is evaluated anew
          if (c.je < te || c.je > te + 1 || c.jb < tb || c.jb > tb + 1) {
            te = c.je;
            tb = c.jb;
            tile.fill(q, sm, te, tb, n, xi_diag);
          }
          je = c.je;
          jb = c.jb;
          tile.read(sm, false, je, n, E.v0, E.v1);
          tile.read(sm, true, jb, n, B.v0, B.v1);
        }
        E.sums(wE);
        B.sums(wB);
        take(j);
        ey = ef + c.we * ed;
        bz = bf + c.wb * bd;
      }
      take(j + 1);
      Mom64 pn;
      const bool ok = push64_try<UNIT, false>(0.0, ey, bz, half, q.qm, p, pn, r);
      double xn = xi + h * r.vx;
      if (!ok) {
        pn = p;
        r = push64_any<UNIT, false>(0.0, ey, bz, half, q.qm, &pn);
        xn = xi + h * r.vx;
      }
      p = pn;
      xi = xn;
      half = 0.5 * h;
    }
    k_prev = k;
    const double dR = fabs((r.gam - p.x) - 1.0);
    if (dR > eps_r) eps_r = dR;
    if (r.gam > gmax) gmax = r.gam;
    const double t_p = ll_to_double(n + 1) * dt - 0.5 * h;
    xi_diag = t_p - (xi - 0.5 * h * r.vx);
    g_diag = r.gam;
  }
  if (q.n_steps > 0) {
    Coords64 c;
    locate(c);
    diagnose(tile.fill(q, sm, c.je, c.jb, q.n_steps, xi_diag));
  }
  *out_eps_r = eps_r;
  *out_eps_e = eps_e;
  *out_gmax = gmax;
  *n_star = ns;
  *substeps = sub;
  *k_count = count;
}

// The field values of one grid at a node pair for the levels n - P .. n (E:
// times l dt; B: half a step on), from the formula as the electron comes to
// them: a macro step that keeps the nodes computes only the newest level.
template <int P, bool IS_B>
struct FieldPair {
  NodePair<P> v;
  int64_t node = INT64_MIN, level = INT64_MIN;
  static __device__ __forceinline__ double at(const pic_study_case& q, int64_t l, int64_t i) {
    const double off = IS_B ? 0.5 : 0.0;
    const double xi = (ll_to_double(l) + off) * q.dt - (ll_to_double(i) + off) * q.dx;
    const double d = xi - q.xi0, ss = q.sigma * q.sigma;
    const double env = q.a0 * exp(div_rn(-(d * d), 2.0 * q.sigma * q.sigma));
    double sn, cs;
    sincos(xi, &sn, &cs);
    return -(env * (cs - div_rn(d, ss) * sn));  // as FieldTile::fill
  }
  __device__ __forceinline__ void ensure(const pic_study_case& q, int64_t j, int64_t n) {
    if (j == node && n == level) return;
    int first = 0;
    if (j == node && n == level + 1) {
#pragma unroll
      for (int l = 0; l < P; ++l) {
        v.v0[l] = v.v0[l + 1];
        v.v1[l] = v.v1[l + 1];
      }
      first = P;
    }
#pragma unroll 1
    for (int l = first; l <= P; ++l) {
      const double a = at(q, n - P + l, j), b = at(q, n - P + l, j + 1);
#pragma unroll
      for (int r = 0; r <= P; ++r)
        if (r == l) {
          v.v0[r] = a;
          v.v1[r] = b;
        }
    }
    node = j;
    level = n;
  }
};

// study_electron by one thread.
template <int P, bool UNIT>
__device__ __forceinline__ void study_electron_alone(const pic_study_case& q, double x0, double* out_eps_r,
                                                     double* out_eps_e, double* out_gmax, int64_t* n_star,
                                                     int64_t* substeps, int64_t* k_count) {
  const double dt = q.dt, inv_dx = 1.0 / q.dx;
  const double qm_abs = fabs(q.qm);
  const float scale = criterion_f64_scale(qm_abs, dt, q.psi_max);
  FieldPair<P, false> E;
  FieldPair<P, true> B;
  Mom64 p = mom64(0.0, 0.0, 0.0);
  double xi = x0;
  int k_prev = 0;
  double eps_r = 0.0, eps_e = 0.0, gmax = 1.0;
  int64_t ns = 0, sub = 0;
  double w[P + 1];
  Coords64 c;
  auto locate = [&]() {
    const double s = xi * inv_dx;
    if (!coords64_fast(s, c)) coords64_any(s, c);
  };
  auto gather = [&](auto& F, bool is_b, int64_t j, int64_t n, double theta, double off) {
    F.ensure(q, j, n);
    lagrange<P>(is_b ? false : true, theta, w);
    F.v.sums(w);
    return F.v.f + off * F.v.d;
  };
  for (int64_t n = 0; n < q.n_steps; ++n) {
    locate();
    const double b0 = gather(B, true, c.jb, n, 0.5, c.wb);
    bool capped;
    const int k = criterion_f64(scale, qm_abs, dt, q.psi_max, q.k_max, b0, p.x, p.y, p.z, capped);
    const int m = 1 << (2 * k);
    const double h = pow4_down64(dt, k), h_old = pow4_down64(dt, k_prev);
    k_count[k] += 1;
    sub += m;
    if (k > 0) ns += m;
    double half = 0.5 * (0.5 * (h_old + h));
    Push64 r;
#pragma unroll 1
    for (int j = 0; j < m; ++j) {
      if (j > 0) locate();
      const double th = theta_of(q.field_time, j, k);
      const double ey = gather(E, false, c.je, n, th, c.we), bz = gather(B, true, c.jb, n, th, c.wb);
      r = push64<UNIT, false>(0.0, ey, bz, half, q.qm, p);
      xi = xi + h * r.vx;
      half = 0.5 * h;
    }
    k_prev = k;
    const double dR = fabs((r.gam - p.x) - 1.0);
    if (dR > eps_r) eps_r = dR;
    if (r.gam > gmax) gmax = r.gam;
    const double t_p = ll_to_double(n + 1) * dt - 0.5 * h;
    const double ph = t_p - (xi - 0.5 * h * r.vx), d = ph - q.xi0;
    double sn, cs;
    sincos(ph, &sn, &cs);
    const double a = q.a0 * exp(div_rn(-(d * d), 2.0 * q.sigma * q.sigma)) * sn;
    const double g_th = 1.0 + 0.5 * a * a;
    const double de = div_rn(fabs(r.gam - g_th), g_th);
    if (de > eps_e) eps_e = de;
  }
  *out_eps_r = eps_r;
  *out_eps_e = eps_e;
  *out_gmax = gmax;
  *n_star = ns;
  *substeps = sub;
}

__device__ __forceinline__ void atomic_max_pos(unsigned long long* a, double v) {
  atomicMax(a, (unsigned long long)__double_as_longlong(v));  // v >= 0
}

struct StudyAcc {
  unsigned long long eps_r, eps_e, gmax;  // doubles >= 0 as bits
  unsigned long long n_star_sum, substeps_sum;
  unsigned long long k_hist[8];
};

template <int P>
__device__ __forceinline__ void study_order(const pic_study_case& q, double x0, double* sm, double* er,
                                            double* ee, double* gm, int64_t* ns, int64_t* sub, int64_t* kc) {
  if (fabs(q.qm) == 1.0)
    study_electron<P, true>(q, x0, sm, er, ee, gm, ns, sub, kc);
  else
    study_electron<P, false>(q, x0, sm, er, ee, gm, ns, sub, kc);
}

template <int P>
__device__ __forceinline__ void study_order_alone(const pic_study_case& q, double x0, double* er, double* ee,
                                                  double* gm, int64_t* ns, int64_t* sub, int64_t* kc) {
  if (fabs(q.qm) == 1.0)
    study_electron_alone<P, true>(q, x0, er, ee, gm, ns, sub, kc);
  else
    study_electron_alone<P, false>(q, x0, er, ee, gm, ns, sub, kc);
}

// An electron's part in its case's results.
__device__ __forceinline__ void study_report(StudyAcc& A, pic_study_result& r, int e, double er, double ee,
                                             double gm, int64_t ns, int64_t sub) {
  atomic_max_pos(&A.eps_r, er);
  atomic_max_pos(&A.eps_e, ee);
  atomic_max_pos(&A.gmax, gm);
  atomicAdd(&A.n_star_sum, (unsigned long long)ns);
  atomicAdd(&A.substeps_sum, (unsigned long long)sub);
  if (e == 0) {
    r.eps_dephasing_first = er;
    r.eps_energy_first = ee;
    r.gamma_max_first = gm;
    r.n_star_first = ns;
  }
}

// One warp per CTA and electron: block b runs electron b mod per_case of case
// b / per_case; every order in one launch, so the cases of all orders run at
// once.
__global__ void __launch_bounds__(32) study_kernel(const pic_study_case* cases, pic_study_result* out,
                                                   StudyAcc* acc, int per_case) {
  __shared__ double sm[FieldTile<kMaxOrder>::kSlots];
  const int c = blockIdx.x / per_case;
  const pic_study_case q = cases[c];
  const int e = blockIdx.x % per_case;
  if (e >= q.n_electrons) return;
  const double x0 = (2.0 * M_PI) * (double)e / (double)q.n_electrons;
  double er, ee, gm;
  int64_t ns, sub, kc;
  switch (q.order) {
    case 1: study_order<1>(q, x0, sm, &er, &ee, &gm, &ns, &sub, &kc); break;
    case 2: study_order<2>(q, x0, sm, &er, &ee, &gm, &ns, &sub, &kc); break;
    case 3: study_order<3>(q, x0, sm, &er, &ee, &gm, &ns, &sub, &kc); break;
    case 4: study_order<4>(q, x0, sm, &er, &ee, &gm, &ns, &sub, &kc); break;
    default: study_order<5>(q, x0, sm, &er, &ee, &gm, &ns, &sub, &kc); break;
  }
  StudyAcc& A = acc[c];
  if (threadIdx.x < 8 && kc) atomicAdd(&A.k_hist[threadIdx.x], (unsigned long long)kc);
  if (threadIdx.x == 0) study_report(A, out[c], e, er, ee, gm, ns, sub);
}

// One thread per electron, one warp per CTA: block b runs electrons 32 (b mod
// per_case) .. + 31 of case b / per_case.
__global__ void __launch_bounds__(32) study_many_kernel(const pic_study_case* cases, pic_study_result* out,
                                                        StudyAcc* acc, int per_case) {
  const int c = blockIdx.x / per_case;
  const pic_study_case q = cases[c];
  const int e = (blockIdx.x % per_case) * 32 + (int)threadIdx.x;
  if (e >= q.n_electrons) return;
  const double x0 = (2.0 * M_PI) * (double)e / (double)q.n_electrons;
  double er, ee, gm;
  int64_t ns, sub;
  int64_t kc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  switch (q.order) {
    case 1: study_order_alone<1>(q, x0, &er, &ee, &gm, &ns, &sub, kc); break;
    case 2: study_order_alone<2>(q, x0, &er, &ee, &gm, &ns, &sub, kc); break;
    case 3: study_order_alone<3>(q, x0, &er, &ee, &gm, &ns, &sub, kc); break;
    case 4: study_order_alone<4>(q, x0, &er, &ee, &gm, &ns, &sub, kc); break;
    default: study_order_alone<5>(q, x0, &er, &ee, &gm, &ns, &sub, kc); break;
  }
  StudyAcc& A = acc[c];
  for (int k = 0; k < 8; ++k)
    if (kc[k]) atomicAdd(&A.k_hist[k], (unsigned long long)kc[k]);
  study_report(A, out[c], e, er, ee, gm, ns, sub);
}

// Whether a warp per electron is the faster form.  It takes the FP64 unit's time
// for every electron and macro step; a thread per electron takes the longest
// case's chain, in which a warp runs as long as its largest 4^k.  Measured per macro
// step and order, a0 = 25, lambda/75 (5 to 100 likewise): without and with sub-cycles,
// which an electron from rest takes once the pulse's envelope reaches four times the
// criterion's threshold.  4,352 electrons at order 3: 72 us by warps and 77 by
// threads, 10,240 162 and 79; without sub-cycles 49 and 25, 111 and 25.
bool study_by_warp(const pic_study_case* cases, int32_t n, int sms) {
  static const double chain_us[2][kMaxOrder] = {{16.7, 20.6, 24.6, 28.4, 32.3}, {42.0, 61.0, 77.0, 94.0, 111.0}};
  static const double warp_ns[2][kMaxOrder] = {{10.4, 10.8, 11.3, 11.9, 15.8}, {15.1, 15.9, 16.6, 17.3, 22.0}};
  double by_warp = 0.0, by_thread = 0.0;  // us
  for (int32_t i = 0; i < n; ++i) {
    const pic_study_case& q = cases[i];
    const double steps = (double)q.n_steps, top = fabs(q.qm * q.a0) * q.dt / (8.0 * q.psi_max);
    double plain = steps;  // macro steps before the sub-cycles
    if (q.k_max > 0 && top > 1.0) plain = fmin(steps, fmax(0.0, (q.xi0 - q.sigma * sqrt(2.0 * log(top))) / q.dt));
    const int o = q.order - 1;
    const double chain = plain * chain_us[0][o] + (steps - plain) * chain_us[1][o];
    by_warp += (plain * warp_ns[0][o] + (steps - plain) * warp_ns[1][o]) * (double)q.n_electrons;
    by_thread = chain > by_thread ? chain : by_thread;
  }
  return by_warp * 1e-3 * 152.0 / (double)(sms > 0 ? sms : 152) <= by_thread;
}

}  // namespace
}  // namespace pic

using namespace pic;

extern "C" int pic_study_run(const pic_study_case* cases, int32_t n_cases, pic_study_result* out,
                             void* stream) {
  if (!cases || !out || n_cases < 1 || n_cases > 65535) {
    set_global_error("pic_study_run: bad arguments");
    return PIC_EINVAL;
  }
  for (int32_t i = 0; i < n_cases; ++i) {
    const pic_study_case& q = cases[i];
    if (!(q.dt > 0) || !(q.dx > 0) || !(q.psi_max > 0) || !(q.sigma > 0) || q.order < 1 ||
        q.order > kMaxOrder || q.k_max < 0 || q.k_max > kMaxK || q.n_electrons < 1 ||
        q.n_electrons > 256 || q.n_steps < 0 || (q.field_time != 0 && q.field_time != 1)) {
      set_global_error("pic_study_run: case parameter out of range");
      return PIC_EINVAL;
    }
  }
  cudaStream_t st = (cudaStream_t)stream;
  pic_study_case* dcases = nullptr;
  pic_study_result* dout = nullptr;
  StudyAcc* dacc = nullptr;
  auto cleanup = [&]() {
    cudaFree(dcases);
    cudaFree(dout);
    cudaFree(dacc);
  };
  cudaError_t e = cudaMalloc(&dcases, sizeof(pic_study_case) * n_cases);
  if (e == cudaSuccess) e = cudaMalloc(&dout, sizeof(pic_study_result) * n_cases);
  if (e == cudaSuccess) e = cudaMalloc(&dacc, sizeof(StudyAcc) * n_cases);
  if (e != cudaSuccess) {
    cleanup();
    set_global_error("pic_study_run: device allocation failed");
    return PIC_ENOMEM;
  }
  e = cudaMemcpyAsync(dcases, cases, sizeof(pic_study_case) * n_cases, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(dacc, 0, sizeof(StudyAcc) * n_cases, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(dout, 0, sizeof(pic_study_result) * n_cases, st);
  int per_case = 1;
  for (int32_t i = 0; i < n_cases; ++i)
    per_case = cases[i].n_electrons > per_case ? cases[i].n_electrons : per_case;
  if (e == cudaSuccess) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (study_by_warp(cases, n_cases, sms)) {
      study_kernel<<<(unsigned)(n_cases * per_case), 32, 0, st>>>(dcases, dout, dacc, per_case);
    } else {
      per_case = (per_case + 31) / 32;
      study_many_kernel<<<(unsigned)(n_cases * per_case), 32, 0, st>>>(dcases, dout, dacc, per_case);
    }
    e = cudaGetLastError();
  }
  std::vector<StudyAcc> acc(n_cases);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(out, dout, sizeof(pic_study_result) * n_cases, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(acc.data(), dacc, sizeof(StudyAcc) * n_cases, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cleanup();
  if (e != cudaSuccess) {
    set_global_error(cudaGetErrorString(e));
    return PIC_ECUDA;
  }
  for (int32_t i = 0; i < n_cases; ++i) {
    pic_study_result& r = out[i];
    memcpy(&r.eps_dephasing, &acc[i].eps_r, 8);
    memcpy(&r.eps_energy, &acc[i].eps_e, 8);
    memcpy(&r.gamma_max, &acc[i].gmax, 8);
    r.n_steps = cases[i].n_steps;
    r.n_star_mean = (double)acc[i].n_star_sum / (double)cases[i].n_electrons;
    r.substeps = (int64_t)acc[i].substeps_sum;
    for (int k = 0; k < 8; ++k) r.k_hist[k] = (int64_t)acc[i].k_hist[k];
  }
  return PIC_OK;
}
