// Particle arrays between FP64 (the ABI's) and the mixed layout: x = (cell +
// frac) dx with an int32 cell and an FP32 offset in [0, 1), FP32 momenta.
//
// 52 bytes per particle pass through memory either way.  What bounded a plain
// conversion was not that but the FP64 unit: FP64 <-> FP32 and integer
// conversions, floors and sums each take its 19 clocks per warp instruction,
// eight and six of them per particle (4,194,304 particles: 73 us to the mixed
// layout, 3.0 TB/s, and 62 us back).  Below the conversions are integer
// arithmetic (same bits) and the unit sees one multiplication per particle one
// way, an addition and a multiplication the other; two particles per thread,
// 16-byte accesses where the arrays allow: 34 us (6.4 TB/s) and 43 us.  A batch
// converts all its ensembles in one launch (512 ensembles, 11.9M particles: 2.1
// ms each way as a launch per ensemble, 0.11 ms so).
#include <math.h>

#include "fp64_push.cuh"
#include "pic_internal.h"

namespace pic {
namespace {

// (float)v, to nearest: the significand cut to 24 bits in integers where the
// result is normal.
__device__ __forceinline__ float to_f32(double v) {
  const uint64_t u = (uint64_t)__double_as_longlong(v);
  const uint32_t e = (uint32_t)(u >> 52) & 0x7ffu;
  const uint64_t m = (u & 0x7fffffffffffffffull) - ((uint64_t)(1023 - 127) << 52);
  const uint32_t r = (uint32_t)((m + 0xfffffffull + ((m >> 29) & 1)) >> 29);
  if (e - 897u < 254u) return __int_as_float((int32_t)(r | ((uint32_t)(u >> 63) << 31)));
  return (u << 1) == 0 ? __int_as_float((int32_t)(u >> 32)) : (float)v;
}
// (double)f.
__device__ __forceinline__ double to_f64(float f) {
  const uint32_t u = (uint32_t)__float_as_int(f);
  const uint32_t e = (u >> 23) & 0xffu;
  if (e - 1u < 254u) {
    const uint64_t v = ((uint64_t)(u & 0x7fffffffu) << 29) + ((uint64_t)(1023 - 127) << 52);
    return __longlong_as_double((long long)(v | ((uint64_t)(u & 0x80000000u) << 32)));
  }
  return (u << 1) == 0 ? __longlong_as_double((long long)((uint64_t)u << 32)) : (double)f;
}
// (double)c of an int32.
__device__ __forceinline__ double i32_to_f64(int32_t c) {
  const uint32_t a = c < 0 ? 0u - (uint32_t)c : (uint32_t)c;
  const double d = ll_to_double((int64_t)a);
  return __longlong_as_double(__double_as_longlong(d) | (c < 0 ? (long long)0x8000000000000000ull : 0ll));
}

__device__ __forceinline__ void split_x(double x, double inv_dx, int32_t& cell, float& frac) {
  const double s = __dmul_rn(x, inv_dx);
  const uint32_t h = (uint32_t)((uint64_t)__double_as_longlong(s) >> 32);
  float f;
  int32_t c;
  if (h - 0x3ff00000u < 0x01500000u) {  // 1 <= s < 2^21
    int64_t j;
    double w;
    floor_frac64(s, j, w);
    c = (int32_t)j;
    f = to_f32(w);
    if (f >= 1.0f) {
      f = 0.0f;
      c += 1;
    }
  } else {
    double fl = floor(s);
    f = (float)__dsub_rn(s, fl);
    if (f >= 1.0f) {
      f = 0.0f;
      fl += 1.0;
    }
    c = (int32_t)fl;
  }
  cell = c;
  frac = f;
}
__device__ __forceinline__ double join_x(int32_t cell, float frac, double dx) {
  return __dmul_rn(__dadd_rn(i32_to_f64(cell), to_f64(frac)), dx);
}

// The cell size of a particle: one problem's, or its ensemble's.
struct OneCell {
  double v;
  __device__ __forceinline__ double operator()(int64_t, int&) const { return v; }
};
template <bool INV>
struct EnsCell {
  const EnsDev* ens;
  int32_t n_ens;
  int64_t off;
  // e: the caller's last ensemble (its particles' indexes increase)
  __device__ __forceinline__ double operator()(int64_t i, int& e) const {
    i += off;
    if (e < 0 || i >= ens[e].first + ens[e].count) {
      int lo = e < 0 ? 0 : e, hi = n_ens - 1;  // last one that starts at or before i
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (ens[mid].first <= i) lo = mid; else hi = mid - 1;
      }
      e = lo;
    }
    return INV ? ens[e].inv_dx64 : ens[e].dx;
  }
};

constexpr int kConvThreads = 256;

// VEC: every array starts on a boundary of two elements.
template <bool VEC, class CELL>
__global__ void __launch_bounds__(kConvThreads) to_mixed_kernel(const double* x, const double* px, const double* py,
                                                                const double* pz, MixedStore m, CELL cell, int64_t n) {
  int e = -1;
  for (int64_t i = 2 * (blockIdx.x * (int64_t)kConvThreads + threadIdx.x); i < n;
       i += 2 * (int64_t)gridDim.x * kConvThreads) {
    const bool two = i + 1 < n;
    int2 c;
    float2 f;
    if (VEC && two) {
      const double2 X = __ldcs(reinterpret_cast<const double2*>(x + i));
      const double2 A = __ldcs(reinterpret_cast<const double2*>(px + i));
      const double2 B = __ldcs(reinterpret_cast<const double2*>(py + i));
      const double2 C = __ldcs(reinterpret_cast<const double2*>(pz + i));
      split_x(X.x, cell(i, e), c.x, f.x);
      split_x(X.y, cell(i + 1, e), c.y, f.y);
      *reinterpret_cast<int2*>(m.cell + i) = c;
      *reinterpret_cast<float2*>(m.frac + i) = f;
      *reinterpret_cast<float2*>(m.px + i) = make_float2(to_f32(A.x), to_f32(A.y));
      *reinterpret_cast<float2*>(m.py + i) = make_float2(to_f32(B.x), to_f32(B.y));
      *reinterpret_cast<float2*>(m.pz + i) = make_float2(to_f32(C.x), to_f32(C.y));
    } else {
      for (int64_t q = i; q < (two ? i + 2 : i + 1); ++q) {
        split_x(x[q], cell(q, e), c.x, f.x);
        m.cell[q] = c.x;
        m.frac[q] = f.x;
        m.px[q] = to_f32(px[q]);
        m.py[q] = to_f32(py[q]);
        m.pz[q] = to_f32(pz[q]);
      }
    }
  }
}

template <bool VEC, class CELL>
__global__ void __launch_bounds__(kConvThreads) from_mixed_kernel(MixedStore m, double* x, double* px, double* py,
                                                                  double* pz, CELL cell, int64_t n) {
  int e = -1;
  for (int64_t i = 2 * (blockIdx.x * (int64_t)kConvThreads + threadIdx.x); i < n;
       i += 2 * (int64_t)gridDim.x * kConvThreads) {
    const bool two = i + 1 < n;
    if (VEC && two) {
      if (x) {
        const int2 c = *reinterpret_cast<const int2*>(m.cell + i);
        const float2 f = *reinterpret_cast<const float2*>(m.frac + i);
        const double d0 = cell(i, e), d1 = cell(i + 1, e);
        __stcs(reinterpret_cast<double2*>(x + i), make_double2(join_x(c.x, f.x, d0), join_x(c.y, f.y, d1)));
      }
      auto copy = [&](double* to, const float* from) {
        const float2 v = *reinterpret_cast<const float2*>(from + i);
        __stcs(reinterpret_cast<double2*>(to + i), make_double2(to_f64(v.x), to_f64(v.y)));
      };
      if (px) copy(px, m.px);
      if (py) copy(py, m.py);
      if (pz) copy(pz, m.pz);
    } else {
      for (int64_t q = i; q < (two ? i + 2 : i + 1); ++q) {
        if (x) x[q] = join_x(m.cell[q], m.frac[q], cell(q, e));
        if (px) px[q] = to_f64(m.px[q]);
        if (py) py[q] = to_f64(m.py[q]);
        if (pz) pz[q] = to_f64(m.pz[q]);
      }
    }
  }
}

int conv_blocks(int64_t n) {
  const int64_t want = (n + 2 * kConvThreads - 1) / (2 * kConvThreads);
  return (int)(want < 1 ? 1 : want < 152 * 32 ? want : 152 * 32);
}
bool pairs(const MixedStore& m, const void* a, const void* b, const void* c, const void* d) {
  return (((uintptr_t)m.cell | (uintptr_t)m.frac | (uintptr_t)m.px | (uintptr_t)m.py | (uintptr_t)m.pz) & 7) == 0 &&
         (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d) & 15) == 0;
}
template <class CELL>
cudaError_t to_mixed(const double* x, const double* px, const double* py, const double* pz, const MixedStore& m,
                     const CELL& cell, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (pairs(m, x, px, py, pz))
    to_mixed_kernel<true><<<conv_blocks(n), kConvThreads, 0, s>>>(x, px, py, pz, m, cell, n);
  else
    to_mixed_kernel<false><<<conv_blocks(n), kConvThreads, 0, s>>>(x, px, py, pz, m, cell, n);
  return cudaGetLastError();
}
template <class CELL>
cudaError_t from_mixed(const MixedStore& m, double* x, double* px, double* py, double* pz, const CELL& cell,
                       int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (pairs(m, x, px, py, pz))
    from_mixed_kernel<true><<<conv_blocks(n), kConvThreads, 0, s>>>(m, x, px, py, pz, cell, n);
  else
    from_mixed_kernel<false><<<conv_blocks(n), kConvThreads, 0, s>>>(m, x, px, py, pz, cell, n);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_to_mixed(const double* x, const double* px, const double* py, const double* pz,
                            const MixedStore& m, double inv_dx, int64_t n, cudaStream_t s) {
  return to_mixed(x, px, py, pz, m, OneCell{inv_dx}, n, s);
}
cudaError_t launch_from_mixed(const MixedStore& m, double* x, double* px, double* py, double* pz, double dx,
                              int64_t n, cudaStream_t s) {
  return from_mixed(m, x, px, py, pz, OneCell{dx}, n, s);
}
cudaError_t launch_to_mixed_batch(const double* x, const double* px, const double* py, const double* pz,
                                  const MixedStore& m, const EnsDev* ens, int32_t n_ens, int64_t off, int64_t n,
                                  cudaStream_t s) {
  return to_mixed(x, px, py, pz, m, EnsCell<true>{ens, n_ens, off}, n, s);
}
cudaError_t launch_from_mixed_batch(const MixedStore& m, double* x, double* px, double* py, double* pz,
                                    const EnsDev* ens, int32_t n_ens, int64_t n, cudaStream_t s) {
  return from_mixed(m, x, px, py, pz, EnsCell<false>{ens, n_ens, 0}, n, s);
}

}  // namespace pic
