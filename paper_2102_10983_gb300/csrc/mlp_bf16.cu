// Learned sub-cycle-count predictor: MLP 6 -> 64 -> 64 -> 8 (ReLU, softmax
// cross-entropy over k = 0..7), BF16 operands with FP32 accumulation.
//
// Not part of the paper: it only predicts, per particle, the exponent k the
// criterion of Sec. IV will choose at the next macro step, so that the push can
// bin work before launch.  The criterion still decides every sub-step.
//
// Row-vector convention: h1 = relu(phi W1^T + b1), h2 = relu(h1 W2^T + b2),
// z = h2 W3^T + b3; W_l is (out, in).  phi = (asinh|E|, asinh|B|, asinh p_x,
// asinh p_y, asinh p_z, log gamma).
//
// Training (this file): warp-level mma.sync m16n8k16 (BF16 in, FP32
// accumulate), 16 samples per warp tile.  A layer's accumulator fragments are,
// after bias and ReLU, exactly the next layer's A fragments, so hidden
// activations never leave registers in the forward pass.  Backward: dz on the
// CUDA cores, dh2 = dz W3 and dh1 = da2 W2 on the tensor cores, and so the
// weight gradients (batch reductions) from BF16-rounded operands with FP32
// accumulation.  Inference (mlp_tc.cu) runs on tcgen05 with
// TMEM accumulators.
#include <cuda_bf16.h>
#include <math.h>

#include "pic_internal.h"
#include "push_device.cuh"

namespace pic {

namespace {

constexpr int kH = 64, kIn = 6, kOut = 8, kK1 = 16;
// Row strides (BF16 elements) of the weight tiles in shared memory, padded so
// that the eight rows a warp's B-fragment loads touch at once fall in distinct
// banks (a 64-element row is 128 bytes: unpadded, those eight loads conflict).
constexpr int kS1 = 24, kS2 = 72;

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Weights as the kernels read them from shared memory (BF16):
//   W1p [64][16] (cols 6..15 zero), W2 [64][64], W2T [64][64], W3 [8][64] (rows at the
//   padded strides kS1, kS2), W3T [64][8],
// and the FP32 biases.
struct SmemW {
  __nv_bfloat16 W1p[kH * kS1];
  __nv_bfloat16 W2[kH * kS2];
  __nv_bfloat16 W2T[kH * kS2];
  __nv_bfloat16 W3[kOut * kS2];
  __nv_bfloat16 W3T[kH * kOut];
  float b1[kH], b2[kH], b3[kOut];
};

__device__ void load_weights(SmemW& s, const float* P) {
  // packed FP32 master: W1[64][6] b1[64] W2[64][64] b2[64] W3[8][64] b3[8]
  const float* W1 = P;
  const float* b1 = W1 + kH * kIn;
  const float* W2 = b1 + kH;
  const float* b2 = W2 + kH * kH;
  const float* W3 = b2 + kH;
  const float* b3 = W3 + kOut * kH;
  for (int e = threadIdx.x; e < kH * kK1; e += blockDim.x) {
    const int o = e / kK1, i = e % kK1;
    s.W1p[o * kS1 + i] = __float2bfloat16_rn(i < kIn ? W1[o * kIn + i] : 0.0f);
  }
  for (int e = threadIdx.x; e < kH * kH; e += blockDim.x) {
    const int o = e / kH, i = e % kH;
    s.W2[o * kS2 + i] = __float2bfloat16_rn(W2[e]);
    s.W2T[i * kS2 + o] = __float2bfloat16_rn(W2[e]);
  }
  for (int e = threadIdx.x; e < kOut * kH; e += blockDim.x) {
    const int o = e / kH, i = e % kH;
    s.W3[o * kS2 + i] = __float2bfloat16_rn(W3[e]);
    s.W3T[i * kOut + o] = __float2bfloat16_rn(W3[e]);
  }
  for (int e = threadIdx.x; e < kH; e += blockDim.x) {
    s.b1[e] = b1[e];
    s.b2[e] = b2[e];
  }
  if (threadIdx.x < kOut) s.b3[threadIdx.x] = b3[threadIdx.x];
}

__device__ __forceinline__ uint32_t ld32(const __nv_bfloat16* p) {
  return *reinterpret_cast<const uint32_t*>(p);
}
// Forward of one 16-row tile.  a1: layer-1 input fragment.  Outputs the
// pre-activations (kept for the backward pass) and the logits.
struct Fwd {
  float acc1[8][4];  // a1 = phi W1^T + b1 (pre-ReLU)
  float acc2[8][4];  // a2
  float z[4];        // logits, rows (g, g+8), cols 2t, 2t+1
};

__device__ __forceinline__ void forward_tile(const SmemW& s, const uint32_t (&a1)[4], Fwd& f) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const float bl = s.b1[8 * nt + 2 * t], bh = s.b1[8 * nt + 2 * t + 1];
    f.acc1[nt][0] = bl; f.acc1[nt][1] = bh; f.acc1[nt][2] = bl; f.acc1[nt][3] = bh;
    const __nv_bfloat16* w = s.W1p + (8 * nt + g) * kS1;
    mma16816(f.acc1[nt], a1, ld32(w + 2 * t), ld32(w + 2 * t + 8));
  }
  uint32_t a2[4][4];
#pragma unroll
  for (int kc = 0; kc < 4; ++kc) {
    a2[kc][0] = pack2(fmaxf(f.acc1[2 * kc][0], 0.f), fmaxf(f.acc1[2 * kc][1], 0.f));
    a2[kc][1] = pack2(fmaxf(f.acc1[2 * kc][2], 0.f), fmaxf(f.acc1[2 * kc][3], 0.f));
    a2[kc][2] = pack2(fmaxf(f.acc1[2 * kc + 1][0], 0.f), fmaxf(f.acc1[2 * kc + 1][1], 0.f));
    a2[kc][3] = pack2(fmaxf(f.acc1[2 * kc + 1][2], 0.f), fmaxf(f.acc1[2 * kc + 1][3], 0.f));
  }
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const float bl = s.b2[8 * nt + 2 * t], bh = s.b2[8 * nt + 2 * t + 1];
    f.acc2[nt][0] = bl; f.acc2[nt][1] = bh; f.acc2[nt][2] = bl; f.acc2[nt][3] = bh;
    const __nv_bfloat16* w = s.W2 + (8 * nt + g) * kS2;
#pragma unroll
    for (int kc = 0; kc < 4; ++kc)
      mma16816(f.acc2[nt], a2[kc], ld32(w + 16 * kc + 2 * t), ld32(w + 16 * kc + 2 * t + 8));
  }
  uint32_t a3[4][4];
#pragma unroll
  for (int kc = 0; kc < 4; ++kc) {
    a3[kc][0] = pack2(fmaxf(f.acc2[2 * kc][0], 0.f), fmaxf(f.acc2[2 * kc][1], 0.f));
    a3[kc][1] = pack2(fmaxf(f.acc2[2 * kc][2], 0.f), fmaxf(f.acc2[2 * kc][3], 0.f));
    a3[kc][2] = pack2(fmaxf(f.acc2[2 * kc + 1][0], 0.f), fmaxf(f.acc2[2 * kc + 1][1], 0.f));
    a3[kc][3] = pack2(fmaxf(f.acc2[2 * kc + 1][2], 0.f), fmaxf(f.acc2[2 * kc + 1][3], 0.f));
  }
  const float bl = s.b3[2 * t], bh = s.b3[2 * t + 1];
  f.z[0] = bl; f.z[1] = bh; f.z[2] = bl; f.z[3] = bh;
  const __nv_bfloat16* w = s.W3 + g * kS2;
#pragma unroll
  for (int kc = 0; kc < 4; ++kc)
    mma16816(f.z, a3[kc], ld32(w + 16 * kc + 2 * t), ld32(w + 16 * kc + 2 * t + 8));
}

// Layer-1 fragment from an FP32 feature array phi[n][6] (rows >= n are zero).
__device__ __forceinline__ void phi_fragment(const float* phi, int64_t n, int64_t base,
                                             uint32_t (&a1)[4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  if (t < 3) {
    if (base + g < n) { v[0] = phi[(base + g) * kIn + 2 * t]; v[1] = phi[(base + g) * kIn + 2 * t + 1]; }
    if (base + g + 8 < n) { v[2] = phi[(base + g + 8) * kIn + 2 * t]; v[3] = phi[(base + g + 8) * kIn + 2 * t + 1]; }
  }
  a1[0] = pack2(v[0], v[1]);
  a1[1] = pack2(v[2], v[3]);
  a1[2] = 0u;
  a1[3] = 0u;
}

// Per-block gradients, same packed order as the parameters.
constexpr int kNParams = kH * kIn + kH + kH * kH + kH + kOut * kH + kOut;
constexpr int kOffB1 = kH * kIn, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH, kOffW3 = kOffB2 + kH,
              kOffB3 = kOffW3 + kOut * kH;
// A block's partial result: the gradients, then the loss.
constexpr int kPartial = kNParams + 8;
constexpr int kGradWarps = 4, kGradRows = 16 * kGradWarps;  // samples per block and pass
constexpr int kSN = 24;                                     // row stride of the 8-column operands

// The BF16 operands of the weight gradients of a block's samples, rows padded
// so that the eight rows of a transposing matrix load fall in distinct banks.
// X: the six features, a one (whose column of a product is the bias gradient)
// and a zero.
struct GradStage {
  __nv_bfloat16 h1[kGradRows][kS2], h2[kGradRows][kS2], da1[kGradRows][kS2], da2[kGradRows][kS2];
  __nv_bfloat16 dz[kGradRows][kSN], X[kGradRows][kSN];
  float loss[kGradWarps];
};

__device__ __forceinline__ void st2(__nv_bfloat16* p, float lo, float hi) {
  *reinterpret_cast<uint32_t*>(p) = pack2(lo, hi);
}
// Four (two) 8 x 8 matrices of 16-bit elements, transposed on the way: lane l
// gives the address of row l mod 8 of matrix l / 8.
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_addr(p))
               : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(smem_addr(p))
               : "memory");
}

}  // namespace

// ---------------------------------------------------------------- training (gradients)

// Forward and backward pass, and this block's share of the gradients in
// part[block].  Each warp takes 16 samples through the network; then the
// weight gradients, which are contractions over the samples (da2^T h1 and so
// on), run on the tensor cores too, the block's 64 samples at a time: warp w
// forms rows 16 w .. 16 w + 15 of each, its operands by transposing matrix
// loads from the staged tiles, and keeps its sums in registers over all of the
// block's samples.  The tensor cores truncate where they add into an
// accumulator, a bias that grows with the number of additions: so they sum the
// 64 samples of a pass from zero, and the passes' sums are added in FP32, to
// nearest (a batch of 1,048,576, against 64-bit sums of the same operands:
// relative error 2.0e-5 if the accumulators run on, 5e-8 so, 1.8e-7 on the FP32
// pipes).
// (On the FP32 pipes -- 16 products per element and shared atomics between the
// warps, then an atomic per block and parameter -- a batch of 8,192 took 30 us;
// this kernel 7.3 us and mlp_finish_kernel 3.2 us.)
__global__ void __launch_bounds__(32 * kGradWarps) mlp_grad_kernel(const float* P, const float* phi,
                                                                   const uint8_t* label, int64_t n,
                                                                   float inv_batch, float* part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemW& s = *reinterpret_cast<SmemW*>(smem_raw);
  GradStage& S = *reinterpret_cast<GradStage*>(smem_raw + ((sizeof(SmemW) + 15) & ~(size_t)15));
  load_weights(s, P);
  __syncthreads();
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, warp = threadIdx.x >> 5;
  const int r0w = 16 * warp;  // this warp's rows of the stage, and of every gradient
  // the gradients of a pass, and of the passes before it: W2 in 0 .. 7, then W1,
  // W3, b2 and b3 (W1's and b2's column 6: the bias gradients)
  float g4[12][4], sum[12][4];
#pragma unroll
  for (int r = 0; r < 12; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) g4[r][q] = sum[r][q] = 0.f;
  float (&gW1)[4] = g4[8], (&gW3)[4] = g4[9], (&gB2)[4] = g4[10], (&gB3)[4] = g4[11];
  auto add_pass = [&]() {
#pragma unroll
    for (int r = 0; r < 12; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        sum[r][q] = __fadd_rn(sum[r][q], g4[r][q]);
        g4[r][q] = 0.f;
      }
  };
  float my_loss = 0.f;
  const int64_t blocks = (n + kGradRows - 1) / kGradRows;
  for (int64_t blk = blockIdx.x; blk < blocks; blk += gridDim.x) {
    if (blk != blockIdx.x) add_pass();
    const int64_t base = blk * kGradRows + r0w;
    uint32_t a1[4];
    phi_fragment(phi, n, base, a1);
    Fwd f;
    forward_tile(s, a1, f);
    const bool r0 = base + g < n, r1 = base + g + 8 < n;
    // softmax cross-entropy; dz = (softmax - onehot) / batch
    float m0 = fmaxf(f.z[0], f.z[1]), m1 = fmaxf(f.z[2], f.z[3]);
    for (int o = 1; o <= 2; o <<= 1) {
      m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, o));
      m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    }
    const float e0 = __expf(f.z[0] - m0), e1 = __expf(f.z[1] - m0);
    const float e2 = __expf(f.z[2] - m1), e3 = __expf(f.z[3] - m1);
    float s0 = e0 + e1, s1 = e2 + e3;
    for (int o = 1; o <= 2; o <<= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    const int y0 = r0 ? label[base + g] : -1, y1 = r1 ? label[base + g + 8] : -1;
    float dz[4];
    dz[0] = r0 ? (e0 / s0 - (y0 == 2 * t ? 1.f : 0.f)) * inv_batch : 0.f;
    dz[1] = r0 ? (e1 / s0 - (y0 == 2 * t + 1 ? 1.f : 0.f)) * inv_batch : 0.f;
    dz[2] = r1 ? (e2 / s1 - (y1 == 2 * t ? 1.f : 0.f)) * inv_batch : 0.f;
    dz[3] = r1 ? (e3 / s1 - (y1 == 2 * t + 1 ? 1.f : 0.f)) * inv_batch : 0.f;
    if (r0 && (y0 >> 1) == t) my_loss += logf(s0) - ((y0 & 1 ? f.z[1] : f.z[0]) - m0);
    if (r1 && (y1 >> 1) == t) my_loss += logf(s1) - ((y1 & 1 ? f.z[3] : f.z[2]) - m1);
    // dh2 = dz W3 (K = 8 classes, padded to 16): B[k][n] = W3[k][n] = W3T[n][k]
    uint32_t adz[4] = {pack2(dz[0], dz[1]), pack2(dz[2], dz[3]), 0u, 0u};
    float dh2[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      dh2[nt][0] = dh2[nt][1] = dh2[nt][2] = dh2[nt][3] = 0.f;
      mma16816(dh2[nt], adz, ld32(s.W3T + (8 * nt + g) * kOut + 2 * t), 0u);
    }
    // da2 = dh2 * (a2 > 0); dh1 = da2 W2: B[k][n] = W2[k][n] = W2T[n][k]
    uint32_t ada2[4][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
      for (int q = 0; q < 4; ++q) dh2[nt][q] = f.acc2[nt][q] > 0.f ? dh2[nt][q] : 0.f;
      ada2[nt >> 1][2 * (nt & 1)] = pack2(dh2[nt][0], dh2[nt][1]);
      ada2[nt >> 1][2 * (nt & 1) + 1] = pack2(dh2[nt][2], dh2[nt][3]);
    }
    float dh1[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      dh1[nt][0] = dh1[nt][1] = dh1[nt][2] = dh1[nt][3] = 0.f;
      const __nv_bfloat16* w = s.W2T + (8 * nt + g) * kS2;
#pragma unroll
      for (int kc = 0; kc < 4; ++kc)
        mma16816(dh1[nt], ada2[kc], ld32(w + 16 * kc + 2 * t), ld32(w + 16 * kc + 2 * t + 8));
    }
    // stage the operands (BF16-rounded)
    __syncthreads();  // the block is done with the last pass's
    const int ra = r0w + g, rb = ra + 8;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const int c = 8 * nt + 2 * t;
      st2(&S.h1[ra][c], fmaxf(f.acc1[nt][0], 0.f), fmaxf(f.acc1[nt][1], 0.f));
      st2(&S.h1[rb][c], fmaxf(f.acc1[nt][2], 0.f), fmaxf(f.acc1[nt][3], 0.f));
      st2(&S.h2[ra][c], fmaxf(f.acc2[nt][0], 0.f), fmaxf(f.acc2[nt][1], 0.f));
      st2(&S.h2[rb][c], fmaxf(f.acc2[nt][2], 0.f), fmaxf(f.acc2[nt][3], 0.f));
      *reinterpret_cast<uint32_t*>(&S.da2[ra][c]) = ada2[nt >> 1][2 * (nt & 1)];
      *reinterpret_cast<uint32_t*>(&S.da2[rb][c]) = ada2[nt >> 1][2 * (nt & 1) + 1];
      st2(&S.da1[ra][c], f.acc1[nt][0] > 0.f ? dh1[nt][0] : 0.f, f.acc1[nt][1] > 0.f ? dh1[nt][1] : 0.f);
      st2(&S.da1[rb][c], f.acc1[nt][2] > 0.f ? dh1[nt][2] : 0.f, f.acc1[nt][3] > 0.f ? dh1[nt][3] : 0.f);
    }
    *reinterpret_cast<uint32_t*>(&S.dz[ra][2 * t]) = adz[0];
    *reinterpret_cast<uint32_t*>(&S.dz[rb][2 * t]) = adz[1];
    *reinterpret_cast<uint32_t*>(&S.X[ra][2 * t]) = t < 3 ? a1[0] : pack2(1.f, 0.f);
    *reinterpret_cast<uint32_t*>(&S.X[rb][2 * t]) = t < 3 ? a1[1] : pack2(1.f, 0.f);
    __syncthreads();
    // this warp's rows of the gradients, 16 samples at a time
    const int mr = lane & 7, m1b = (lane >> 3) & 1, m2b = lane >> 4;  // row and matrix of the loads
#pragma unroll 1
    for (int kc = 0; kc < kGradWarps; ++kc) {
      const int k0 = 16 * kc;
      uint32_t A[4], B[4], D[2], Xf[2];
      // A (16 x 16): matrices (rows 0-7, k 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15)
      auto a_of = [&](const __nv_bfloat16(&T)[kGradRows][kS2]) { ldsm4t(A, &T[k0 + 8 * m2b + mr][r0w + 8 * m1b]); };
      ldsm2t(D, &S.dz[k0 + 8 * m1b + mr][0]);
      ldsm2t(Xf, &S.X[k0 + 8 * m1b + mr][0]);
      a_of(S.da2);
      mma16816(gB2, A, Xf[0], Xf[1]);
#pragma unroll
      for (int nt = 0; nt < 8; nt += 2) {
        ldsm4t(B, &S.h1[k0 + 8 * m1b + mr][8 * (nt + m2b)]);
        mma16816(g4[nt], A, B[0], B[1]);
        mma16816(g4[nt + 1], A, B[2], B[3]);
      }
      a_of(S.da1);
      mma16816(gW1, A, Xf[0], Xf[1]);
      a_of(S.h2);
      mma16816(gW3, A, D[0], D[1]);  // transposed: rows = inputs, columns = classes
      if (warp == 0) {
        const uint32_t one = pack2(1.f, 1.f), ones[4] = {one, one, one, one};
        mma16816(gB3, ones, D[0], D[1]);
      }
    }
  }
  if (blocks > gridDim.x) {  // several passes
    add_pass();
#pragma unroll
    for (int r = 0; r < 12; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) g4[r][q] = sum[r][q];
  }
  float* out = part + (int64_t)blockIdx.x * kPartial;
  const int oa = r0w + g, ob = oa + 8;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const int c = 8 * nt + 2 * t;
    *reinterpret_cast<float2*>(out + kOffW2 + oa * kH + c) = make_float2(g4[nt][0], g4[nt][1]);
    *reinterpret_cast<float2*>(out + kOffW2 + ob * kH + c) = make_float2(g4[nt][2], g4[nt][3]);
  }
  if (t < 3) {
    *reinterpret_cast<float2*>(out + oa * kIn + 2 * t) = make_float2(gW1[0], gW1[1]);
    *reinterpret_cast<float2*>(out + ob * kIn + 2 * t) = make_float2(gW1[2], gW1[3]);
  } else {  // column 6: the ones
    out[kOffB1 + oa] = gW1[0];
    out[kOffB1 + ob] = gW1[2];
    out[kOffB2 + oa] = gB2[0];
    out[kOffB2 + ob] = gB2[2];
  }
  out[kOffW3 + (2 * t) * kH + oa] = gW3[0];
  out[kOffW3 + (2 * t + 1) * kH + oa] = gW3[1];
  out[kOffW3 + (2 * t) * kH + ob] = gW3[2];
  out[kOffW3 + (2 * t + 1) * kH + ob] = gW3[3];
  if (warp == 0 && g == 0) {
    out[kOffB3 + 2 * t] = gB3[0];
    out[kOffB3 + 2 * t + 1] = gB3[1];
  }
  for (int o = 16; o > 0; o >>= 1) my_loss += __shfl_xor_sync(0xffffffffu, my_loss, o);
  if (lane == 0) S.loss[warp] = my_loss;
  __syncthreads();
  if (threadIdx.x == 0) {
    float l = 0.f;
    for (int w = 0; w < kGradWarps; ++w) l += S.loss[w];
    out[kNParams] = l * inv_batch;
  }
}

// Sums the blocks' partial results, in the blocks' order: the gradients into G
// (G != nullptr), the loss into *loss (where the host reads it); with lr > 0
// also the Adam step on the FP32 master parameters.  Thirty-two parameters per
// block, eight threads each on an eighth of the partials.
__global__ void __launch_bounds__(256) mlp_finish_kernel(const float* part, int blocks, float* G, float* loss,
                                                         float* P, float* m1, float* m2, float lr, float beta1,
                                                         float beta2, float eps, float bc1, float bc2) {
  __shared__ float sum[8][33];
  const int e = blockIdx.x * 32 + (threadIdx.x & 31), slice = threadIdx.x >> 5;
  float g = 0.f;
  if (e <= kNParams)
    for (int b = slice; b < blocks; b += 8) g += part[(int64_t)b * kPartial + e];
  sum[slice][threadIdx.x & 31] = g;
  __syncthreads();
  if (slice > 0 || e > kNParams) return;
  for (int q = 1; q < 8; ++q) g += sum[q][threadIdx.x];
  if (e == kNParams) {
    *loss = g;
    return;
  }
  if (G) G[e] = g;
  if (lr > 0.f) {
    const float a = beta1 * m1[e] + (1.f - beta1) * g;
    const float b = beta2 * m2[e] + (1.f - beta2) * g * g;
    m1[e] = a;
    m2[e] = b;
    P[e] -= lr * (a / bc1) / (sqrtf(b / bc2) + eps);
  }
}

int mlp_param_count() { return kNParams; }

static int grad_blocks(int64_t n, int sm_count) {
  const int64_t want = (n + kGradRows - 1) / kGradRows, cap = sm_count > 0 ? sm_count : 152;
  return (int)(want < cap ? want : cap);
}
size_t mlp_partial_floats(int sm_count) { return (size_t)(sm_count > 0 ? sm_count : 152) * kPartial; }

cudaError_t launch_mlp_grad(const float* P, const float* phi, const uint8_t* label, int64_t n,
                            float* part, int sm_count, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const size_t smem = ((sizeof(SmemW) + 15) & ~(size_t)15) + sizeof(GradStage);
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  mlp_grad_kernel<<<grad_blocks(n, sm_count), 32 * kGradWarps, smem, s>>>(P, phi, label, n, 1.0f / (float)n,
                                                                          part);
  return cudaGetLastError();
}

cudaError_t launch_mlp_finish(const float* part, int64_t n, float* grad, float* loss, float* P, float* m1,
                              float* m2, float lr, int step, int sm_count, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
  mlp_finish_kernel<<<(kNParams + 32) / 32, 256, 0, s>>>(part, grad_blocks(n, sm_count), grad, loss, P, m1, m2,
                                                         lr, b1, b2, 1e-8f, bc1, bc2);
  return cudaGetLastError();
}

}  // namespace pic
