// Inference of the sub-cycle-count predictor on the 5th-generation tensor
// cores: tcgen05.mma with operands in shared memory and FP32 accumulators in
// tensor memory (TMEM).  Not part of the paper: the network only predicts the
// exponent k the criterion of Sec. IV will pick next, for binning; the
// criterion still decides every sub-step.
//
// One CTA per SM of five warpgroups, each with a tile of 128 particles of its
// own (thread = row = TMEM lane):
//   features: each thread forms one particle's phi (6 values, BF16, zero-
//     padded to K = 16) and stores it as its row of A1, in TMEM;
//   layer 1: one tcgen05.mma M=128 N=64 K=16, A1 x W1^T -> D;
//   epilogue 1: each warp reads its 32 TMEM lanes (rows) of D, adds b1, applies
//     ReLU, rounds to BF16 and stores A2 [128 x 64] in TMEM, over A1;
//   layer 2: four MMAs (K = 16 each) A2 x W2^T -> D; epilogue 2: b2, the same;
//   layer 3: four MMAs A2 x W3^T (N = 16, rows 8..15 of W3 zero) -> D;
//   epilogue 3: b3, argmax over the 8 classes (ties: the smaller k).
// What bounds it is the SM's shared-memory and L1 data path: with A1 and A2 in
// shared memory (128 threads per CTA, seven CTAs) its wavefronts per tile were
// 410 of epilogue loads (biases), 330 of stores, 380 of the MMAs' reads and 140
// of the particles' loads, 1,260 of the 1,280 clocks a tile took.  With A in
// TMEM the stores and the A part of the MMAs' reads are gone.  A tile needs 96
// TMEM columns (A 32, D 64), so five fit the SM's 512 and cover each other's
// chains (features, three MMA round trips, three epilogues).  8,388,608
// electrons, order 3: 277 us with A in shared memory, 264 here, 236 with the next
// tile's features formed during the first layer.
// One thread of the warpgroup issues the MMAs and commits them to the
// warpgroup's mbarrier, on which every warp waits itself (a bounded wait: on a
// give-up the warpgroup records it, marks the tile's predictions 0xFF, an
// invalid class, and stops); one barrier of the warpgroup comes ahead of each
// layer's MMAs, where rows that all its warps wrote are handed over.
//
// Shared-memory operands use the no-swizzle K-major layout of 8 x 16-byte
// core matrices: element (r, k) of an R x K tile sits at
// (r / 8) * (K / 8) * 128 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2 bytes;
// the descriptors give the step between core matrices along K (128 B) and
// along R ((K / 8) * 128 B).
#include <cuda_bf16.h>
#include <math.h>

#include "pic_internal.h"
#include "push_device.cuh"

namespace pic {
namespace {

constexpr int kTcRows = 128;  // particles per tile (MMA M)
constexpr int kTcGroups = 5;    // warpgroups per CTA, a tile each
constexpr int kTcThreads = kTcRows * kTcGroups;
constexpr int kTcH = 64, kTcIn = 6, kTcOut = 8;
// TMEM columns of a tile: A (BF16, two per 32-bit column), then D.
constexpr uint32_t kACols = 32, kTileCols = 96, kTmemCols = 512;
static_assert(kTcGroups * kTileCols <= kTmemCols, "the tiles' columns");

struct TcSmem {
  __align__(1024) unsigned char W1[kTcH * 16 * 2];    // [64 x 16]
  __align__(1024) unsigned char W2[kTcH * kTcH * 2];  // [64 x 64]
  __align__(1024) unsigned char W3[16 * kTcH * 2];    // [16 x 64], rows 8..15 zero
  float b1[kTcH], b2[kTcH], b3[kTcOut];
  __align__(8) uint64_t bar[kTcGroups];
  uint32_t tmem;
  int failed[kTcGroups][2];  // a wait of an even, an odd tile of the warpgroup gave up
};
// Reserved per CTA: more than half of an SM's shared memory, so that no second
// CTA waits there for the TMEM columns of the first.
constexpr size_t kTcSmemBytes = 116 * 1024;
static_assert(sizeof(TcSmem) + 1024 <= kTcSmemBytes, "the operands, with the slack for their alignment");
static_assert(2 * (kTcSmemBytes + 1024) > 228 * 1024, "one CTA per SM");

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t cm_off(int r, int k, int K) {
  return (uint32_t)(r >> 3) * (uint32_t)(K / 8) * 128u + (uint32_t)(k >> 3) * 128u +
         (uint32_t)(r & 7) * 16u + (uint32_t)(k & 7) * 2u;
}

// Shared-memory matrix descriptor (no swizzle): start address, the byte step
// between core matrices along K (leading) and along the rows (stride), and the
// descriptor version of this architecture.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t k_step, uint32_t r_step) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((k_step >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((r_step >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N and M.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// A in TMEM: row = lane, two consecutive K elements per 32-bit column.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                         int accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
               : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Bounded wait for phase `parity` of the barrier: false = gave up.
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 22); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(saddr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// Consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = __uint_as_float(r[q]);
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int q = 0; q < 32; ++q) v[q] = __uint_as_float(r[q]);
}

// 32-bit columns of this thread's TMEM lane from registers; tmem_st_wait: the
// stores have completed.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t bf2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// max(lo, 0), max(hi, 0) rounded to BF16 and packed (lo in the low half): the
// conversion's relu clamps a negative value to zero, in one instruction.
__device__ __forceinline__ uint32_t bf2_relu(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// Packed FP32 master parameters (W1[64][6] b1[64] W2[64][64] b2[64] W3[8][64]
// b3[8]) to BF16 operand tiles and FP32 biases.
__device__ void tc_load_weights(TcSmem& s, const float* P) {
  const float* W1 = P;
  const float* b1 = W1 + kTcH * kTcIn;
  const float* W2 = b1 + kTcH;
  const float* b2 = W2 + kTcH * kTcH;
  const float* W3 = b2 + kTcH;
  const float* b3 = W3 + kTcOut * kTcH;
  for (int e = threadIdx.x; e < kTcH * 16; e += blockDim.x) {
    const int o = e / 16, i = e % 16;
    *reinterpret_cast<__nv_bfloat16*>(s.W1 + cm_off(o, i, 16)) =
        __float2bfloat16_rn(i < kTcIn ? W1[o * kTcIn + i] : 0.0f);
  }
  for (int e = threadIdx.x; e < kTcH * kTcH; e += blockDim.x) {
    const int o = e / kTcH, i = e % kTcH;
    *reinterpret_cast<__nv_bfloat16*>(s.W2 + cm_off(o, i, kTcH)) = __float2bfloat16_rn(W2[e]);
  }
  for (int e = threadIdx.x; e < 16 * kTcH; e += blockDim.x) {
    const int o = e / kTcH, i = e % kTcH;
    *reinterpret_cast<__nv_bfloat16*>(s.W3 + cm_off(o, i, kTcH)) =
        __float2bfloat16_rn(o < kTcOut ? W3[o * kTcH + i] : 0.0f);
  }
  for (int e = threadIdx.x; e < kTcH; e += blockDim.x) {
    s.b1[e] = b1[e];
    s.b2[e] = b2[e];
  }
  if (threadIdx.x < kTcOut) s.b3[threadIdx.x] = b3[threadIdx.x];
}

// A thread's place: its warpgroup, and its row of the warpgroup's tile in TMEM.
struct TcPlace {
  int wg;
  uint32_t a, d;        // the tile's A and D columns (lane 0)
  uint32_t a_row, d_row;  // the same at this warp's lanes
  __device__ __forceinline__ TcPlace(const TcSmem& s) {
    wg = threadIdx.x >> 7;
    a = s.tmem + kTileCols * (uint32_t)wg;
    d = a + kACols;
    const uint32_t lane = (uint32_t)(threadIdx.x & 96) << 16;
    a_row = a + lane;
    d_row = d + lane;
  }
  __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, 128;" ::"r"(wg + 1) : "memory"); }
  __device__ __forceinline__ bool sync_or(bool v) const {
    uint32_t out;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, %2, 128, p;\n"
        " selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(out)
        : "r"((uint32_t)v), "r"(wg + 1)
        : "memory");
    return out != 0;
  }
};

// A particle's features in BF16.
struct TcRow {
  uint32_t w[3];
  bool fieldless;  // no field at the particle
  __device__ __forceinline__ void set(const float (&f)[6]) {
    w[0] = bf2(f[0], f[1]);
    w[1] = bf2(f[2], f[3]);
    w[2] = bf2(f[4], f[5]);
    fieldless = f[0] == 0.f && f[1] == 0.f;
  }
};

// This thread's row of A1 (columns 6..15 zero).
__device__ __forceinline__ void put_features(const TcPlace& at, const TcRow& row) {
  const uint32_t w[8] = {row.w[0], row.w[1], row.w[2], 0u, 0u, 0u, 0u, 0u};
  tmem_st8(at.a_row, w);
}

// Hidden layer epilogue: D's 64 columns of this thread's row, plus bias, ReLU,
// BF16, into its row of A2.
__device__ __forceinline__ void hidden_epilogue(const TcPlace& at, const float* bias) {
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    float v[32];
    tmem_ld32(at.d_row + (uint32_t)(32 * half), v);
    const float4* b4 = reinterpret_cast<const float4*>(bias + 32 * half);
    uint32_t w[16];
#pragma unroll
    for (int q = 0; q < 8; ++q) {  // bias in paired FP32 adds, ReLU in the BF16 conversion
      const float4 b = b4[q];
      const float2 lo = add2(make_float2(v[4 * q], v[4 * q + 1]), make_float2(b.x, b.y));
      const float2 hi = add2(make_float2(v[4 * q + 2], v[4 * q + 3]), make_float2(b.z, b.w));
      w[2 * q] = bf2_relu(lo.x, lo.y);
      w[2 * q + 1] = bf2_relu(hi.x, hi.y);
    }
    tmem_st16(at.a_row + (uint32_t)(16 * half), w);
  }
}

// This thread's wait for the layer just issued: false after a give-up, which
// the tile's flag then records.
__device__ __forceinline__ bool layer_wait(TcSmem& s, const TcPlace& at, uint32_t& ph, int odd) {
  uint64_t* bar = &s.bar[at.wg];
  const bool done = bar_wait(bar, ph) || bar_wait(bar, ph);  // gives up after two waits
  if (!done) s.failed[at.wg][odd] = 1;
  ph ^= 1u;
  __syncwarp();
  fence_after();
  return done;
}

// This warp's TMEM stores (its loads have waited) come before MMAs issued after
// the barrier that follows.
__device__ __forceinline__ void rows_ready() {
  tmem_st_wait();
  fence_before();
}

// The network on the warpgroup's tile, whose features (A1) all its threads have
// stored before a barrier: the first layer's MMA, then, once other work has
// been found for its latency, the rest.  Each thread returns its row's class
// (argmax, ties to the smaller k), or 0xFF after a give-up (a row depends on its
// own row of A only, so the others' classes stand).  Collective over the
// warpgroup.  ph: the mbarrier's phase; odd: the tile's flag.
__device__ __forceinline__ void tc_start(TcSmem& s, const TcPlace& at) {
  if ((threadIdx.x & 127) == 0) {
    mma_bf16(at.d, at.a, sdesc(saddr(s.W1), 128, 256), idesc_bf16(kTcRows, kTcH), 0);
    mma_commit(&s.bar[at.wg]);
  }
}
__device__ __forceinline__ int tc_finish(TcSmem& s, const TcPlace& at, uint32_t& ph, int odd) {
  const bool issuer = (threadIdx.x & 127) == 0;
  __syncwarp();
  bool ok = layer_wait(s, at, ph, odd);
  if (__all_sync(0xffffffffu, ok)) hidden_epilogue(at, s.b1);
  rows_ready();
  at.sync();
  fence_after();
  // layer 2
  if (issuer) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      mma_bf16(at.d, at.a + 8u * k, sdesc(saddr(s.W2) + 256u * k, 128, 1024), idesc_bf16(kTcRows, kTcH), k > 0);
    mma_commit(&s.bar[at.wg]);
  }
  __syncwarp();
  ok &= layer_wait(s, at, ph, odd);
  if (__all_sync(0xffffffffu, ok)) hidden_epilogue(at, s.b2);
  rows_ready();
  at.sync();
  fence_after();
  // layer 3
  if (issuer) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      mma_bf16(at.d, at.a + 8u * k, sdesc(saddr(s.W3) + 256u * k, 128, 1024), idesc_bf16(kTcRows, 16), k > 0);
    mma_commit(&s.bar[at.wg]);
  }
  __syncwarp();
  ok &= layer_wait(s, at, ph, odd);
  if (!__all_sync(0xffffffffu, ok)) return 0xFF;
  float z[8];
  tmem_ld8(at.d_row, z);
  float best = z[0] + s.b3[0];
  int cls = 0;
#pragma unroll
  for (int c = 1; c < kTcOut; ++c) {
    const float v = z[c] + s.b3[c];
    if (v > best) { best = v; cls = c; }
  }
  return cls;
}

__device__ __forceinline__ void tc_begin(TcSmem& s, const float* P) {
  tc_load_weights(s, P);
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&s.tmem)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int g = 0; g < kTcGroups; ++g) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&s.bar[g])));
      s.failed[g][0] = s.failed[g][1] = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
}

__device__ __forceinline__ void tc_end(TcSmem& s, DevStats* stats) {
  fence_before();
  __syncthreads();
  fence_after();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s.tmem), "r"(kTmemCols));
  if (threadIdx.x == 0 && stats) {
    int failed = 0;
    for (int g = 0; g < kTcGroups; ++g) failed |= s.failed[g][0] | s.failed[g][1];
    if (failed) atomicExch(&stats->error, 2);
  }
}

}  // namespace

// pic_predict: features of every particle after step a (a.featE / a.featB: its
// feature nodes; the same code as the features kernel) and the network's
// class, in one pass.
__global__ void __launch_bounds__(kTcThreads, 1) predict_tc_kernel(PushArgsMixed a, const float* Pm, uint8_t* pred,
                                                                int fieldless_zero) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  TcSmem& s = *reinterpret_cast<TcSmem*>(smem_raw + ((1024 - (saddr(smem_raw) & 1023)) & 1023));
  tc_begin(s, Pm);
  const TcPlace at(s);
  uint32_t ph = 0;
  const int row = threadIdx.x & 127;
  const int64_t n_tiles = (a.n + kTcRows - 1) / kTcRows, step = (int64_t)gridDim.x * kTcGroups;
  // a tile's features are formed while the first layer of the tile before it
  // runs, its particle loads issued one tile ahead of that
  auto input = [&](int64_t t) { return feature_input(a, t < n_tiles ? t * kTcRows + row : a.n); };
  auto form = [&](const FeatureInput& in) {
    float f[6];
    features_of(a, a.featE, a.featB, a.lo, a.hi, in, f);
    TcRow r;
    r.set(f);
    return r;
  };
  int64_t t = blockIdx.x + (int64_t)gridDim.x * at.wg;
  TcRow cur = form(input(t));
  FeatureInput nxt = input(t + step);
  for (int odd = 0; t < n_tiles; t += step, odd ^= 1) {
    const int64_t i = t * kTcRows + row;
    // no field at the particle: no rotation, the criterion takes k = 0
    const bool fieldless = fieldless_zero && cur.fieldless;
    __syncwarp();
    put_features(at, cur);
    rows_ready();
    const bool any = at.sync_or(!fieldless);  // uniform over the warpgroup
    fence_after();
    // the last tile's flag: set ahead of this barrier if at all, and not again
    // before the next tile's
    const bool stop = s.failed[at.wg][odd ^ 1];
    const bool run = any && !stop;
    if (run) tc_start(s, at);
    cur = form(nxt);
    nxt = input(t + 2 * step);
    int c = stop ? 0xFF : 0;
    if (run) c = tc_finish(s, at, ph, odd);
    if (fieldless && c != 0xFF) c = 0;
    if (i < a.n) pred[i] = (uint8_t)c;
    if (stop) break;
  }
  tc_end(s, a.stats);
}

// pic_mlp_infer: the network's class of n feature rows phi[n][6].
__global__ void __launch_bounds__(kTcThreads, 1) mlp_infer_tc_kernel(const float* Pm, const float* phi,
                                                                  int64_t n, uint8_t* pred) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  TcSmem& s = *reinterpret_cast<TcSmem*>(smem_raw + ((1024 - (saddr(smem_raw) & 1023)) & 1023));
  tc_begin(s, Pm);
  const TcPlace at(s);
  uint32_t ph = 0;
  const int64_t n_tiles = (n + kTcRows - 1) / kTcRows, step = (int64_t)gridDim.x * kTcGroups;
  int odd = 0;
  for (int64_t t = blockIdx.x + (int64_t)gridDim.x * at.wg; t < n_tiles; t += step, odd ^= 1) {
    const int64_t i = t * kTcRows + (threadIdx.x & 127);
    float f[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (i < n) {
#pragma unroll
      for (int q = 0; q < 6; ++q) f[q] = phi[i * 6 + q];
    }
    TcRow cur;
    cur.set(f);
    __syncwarp();
    put_features(at, cur);
    rows_ready();
    at.sync();
    fence_after();
    const bool stop = s.failed[at.wg][odd ^ 1];
    int c = 0xFF;
    if (!stop) {
      tc_start(s, at);
      c = tc_finish(s, at, ph, odd);
    }
    if (i < n) pred[i] = (uint8_t)c;
    if (stop) break;
  }
  tc_end(s, nullptr);
}

static int tc_grid(int64_t n, int sm_count) {
  const int64_t tiles = (n + kTcRows - 1) / kTcRows, sms = sm_count > 0 ? sm_count : 152;
  return (int)(tiles < sms ? tiles : sms);
}

template <class K>
static cudaError_t tc_configure(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmemBytes);
}

cudaError_t launch_predict_fused(const PushArgsMixed& a, int order, const float* P, uint8_t* pred,
                                 int sm_count, cudaStream_t st, bool fieldless_zero) {
  const int fz = fieldless_zero ? 1 : 0;
  if (a.n <= 0) return cudaSuccess;
  if (order < 1 || order > kMaxOrder) return cudaErrorInvalidValue;
  const int blocks = tc_grid(a.n, sm_count);
  cudaError_t e = tc_configure(predict_tc_kernel);
  if (e != cudaSuccess) return e;
  predict_tc_kernel<<<blocks, kTcThreads, kTcSmemBytes, st>>>(a, P, pred, fz);
  return cudaGetLastError();
}

cudaError_t launch_mlp_infer(const float* P, const float* phi, int64_t n, uint8_t* pred,
                             int sm_count, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  cudaError_t e = tc_configure(mlp_infer_tc_kernel);
  if (e != cudaSuccess) return e;
  mlp_infer_tc_kernel<<<tc_grid(n, sm_count), kTcThreads, kTcSmemBytes, s>>>(P, phi, n, pred);
  return cudaGetLastError();
}

}  // namespace pic
