// Learned selectivity surrogate (not in the paper; evaluated against exact ESC):
// an MLP 64 -> 128 -> ReLU -> 128 -> ReLU -> 1 predicting log10 selectivity
// from encoded predicate features.  Weights are used in bfloat16, biases
// and every accumulation are float32, the optimiser keeps float32 master
// weights (Adam).
//
// Flat parameter layout (ESC_MLP_PARAMS = 24961 floats): W1 [128][64], b1
// [128], W2 [128][128], b2 [128], w3 [128], b3.  The bfloat16 copy has the
// same layout (its bias entries are unused).
//
// The matrix products run on the tensor cores (tcgen05.mma, kind::f16): a
// block takes 128 samples at a time, accumulators and some operands sit in
// tensor memory.  Nothing loses precision on the way: features and weights are
// bfloat16 already, and a float32 operand (an activation, a gradient) is the
// sum of three bfloat16 numbers, its upper, middle and lower 8 significand
// bits, each multiplied by the other operand in full and accumulated in
// float32.  The gradient uses that w3 is bfloat16 and that the second layer's
// gradient is the outer product of dy and w3 under the ReLU mask:
//   d1 = dy (mask w3) W2,   gW2 = w3 (mask^T (dy z1)),   gb2 = w3 (mask^T dy),
//   gw3[j] = sum_k W2[j][k] (mask^T (dy z1))[j][k] + b2[j] (mask^T dy)[j],
// so that only z1, dy z1 and d1 need the split.  A factor of these sums over
// samples that is infinite or NaN would reach every unit, active or not (0
// times it is NaN), so such samples take part in them with zeros and are added
// by plain arithmetic (add_samples): only what they reach becomes non-finite.
//
// Shared-memory operands are rows of 128 bytes with 128-byte swizzle (the
// 16-byte chunk c of row r at c ^ (r % 8)), 64 columns a block of 16 KB per 128
// rows.  One such block is read along its rows (K-major) or across them
// (MN-major): X, z1 and the mask need no second copy for the transposed
// products.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cstring>
#include <mutex>
#include <string>

#include "esc_internal.h"
#include "esc_ptx.cuh"

namespace esc {

constexpr int kIn = 64, kH = 128;            // inputs, hidden width
constexpr int kTileS = 128;                  // samples per tile (rows of an accumulator: one tensor-memory lane each)
constexpr int kFwdThreads = 256;    // two warps per 32 lanes of tensor memory: half of the columns each
constexpr int kGradThreads = 512;   // four, a quarter of the columns each
constexpr int kW1 = 0, kB1 = kW1 + kH * kIn, kW2 = kB1 + kH, kB2 = kW2 + kH * kH, kW3 = kB2 + kH, kB3 = kW3 + kH;
constexpr int kParams = kB3 + 1;  // 24961
static_assert(kParams == ESC_MLP_PARAMS, "flat parameter layout");
static_assert(kW2 % 8 == 0, "16-byte chunks of W2");

constexpr uint32_t kBlock = 128 * 128;       // bytes of a 128-row operand block (64 columns)

// A wait on the tensor cores that gives up raises its status in a header of the
// block's own, in shared memory (these entry points do not synchronise and have
// no status to return): the outputs say so.  Later waits of the block then give
// up at once; it adds and writes nothing that depends on a wait, waits once more
// for its products in flight, and leaves NaN in the outputs it did not compute
// (y) or in loss_sum.  (With this and the search for infinite weights below, 1M
// predictions take 145.8 us, 147.5 before.)
#ifdef ESC_CHECKED
__device__ uint32_t g_mlp_give_up;   // test hook: each block's wait of this number gives up (0: none)
#endif

__device__ __forceinline__ float bf(const uint16_t v) {
  return __uint_as_float((uint32_t)v << 16);
}

// ------------------------------------------------------------------ tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols) {   // one warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t cols) {   // the same warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols));
}
__device__ __forceinline__ void tc_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Arrives on the barrier when this thread's earlier products are done.
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}
// Bounded wait for the phase of parity `parity`; `waits`: this block's so far.
__device__ __forceinline__ bool tc_wait(uint64_t *bar, uint32_t parity, ScratchHdr *hdr, uint32_t &waits) {
  const bool done = mbar_wait(bar, parity, hdr, kWaitLimitNs, true);
#ifdef ESC_CHECKED
  if (++waits == *(volatile const uint32_t *)&g_mlp_give_up) return false;   // (the products are done all the same)
#else
  (void)waits;
#endif
  return done;
}
// Instruction descriptor: float32 accumulators, bfloat16 operands, M = 128;
// transposed operands are MN-major.
__device__ __forceinline__ constexpr uint32_t idesc(uint32_t n, bool a_mn, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((n >> 3) << 17) |
         ((128u >> 4) << 24);
}
// Shared-memory operand descriptor, 128-byte swizzle: 8-row groups 1024 bytes
// apart, 64-column blocks (MN-major) kBlock apart.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
  return (uint64_t)((addr & 0x3ffffu) >> 4) | ((uint64_t)(kBlock >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t id, bool add) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
               "l"(a), "l"(b), "r"(id), "r"((uint32_t)add)
               : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t id, bool add) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
               "r"(a), "l"(b), "r"(id), "r"((uint32_t)add)
               : "memory");
}
// 32 columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
}
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(addr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

// Two floats as three pairs of bfloat16: x = hi + mid + lo exactly (a float's
// 24 significand bits, 8 in each; the low half holds a).  Infinities and NaN
// stay in hi, their other parts are 0: a truncated remainder has the sign of x,
// so that for x >= 0 a maximum with 0 clears a NaN.
template <bool NONNEG>
__device__ __forceinline__ float finite_part(float r) {
  return NONNEG ? fmaxf(r, 0.0f) : r == r ? r : 0.0f;
}
template <bool NONNEG>
__device__ __forceinline__ void split3(float2 x, uint32_t &hi, uint32_t &mid, uint32_t &lo) {
  // minus the upper half of a float's bits, as a float
  auto minus_hi = [](float v) { return __uint_as_float((__float_as_uint(v) & 0xffff0000u) ^ 0x80000000u); };
  float2 r = __fadd2_rn(x, make_float2(minus_hi(x.x), minus_hi(x.y)));
  r = make_float2(finite_part<NONNEG>(r.x), finite_part<NONNEG>(r.y));
  const float2 l = __fadd2_rn(r, make_float2(minus_hi(r.x), minus_hi(r.y)));
  hi = __byte_perm(__float_as_uint(x.x), __float_as_uint(x.y), 0x7632);
  mid = __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x7632);
  lo = __byte_perm(__float_as_uint(l.x), __float_as_uint(l.y), 0x7632);
}

// ------------------------------------------------------------------ operands
// 8 values (16 bytes); plain loads where the array is not 16-byte aligned.
__device__ __forceinline__ uint4 load8(const uint16_t *p, bool vec) {
  if (vec) return *reinterpret_cast<const uint4 *>(p);
  uint32_t w[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = (uint32_t)p[2 * k] | (uint32_t)p[2 * k + 1] << 16;
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ uint8_t *chunk(uint8_t *block, uint32_t row, uint32_t c) {
  return block + row * 128u + ((c ^ (row & 7u)) << 4);
}

struct MlpVectors {
  float b1[kH], b2[kH], w3[kH];
  float b3;
  uint32_t inf;   // forward kernel: an infinity in W2
  float pad[2];
};

// W1 (one block) and W2 (two) to shared memory, and the float32 vectors.  True
// when this thread has met an infinity in W2: the tensor cores would multiply
// it with z1's three parts, of which some are 0 (0 times it is NaN, and the
// unit would count as inactive), so that such weights take plain arithmetic.
// (A negative infinity makes its unit inactive either way.)
template <int NT>
__device__ __forceinline__ bool load_weights(uint8_t *w1, uint8_t *w2, MlpVectors &V, const uint16_t *wbf, const float *pf) {
  const bool vec = ((uintptr_t)wbf & 15u) == 0;
  for (uint32_t i = threadIdx.x; i < kH * kIn / 8; i += NT)
    *reinterpret_cast<uint4 *>(chunk(w1, i >> 3, i & 7u)) = load8(wbf + kW1 + 8 * i, vec);
  uint32_t most = 0;   // the largest of either half's values (as signed numbers: infinity, or a NaN, which is no matter)
  for (uint32_t i = threadIdx.x; i < kH * kH / 8; i += NT) {
    const uint4 w = load8(wbf + kW2 + 8 * i, vec);
    *reinterpret_cast<uint4 *>(chunk(w2 + ((i >> 3) & 1u) * kBlock, i >> 4, i & 7u)) = w;
    most = __vmaxs2(most, __vmaxs2(__vmaxs2(w.x, w.y), __vmaxs2(w.z, w.w)));
  }
  for (uint32_t i = threadIdx.x; i < kH; i += NT) {
    V.b1[i] = pf[kB1 + i];
    V.b2[i] = pf[kB2 + i];
    V.w3[i] = bf(wbf[kW3 + i]);
  }
  if (threadIdx.x == 0) {
    V.b3 = pf[kB3];
    V.inf = 0;
  }
  return (most & 0xffffu) >= 0x7f80u || (most >> 16) >= 0x7f80u;
}

// Value i of a row of an operand block (two blocks for 128 columns).
__device__ __forceinline__ float operand(const uint8_t *blocks, uint32_t row, uint32_t i) {
  const uint8_t *b = blocks + (i >> 6) * kBlock + row * 128u + ((((i >> 3) & 7u) ^ (row & 7u)) << 4) + 2u * (i & 7u);
  return bf(*reinterpret_cast<const uint16_t *>(b));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}
// relu of one unit of a layer by plain arithmetic: its row of weights times n values, and its bias.
template <typename V>
__device__ __forceinline__ float plain_unit(const uint8_t *w, uint32_t unit, float bias, uint32_t n, V value) {
  float a = bias;
#pragma unroll 8
  for (uint32_t k = 0; k < n; ++k) a = fmaf(operand(w, unit, k), value(k), a);
  return fmaxf(a, 0.0f);
}

// This thread's chunks of a tile's features (samples past the batch: 0).
template <int NT>
__device__ __forceinline__ void load_x(const uint16_t *x, uint64_t B, uint64_t s0, bool vec, uint4 (&r)[1024 / NT]) {
#pragma unroll
  for (int q = 0; q < 1024 / NT; ++q) {
    const uint32_t i = threadIdx.x + q * NT;
    const uint64_t s = s0 + (i >> 3);
    r[q] = s < B ? load8(x + s * kIn + 8 * (i & 7u), vec) : make_uint4(0, 0, 0, 0);
  }
}
template <int NT>
__device__ __forceinline__ void store_x(uint8_t *xb, const uint4 (&r)[1024 / NT]) {
#pragma unroll
  for (int q = 0; q < 1024 / NT; ++q) {
    const uint32_t i = threadIdx.x + q * NT;
    *reinterpret_cast<uint4 *>(chunk(xb, i >> 3, i & 7u)) = r[q];
  }
}

// ------------------------------------------------------------------ layers
// The tensor cores truncate each sum they write, a bias towards 0 that grows
// with the products added one after the other at full size.  So a float32
// operand's lower parts are multiplied first, and K is shared among two
// accumulators (forward) or four (gradient: 128 columns each), summed rounded
// to nearest here.  How far y is from its 64-bit value (2-norm; features and
// weights as in training, 31 to 1M samples): 1.5e-7 with the float32
// multiply-adds these products replace, 2.7e-7 with one accumulator, 1.1e-7
// with two, 1.0e-7 with four.  The gradient: 1.3e-7 to 3.2e-7 before, 0.8e-7
// to 2.6e-7 now (32 to 20,000 samples).
constexpr uint32_t kTmCols = 512;

// a1 = x W1^T: K = 64, 16 (32 bytes) per accumulator.
__device__ __forceinline__ void issue_layer1(uint32_t tm, uint64_t dx, uint64_t dw1) {
  for (uint32_t k = 0; k < 4; ++k) mma_ss(tm + 128 * k, dx + 2 * k, dw1 + 2 * k, idesc(kH, false, false), false);
}
// a2 = z1 W2^T: K = 128, 32 per accumulator; z1's parts (two blocks each) one
// after the other, the lower ones first.
__device__ __forceinline__ void issue_layer2(uint32_t tm, uint64_t dz, uint64_t dw2) {
  for (int p = 2; p >= 0; --p)
    for (uint32_t k = 0; k < 8; ++k) {
      const uint64_t at = (k >> 2) * (kBlock >> 4) + 2 * (k & 3u);
      mma_ss(tm + 128 * (k >> 1), dz + p * (2 * (kBlock >> 4)) + at, dw2 + at, idesc(kH, false, false), (k & 1u) || p < 2);
    }
}
// 32 columns of the sum of two or four accumulators.
__device__ __forceinline__ float2 as_float2(uint32_t a, uint32_t b) {
  return make_float2(__uint_as_float(a), __uint_as_float(b));
}
__device__ __forceinline__ void load_sum32(uint32_t addr, float2 (&v)[16]) {
  uint32_t a[32], b[32];
  tmem_ld32(addr, a);
  tmem_ld32(addr + 128, b);
  tc_wait_ld();
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = __fadd2_rn(as_float2(a[2 * k], a[2 * k + 1]), as_float2(b[2 * k], b[2 * k + 1]));
}
__device__ __forceinline__ void load_sum32x4(uint32_t addr, float2 (&v)[16]) {
  float2 w[16];
  load_sum32(addr, v);
  load_sum32(addr + 256, w);
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = __fadd2_rn(v[k], w[k]);
}
// relu(v + bias) of a pair of units
__device__ __forceinline__ float2 relu_bias(float2 v, const float *bias) {
  const float2 s = __fadd2_rn(v, *reinterpret_cast<const float2 *>(bias));
  return make_float2(fmaxf(s.x, 0.0f), fmaxf(s.y, 0.0f));
}

// 32 columns of a row of a split operand.
struct Split32 {
  uint32_t hi[16], mid[16], lo[16];
  template <bool NONNEG>
  __device__ __forceinline__ void make(const float2 *v) {
#pragma unroll
    for (int k = 0; k < 16; ++k) split3<NONNEG>(v[k], hi[k], mid[k], lo[k]);
  }
  // To chunks c .. c + 3 of the row; the parts' blocks lie `dist` apart.
  __device__ __forceinline__ void store(uint8_t *block, uint32_t dist, uint32_t c, uint32_t row) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint8_t *at = chunk(block, row, c + q);
      *reinterpret_cast<uint4 *>(at) = make_uint4(hi[4 * q], hi[4 * q + 1], hi[4 * q + 2], hi[4 * q + 3]);
      *reinterpret_cast<uint4 *>(at + dist) = make_uint4(mid[4 * q], mid[4 * q + 1], mid[4 * q + 2], mid[4 * q + 3]);
      *reinterpret_cast<uint4 *>(at + 2 * dist) = make_uint4(lo[4 * q], lo[4 * q + 1], lo[4 * q + 2], lo[4 * q + 3]);
    }
  }
};
// A quarter (32 units) of a row of R: three parts of two blocks.
template <bool NONNEG>
__device__ __forceinline__ void store_split32(uint8_t *r, uint32_t quarter, uint32_t row, const float2 *v) {
  Split32 s;
  s.make<NONNEG>(v);
  s.store(r + (quarter >> 1) * kBlock, 2 * kBlock, 4 * (quarter & 1u), row);
}

// ------------------------------------------------------------------ forward
// Two blocks per SM, so that one converts while the other's products run;
// tiles of 128 samples, two accumulators (tensor memory: 256 columns a block),
// one for each half of K.  Half of z1 is in shared memory at a time, over the
// features.  What bounds it: the instructions that split z1 and the waits
// between products and conversions (0.40 of the issue slots, 2 warps a
// scheduler and block).  Measured on 1M samples: 1822 us with one thread per
// hidden unit and float32 multiply-adds, 173 us with one block of 512 threads
// per SM and four accumulators, 148 us this way.
struct FwdSmem {
  static constexpr uint32_t w1 = 0, w2 = kBlock, z = 3 * kBlock, x = z, vec = 6 * kBlock, ypart = vec + sizeof(MlpVectors),
                            bar = ypart + 4 * kTileS, tmem = bar + 8, hdr = tmem + 8,
                            total = hdr + sizeof(ScratchHdr);
};
constexpr uint32_t kFwdCols = 256;

__global__ void __launch_bounds__(kFwdThreads, 2) mlp_forward_kernel(const uint16_t *x, uint64_t B, const uint16_t *wbf,
                                                                     const float *pf, float *y) {
  extern __shared__ __align__(1024) uint8_t sm[];
  MlpVectors &V = *reinterpret_cast<MlpVectors *>(sm + FwdSmem::vec);
  float *ypart = reinterpret_cast<float *>(sm + FwdSmem::ypart);
  uint64_t *bar = reinterpret_cast<uint64_t *>(sm + FwdSmem::bar);
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + FwdSmem::tmem);
  ScratchHdr *hdr = reinterpret_cast<ScratchHdr *>(sm + FwdSmem::hdr);
  uint8_t *Z = sm + FwdSmem::z;
  const uint32_t warp = threadIdx.x >> 5, half = warp >> 2, row = threadIdx.x & 127u;
  const bool vec = ((uintptr_t)x & 15u) == 0;
  uint4 xr[4];
  load_x<kFwdThreads>(x, B, (uint64_t)blockIdx.x * kTileS, vec, xr);
  if (warp == 0) tmem_alloc(slot, kFwdCols);
  if (threadIdx.x == 0) {
    *hdr = ScratchHdr{};
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const bool inf = load_weights<kFwdThreads>(sm + FwdSmem::w1, sm + FwdSmem::w2, V, wbf, pf);
  store_x<kFwdThreads>(sm + FwdSmem::x, xr);
  fence_proxy_async_smem();
  tc_before_sync();
  __syncthreads();
  if (inf) V.inf = 1;
  tc_after_sync();
  const uint32_t tm = *slot, lanes = tm + ((warp & 3u) << 21);   // + 32 * (warp % 4) lanes
  const uint64_t dw1 = sdesc(smem_addr(sm + FwdSmem::w1)), dw2 = sdesc(smem_addr(sm + FwdSmem::w2)),
                 dx = sdesc(smem_addr(sm + FwdSmem::x)), dz = sdesc(smem_addr(Z));
  constexpr uint32_t id = idesc(kH, false, false);
  uint32_t phase = 0, waits = 0;
  bool ok = true;   // after each barrier: no warp of the block has given up
  uint64_t s0 = (uint64_t)blockIdx.x * kTileS;
  for (; s0 < B; s0 += (uint64_t)gridDim.x * kTileS) {
    if (threadIdx.x == 0) {   // a1 = x W1^T: K = 64 in steps of 16 (32 bytes)
      for (uint32_t k = 0; k < 4; ++k) mma_ss(tm + 128 * (k >> 1), dx + 2 * k, dw1 + 2 * k, id, k & 1u);
      tc_commit(bar);
    }
    ok = tc_wait(bar, phase, hdr, waits);
    phase ^= 1u;
    tc_after_sync();
    float2 v[2][16];   // 32 units of either half of z1
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      load_sum32(lanes + 64 * h + 32 * half, v[h]);
#pragma unroll
      for (int k = 0; k < 16; ++k) v[h][k] = relu_bias(v[h][k], V.b1 + 64 * h + 32 * half + 2 * k);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      Split32 z;
      z.make<true>(v[h]);
      if (h == 1) {   // the first half's products have read Z
        ok = tc_wait(bar, phase, hdr, waits) && ok;
        phase ^= 1u;
      }
      z.store(Z, kBlock, 4 * half, row);
      if (h == 0) load_x<kFwdThreads>(x, B, s0 + (uint64_t)gridDim.x * kTileS, vec, xr);   // the next tile's features
      fence_proxy_async_smem();
      tc_before_sync();
      ok = __syncthreads_and(ok) != 0;
      if (!ok) break;
      if (threadIdx.x == 0) {   // a2 = z1 W2^T, the lower parts first
        tc_after_sync();
        for (int p = 2; p >= 0; --p)
          for (uint32_t k = 0; k < 4; ++k)
            mma_ss(tm + 128 * h, dz + p * (kBlock >> 4) + 2 * k, dw2 + h * (kBlock >> 4) + 2 * k, id, p < 2 || k > 0);
        tc_commit(bar);
      }
    }
    if (!ok) break;
    ok = tc_wait(bar, phase, hdr, waits);
    phase ^= 1u;
    tc_after_sync();
    store_x<kFwdThreads>(sm + FwdSmem::x, xr);
    fence_proxy_async_smem();
    float2 acc[2] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      load_sum32(lanes + 64 * half + 32 * h, v[h]);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int j = 64 * half + 32 * h + 2 * k;
        acc[k & 1] = __ffma2_rn(*reinterpret_cast<const float2 *>(V.w3 + j), relu_bias(v[h][k], V.b2 + j), acc[k & 1]);
      }
    }
    const float part = (acc[0].x + acc[0].y) + (acc[1].x + acc[1].y);
    if (half == 1) ypart[row] = part;
    tc_before_sync();
    ok = __syncthreads_and(ok) != 0;
    if (!ok) break;
    tc_after_sync();
    if (half == 0 && s0 + row < B) y[s0 + row] = part + ypart[row] + V.b3;   // (ypart is written again two barriers later)
  }
  if (!ok) {
    mbar_wait(bar, phase ^ 1u, hdr);   // the products in flight
    for (; s0 < B; s0 += (uint64_t)gridDim.x * kTileS)
      if (half == 0 && s0 + row < B) y[s0 + row] = __int_as_float(0x7fffffff);
  }
  // An infinity in W2: once more, sample by sample, thread = unit.  (Here, by way
  // of shared memory, as leaving before the loop cost it registers: 160 us
  // instead of 147.)
  __syncthreads();
  if (V.inf) {
    float *z1 = ypart, *red = reinterpret_cast<float *>(Z);
#pragma unroll 1
    for (uint64_t s0 = (uint64_t)blockIdx.x * kTileS; s0 < B; s0 += (uint64_t)gridDim.x * kTileS)
#pragma unroll 1
      for (uint64_t s = s0; s < B && s < s0 + kTileS; ++s) {
        if (half == 0) z1[row] = plain_unit(sm + FwdSmem::w1, row, V.b1[row], kIn, [&](uint32_t m) { return bf(x[s * kIn + m]); });
        __syncthreads();
        if (half == 0) {
          const float v = warp_sum(V.w3[row] * plain_unit(sm + FwdSmem::w2, row, V.b2[row], kH, [&](uint32_t k) { return z1[k]; }));
          if ((threadIdx.x & 31u) == 0) red[warp] = v;
        }
        __syncthreads();
        if (threadIdx.x == 0) y[s] = (red[0] + red[1]) + (red[2] + red[3]) + V.b3;
      }
    __syncthreads();
  }
  if (warp == 0) tmem_free(tm, kFwdCols);
}

// ------------------------------------------------------------------ gradient
// One block per SM, tiles of 128 samples; a tile's sums go to the global
// gradient by themselves.  Tensor memory: a1 and a2 take all 512 columns (four
// accumulators); then 0..255 two accumulators of d1 and 448 mask w3 (d1's left
// operand); when d1 has been read, 0, 128 and 256 three accumulators of gW2 /
// w3 (rows: units j), 384 gb2 / w3 and gb1 (products with the block E), 448
// gW1 (rows: units k).
// E (64 columns): columns 1..3 hold the three parts of dy while the mask is
// multiplied with it, column 0 then 1 for gb1.
// R holds z1, then dy z1, then d1, in three parts of two blocks.
// What bounds it at 4096 samples (32 tiles on 32 SMs): the chain of products
// and conversions of one tile, the loading of weights, and the fetching of
// instructions that each block runs once (20 us here by ncu, 24 with 256
// threads and twice the code, 43 before the tensor cores).  A training step
// (two fills, this, Adam): 4096 samples 50.5 -> 28.7 us, 20,000 162 -> 49, 65,536
// 417 -> 82.  Of that, the tests for infinities, NaN and waits that gave up are
// nothing that shows, 2 and 2 to 3 us.
constexpr uint32_t kTgB = 384, kTm = 448, kTgW1 = 448;
struct GradSmem {
  static constexpr uint32_t w1 = 0, w2 = kBlock, x = 3 * kBlock, e = 4 * kBlock, mask = 5 * kBlock, r = 7 * kBlock,
                            vec = 13 * kBlock, part = vec + sizeof(MlpVectors), bar = part + 4 * 4 * kTileS, tmem = bar + 32,
                            hdr = tmem + 16, bad = hdr + sizeof(ScratchHdr), bad_dy = bad + 16,
                            total = bad_dy + 4 * kTileS;
};

__device__ __forceinline__ void add4(float *p, float a, float b, float c, float d, bool vec) {
  if (vec) {
    asm volatile("red.global.add.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
  } else {
    atomicAdd(p, a);
    atomicAdd(p + 1, b);
    atomicAdd(p + 2, c);
    atomicAdd(p + 3, d);
  }
}

// Adds the gradient of the tile's rows in `bad` (128 bits) by plain arithmetic,
// unit by unit: samples with an infinity or NaN among the products' factors.
// Those are left out of the products, where 0 times such a factor would reach
// every unit, active or not.  `dy`: 2 / B times their residuals; with `target`
// (an infinity in W2, see load_weights) the residuals are found here, scale is
// 2 / B, and b3's gradient and the loss are added as well.  Four rows at a
// time, one for each 128 threads; `scratch`: shared memory.  The whole block
// calls, and meets at a barrier before it leaves.  A gradient of 4096 samples
// takes 35 us with one bad residual and 240 us with nothing but bad ones (19
// without; 39 either way before the tensor cores), 1M samples 748 us and 12.5 ms
// (740; 6.1 ms).
struct PlainRows {
  float z1[4][kH], d2[4][kH], d1[4][kH], red[4][4];
  uint8_t row[kTileS];
};
__device__ __noinline__ void add_samples(const uint8_t *sm, const MlpVectors &V, uint8_t *scratch, const uint32_t *bad,
                                         const float *dy, float scale, const float *target, float *grad, float *loss_sum) {
  const uint8_t *w1 = sm + GradSmem::w1, *w2 = sm + GradSmem::w2, *x = sm + GradSmem::x;
  PlainRows &P = *reinterpret_cast<PlainRows *>(scratch);
  const uint32_t j = threadIdx.x & 127u, q = threadIdx.x >> 7;
  uint32_t n = 0, before = 0;
  for (uint32_t k = 0; k < 4; ++k) {
    n += __popc(bad[k]);
    before += __popc(k < (j >> 5) ? bad[k] : k == (j >> 5) ? bad[k] & ((1u << (j & 31u)) - 1u) : 0u);
  }
  if (q == 0 && ((bad[j >> 5] >> (j & 31u)) & 1u)) P.row[before] = (uint8_t)j;
  __syncthreads();
  float g2[32], g1[16], gb1 = 0.0f, gb2 = 0.0f, gw3 = 0.0f;   // row j of W2's and W1's gradients, a quarter of each
#pragma unroll
  for (int k = 0; k < 32; ++k) g2[k] = 0.0f;
#pragma unroll
  for (int k = 0; k < 16; ++k) g1[k] = 0.0f;
#pragma unroll 1
  for (uint32_t i = 0; i < n; i += 4) {
    const uint32_t rows = min(4u, n - i), r = P.row[i + min(q, rows - 1)];
    const bool mine = q < rows;
    if (mine) P.z1[q][j] = plain_unit(w1, j, V.b1[j], kIn, [&](uint32_t m) { return operand(x, r, m); });
    __syncthreads();
    float z2 = 0.0f, dyr = 0.0f;
    if (mine) z2 = plain_unit(w2, j, V.b2[j], kH, [&](uint32_t k) { return P.z1[q][k]; });
    if (target) {
      const float v = warp_sum(V.w3[j] * z2);
      if ((j & 31u) == 0) P.red[q][j >> 5] = v;
      __syncthreads();
      if (mine) {
        const float e = (P.red[q][0] + P.red[q][1]) + (P.red[q][2] + P.red[q][3]) + V.b3 - target[r];
        dyr = e * scale;
        if (j == 0) {
          atomicAdd(&grad[kB3], dyr);
          atomicAdd(loss_sum, e * e);
        }
      }
    } else if (mine) {
      dyr = dy[r];
    }
    if (mine) {
      const float d = z2 > 0.0f ? dyr * V.w3[j] : 0.0f;
      P.d2[q][j] = d;
      gb2 += d;
      gw3 = fmaf(dyr, z2, gw3);
    }
    __syncthreads();
    for (uint32_t p = 0; p < rows; ++p) {
      const float d = P.d2[p][j];
#pragma unroll
      for (int k = 0; k < 32; ++k) g2[k] = fmaf(d, P.z1[p][32 * q + k], g2[k]);
    }
    if (mine) {
      float g = 0.0f;
#pragma unroll 8
      for (uint32_t k = 0; k < kH; ++k) g = fmaf(operand(w2, k, j), P.d2[q][k], g);
      g = P.z1[q][j] > 0.0f ? g : 0.0f;
      P.d1[q][j] = g;
      gb1 += g;
    }
    __syncthreads();
    for (uint32_t p = 0; p < rows; ++p) {
      const float d = P.d1[p][j];
      const uint32_t rp = P.row[i + p];
#pragma unroll
      for (int m = 0; m < 16; ++m) g1[m] = fmaf(d, operand(x, rp, 16 * q + m), g1[m]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < 32; ++k) atomicAdd(&grad[kW2 + j * kH + 32 * q + k], g2[k]);
#pragma unroll
  for (int m = 0; m < 16; ++m) atomicAdd(&grad[kW1 + j * kIn + 16 * q + m], g1[m]);
  atomicAdd(&grad[kB1 + j], gb1);
  atomicAdd(&grad[kB2 + j], gb2);
  atomicAdd(&grad[kW3 + j], gw3);
  __syncthreads();
}

__global__ void __launch_bounds__(kGradThreads, 1) mlp_grad_kernel(const uint16_t *x, const float *t, uint64_t B,
                                                                   const uint16_t *wbf, const float *pf, float *grad,
                                                                   float *loss_sum) {
  extern __shared__ __align__(1024) uint8_t sm[];
  MlpVectors &V = *reinterpret_cast<MlpVectors *>(sm + GradSmem::vec);
  float *part = reinterpret_cast<float *>(sm + GradSmem::part);
  uint64_t *bar = reinterpret_cast<uint64_t *>(sm + GradSmem::bar);   // [3]
  uint32_t *slot = reinterpret_cast<uint32_t *>(sm + GradSmem::tmem);
  ScratchHdr *hdr = reinterpret_cast<ScratchHdr *>(sm + GradSmem::hdr);
  uint8_t *R = sm + GradSmem::r, *E = sm + GradSmem::e, *mask = sm + GradSmem::mask;
  uint32_t *bad = reinterpret_cast<uint32_t *>(sm + GradSmem::bad);   // the tile's samples left to add_samples (bits)
  float *bad_dy = reinterpret_cast<float *>(sm + GradSmem::bad_dy);
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u, quarter = warp >> 2, row = threadIdx.x & 127u;
  const bool vec = ((uintptr_t)x & 15u) == 0, gvec = ((uintptr_t)grad & 15u) == 0;
  uint4 xr[2];
  load_x<kGradThreads>(x, B, (uint64_t)blockIdx.x * kTileS, vec, xr);
  if (warp == 0) tmem_alloc(slot, kTmCols);
  if (threadIdx.x == 0) {
    *hdr = ScratchHdr{};
    for (int k = 0; k < 3; ++k) mbar_init(&bar[k], 1);
    bad[0] = bad[1] = bad[2] = bad[3] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const bool inf = load_weights<kGradThreads>(sm + GradSmem::w1, sm + GradSmem::w2, V, wbf, pf);
#pragma unroll
  for (uint32_t c = 0; c < 2; ++c) *reinterpret_cast<uint4 *>(chunk(E, row, 2 * quarter + c)) = make_uint4(0, 0, 0, 0);
  store_x<kGradThreads>(sm + GradSmem::x, xr);
  fence_proxy_async_smem();
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  const uint32_t tm = *slot, lanes = tm + ((warp & 3u) << 21), mine = lanes + 32 * quarter;   // its 32 columns of 128
  const uint64_t dw1 = sdesc(smem_addr(sm + GradSmem::w1)), dw2 = sdesc(smem_addr(sm + GradSmem::w2)),
                 dx = sdesc(smem_addr(sm + GradSmem::x)), de = sdesc(smem_addr(E)), dm = sdesc(smem_addr(mask)),
                 dr = sdesc(smem_addr(R));
  constexpr uint32_t kPart = 2 * (kBlock >> 4);   // descriptor distance of two parts of R
  constexpr uint32_t kRows16 = 2048 >> 4;         // of 16 rows (MN-major: a step of K)
  uint32_t ph0 = 0, ph1 = 0, waits = 0;
  // No warp of the block has given up (after the two barriers below that agree on
  // it, before the tile's first and last additions).
  bool ok = true;
  float lsum = 0.0f, gb3 = 0.0f;
  const float inv_b = 2.0f / (float)B;
  for (uint64_t s0 = (uint64_t)blockIdx.x * kTileS; s0 < B; s0 += (uint64_t)gridDim.x * kTileS) {
    if (threadIdx.x == 0) {
      issue_layer1(tm, dx, dw1);
      tc_commit(&bar[0]);
    }
    const float target = s0 + row < B ? t[s0 + row] : 0.0f;
    ok = tc_wait(&bar[0], ph0, hdr, waits);
    ph0 ^= 1u;
    tc_after_sync();
    float2 z1[16], v[16];
    load_sum32x4(mine, v);
#pragma unroll
    for (int k = 0; k < 16; ++k) z1[k] = relu_bias(v[k], V.b1 + 32 * quarter + 2 * k);
    store_split32<true>(R, quarter, row, z1);
    fence_proxy_async_smem();
    tc_before_sync();
    __syncthreads();
    if (threadIdx.x == 0) {
      tc_after_sync();
      issue_layer2(tm, dr, dw2);
      tc_commit(&bar[0]);
    }
    ok = tc_wait(&bar[0], ph0, hdr, waits) && ok;
    ph0 ^= 1u;
    tc_after_sync();
    // y, the mask, mask w3
    float2 acc[2] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
    uint32_t mw[16], mk[16];
    load_sum32x4(mine, v);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int j = 32 * quarter + 2 * k;
      const float2 w = *reinterpret_cast<const float2 *>(V.w3 + j), z2 = relu_bias(v[k], V.b2 + j);
      acc[k & 1] = __ffma2_rn(w, z2, acc[k & 1]);
      const uint32_t on = (z2.x > 0.0f ? 0x0000ffffu : 0u) | (z2.y > 0.0f ? 0xffff0000u : 0u);
      mk[k] = on & 0x3f803f80u;   // 1.0 in bfloat16
      mw[k] = on & __byte_perm(__float_as_uint(w.x), __float_as_uint(w.y), 0x7632);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      *reinterpret_cast<uint4 *>(chunk(mask + (quarter >> 1) * kBlock, row, 4 * (quarter & 1u) + c)) =
          make_uint4(mk[4 * c], mk[4 * c + 1], mk[4 * c + 2], mk[4 * c + 3]);
    // y of the row: the quarters' sums
    part[quarter * kTileS + row] = (acc[0].x + acc[0].y) + (acc[1].x + acc[1].y);
    tc_before_sync();
    __syncthreads();   // (a2 has been read by all: its columns are free)
    tc_after_sync();
    tmem_st16(lanes + kTm + 16 * quarter, mw);
    // (every quarter computes dy for itself; rows past the batch: 0, they add nothing)
    const float y = ((part[row] + part[kTileS + row]) + (part[2 * kTileS + row] + part[3 * kTileS + row])) + V.b3;
    const float e = s0 + row < B ? y - target : 0.0f, dy = e * inv_b;
    if (quarter == 0) {
      lsum = fmaf(e, e, lsum);
      gb3 += dy;
    }
    tc_wait_st();
    tc_before_sync();
    __syncthreads();
    if (threadIdx.x == 0) {
      tc_after_sync();
      for (uint32_t k = 0; k < 8; ++k)   // d1 = (mask w3) W2
        mma_ts(tm + 128 * (k >> 2), tm + kTm + 8 * k, dw2 + k * kRows16, idesc(kH, false, true), (k & 3u) > 0);
      tc_commit(&bar[0]);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = make_float2(dy * z1[k].x, dy * z1[k].y);
    store_split32<false>(R, quarter, row, v);   // (layer 2's products have read z1)
    float2 odd = make_float2(dy * 0.0f, 0.0f);   // NaN once a factor is infinite or NaN
#pragma unroll
    for (int k = 0; k < 16; ++k) odd = __ffma2_rn(v[k], make_float2(0.0f, 0.0f), odd);
    if (quarter == 0) {
      uint32_t hi, mid, lo;
      split3<false>(make_float2(dy, 0.0f), hi, mid, lo);
      *reinterpret_cast<uint4 *>(chunk(E, row, 0)) = make_uint4(hi << 16, mid | lo << 16, 0, 0);
    }
    fence_proxy_async_smem();
    ok = tc_wait(&bar[0], ph0, hdr, waits) && ok;
    ph0 ^= 1u;
    tc_after_sync();
    load_sum32(mine, v);
#pragma unroll
    for (int k = 0; k < 16; ++k)   // d1
      z1[k] = make_float2(z1[k].x > 0.0f ? dy * v[k].x : 0.0f, z1[k].y > 0.0f ? dy * v[k].y : 0.0f);
#pragma unroll
    for (int k = 0; k < 16; ++k) odd = __ffma2_rn(z1[k], make_float2(0.0f, 0.0f), odd);
    const bool left_out = !(odd.x + odd.y == 0.0f);
    tc_before_sync();
    if (__syncthreads_or(left_out)) {   // those samples' operands become 0; add_samples makes up for them below
      if (left_out) atomicOr(&bad[row >> 5], 1u << (row & 31u));
      if (quarter == 0) bad_dy[row] = dy;
      __syncthreads();
      if ((bad[row >> 5] >> (row & 31u)) & 1u) {
#pragma unroll
        for (int k = 0; k < 16; ++k) z1[k] = make_float2(0.0f, 0.0f);
#pragma unroll 1
        for (uint32_t c = quarter; c < 6 * 8 + 1; c += 4)   // its 16-byte chunks in R, and the one in use in E
          *reinterpret_cast<uint4 *>(c < 48 ? chunk(R + (c >> 3) * kBlock, row, c & 7u) : chunk(E, row, 0)) = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      tc_after_sync();
      for (int p = 2; p >= 0; --p)         // mask^T (dy z1): every third 16 samples per accumulator
        for (uint32_t k = 0; k < 8; ++k)
          mma_ss(tm + 128 * (k % 3), dm + k * kRows16, dr + p * kPart + k * kRows16, idesc(kH, true, true), p < 2 || k > 2);
      for (uint32_t k = 0; k < 8; ++k)     // mask^T E
        mma_ss(tm + kTgB, dm + k * kRows16, de + k * kRows16, idesc(64, true, true), k > 0);
      tc_commit(&bar[1]);
    }
    load_x<kGradThreads>(x, B, s0 + (uint64_t)gridDim.x * kTileS, vec, xr);
    ok = tc_wait(&bar[1], ph1, hdr, waits) && ok;   // R and E are free
    ph1 ^= 1u;
    tc_after_sync();
    store_split32<false>(R, quarter, row, z1);
    if (quarter == 0) *reinterpret_cast<uint4 *>(chunk(E, row, 0)) = make_uint4(0x3f80u, 0, 0, 0);
    fence_proxy_async_smem();
    tc_before_sync();
    ok = __syncthreads_and(ok && !inf) != 0;
    if (!ok) break;
    if (threadIdx.x == 0) {
      tc_after_sync();
      for (int p = 2; p >= 0; --p)
        for (uint32_t k = 0; k < 8; ++k) {
          const uint64_t a = dr + p * kPart + k * kRows16;
          mma_ss(tm + kTgW1, a, dx + k * kRows16, idesc(kIn, true, true), p < 2 || k > 0);   // d1^T x
          mma_ss(tm + kTgB, a, de + k * kRows16, idesc(64, true, true), true);               // d1^T E
        }
      tc_commit(&bar[0]);
    }
    // meanwhile gW2 goes out: row j is this thread's lane
    const float w3 = fabsf(V.w3[row]) <= FLT_MAX ? V.w3[row] : 0.0f;   // (otherwise every sample was left out)
    float2 dot = make_float2(0.0f, 0.0f);
    load_sum32(mine, v);
    {
      uint32_t a[32];
      tmem_ld32(mine + 256, a);
      tc_wait_ld();
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = __fadd2_rn(v[k], as_float2(a[2 * k], a[2 * k + 1]));
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const uint4 w =
          *reinterpret_cast<const uint4 *>(chunk(sm + GradSmem::w2 + (quarter >> 1) * kBlock, row, 4 * (quarter & 1u) + c));
      const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
      const float2 *g = v + 4 * c;
#pragma unroll
      for (int k = 0; k < 4; ++k) dot = __ffma2_rn(as_float2(ww[k] << 16, ww[k] & 0xffff0000u), g[k], dot);
      float *p = grad + kW2 + row * kH + 32 * quarter + 8 * c;
      add4(p, w3 * g[0].x, w3 * g[0].y, w3 * g[1].x, w3 * g[1].y, gvec);
      add4(p + 4, w3 * g[2].x, w3 * g[2].y, w3 * g[3].x, w3 * g[3].y, gvec);
    }
    if (!(fabsf(dot.x + dot.y) <= FLT_MAX)) {   // a weight is infinite or NaN: 0 where no sample activates the unit
      float any = 0.0f;
#pragma unroll
      for (int k = 0; k < 16; ++k) any += fabsf(v[k].x) + fabsf(v[k].y);
      if (any == 0.0f) dot = make_float2(0.0f, 0.0f);
    }
    part[quarter * kTileS + row] = dot.x + dot.y;   // (dy's sums have been read)
    ok = tc_wait(&bar[0], ph0, hdr, waits);
    ph0 ^= 1u;
    tc_after_sync();
    ok = __syncthreads_and(ok) != 0;
    if (!ok) break;
    {
      uint32_t a[16];
      tmem_ld16(lanes + kTgW1 + 16 * quarter, a);
      tc_wait_ld();
#pragma unroll
      for (int k = 0; k < 16; k += 4)
        add4(grad + kW1 + row * kIn + 16 * quarter + k, __uint_as_float(a[k]), __uint_as_float(a[k + 1]),
             __uint_as_float(a[k + 2]), __uint_as_float(a[k + 3]), gvec);
      if (quarter == 0) {
        tmem_ld16(lanes + kTgB, a);
        tc_wait_ld();
        const float gd = (__uint_as_float(a[1]) + __uint_as_float(a[2])) + __uint_as_float(a[3]);   // mask^T dy
        const float d = (part[row] + part[kTileS + row]) + (part[2 * kTileS + row] + part[3 * kTileS + row]);
        atomicAdd(&grad[kB1 + row], __uint_as_float(a[0]));
        atomicAdd(&grad[kB2 + row], w3 * gd);
        atomicAdd(&grad[kW3 + row], gd != 0.0f ? fmaf(V.b2[row], gd, d) : d);
      }
    }
    const uint4 left = *reinterpret_cast<const uint4 *>(bad);
    if (left.x | left.y | left.z | left.w) {
      add_samples(sm, V, R, bad, bad_dy, 0.0f, nullptr, grad, loss_sum);
      if (threadIdx.x < 4) bad[threadIdx.x] = 0;
    }
    store_x<kGradThreads>(sm + GradSmem::x, xr);
    fence_proxy_async_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
  }
  if (!ok) {
    if (threadIdx.x == 0) tc_commit(&bar[2]);
    mbar_wait(&bar[2], 0, hdr);   // the products in flight
    if (__syncthreads_or(inf)) {   // an infinity in W2 (the first tile has ended here): sample by sample
      lsum = gb3 = 0.0f;
#pragma unroll 1
      for (uint64_t s0 = (uint64_t)blockIdx.x * kTileS; s0 < B; s0 += (uint64_t)gridDim.x * kTileS) {
        const uint64_t left = B - s0;   // rows of the tile
        if (threadIdx.x < 4) bad[threadIdx.x] = left >= 32 * threadIdx.x + 32 ? ~0u : left > 32 * threadIdx.x ? (1u << (left & 31u)) - 1u : 0u;
        __syncthreads();
        add_samples(sm, V, R, bad, nullptr, inv_b, t + s0, grad, loss_sum);
        load_x<kGradThreads>(x, B, s0 + (uint64_t)gridDim.x * kTileS, vec, xr);
        store_x<kGradThreads>(sm + GradSmem::x, xr);
        __syncthreads();
      }
    } else {
      lsum = __int_as_float(0x7fffffff);
    }
  }
  if (quarter == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lsum += __shfl_xor_sync(FULL, lsum, o);
      gb3 += __shfl_xor_sync(FULL, gb3, o);
    }
    if (lane == 0) {
      atomicAdd(&grad[kB3], gb3);
      atomicAdd(loss_sum, lsum);
    }
  }
  __syncthreads();
  if (warp == 0) tmem_free(tm, kTmCols);
}

__global__ void adam_kernel(float *p, uint16_t *wbf, const float *g, float *m, float *v, uint64_t n, float lr,
                            float beta1, float beta2, float eps, float bc1, float bc2) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = beta1 * m[i] + (1.0f - beta1) * gi;
    const float vi = beta2 * v[i] + (1.0f - beta2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    p[i] = pi;
    const __nv_bfloat16 h = __float2bfloat16_rn(pi);
    wbf[i] = *reinterpret_cast<const uint16_t *>(&h);
  }
}

}  // namespace esc

using namespace esc;

#define ESC_MLP_CK(call)                                                                      \
  do {                                                                                        \
    cudaError_t e_ = (call);                                                                  \
    if (e_ != cudaSuccess) return fail(ESC_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

namespace {
// Blocks for a batch: one per tile of samples, at most `per_sm` per SM; the
// kernels' attributes are set on a device's first call.
cudaError_t grid_for(uint64_t B, int per_sm, int *grid) {
  static std::once_flag once[64];
  static cudaError_t attr[64];
  static int sms[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::call_once(once[dev], [&] {
    attr[dev] = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
    if (attr[dev] == cudaSuccess)
      attr[dev] = cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FwdSmem::total);
    if (attr[dev] == cudaSuccess)
      attr[dev] = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GradSmem::total);
  });
  *grid = (int)std::max<uint64_t>(1, std::min<uint64_t>((B + kTileS - 1) / kTileS, (uint64_t)sms[dev] * per_sm));
  return attr[dev];
}
}  // namespace

extern "C" {

esc_status esc_debug_mlp_give_up(uint32_t wait) {
#ifdef ESC_CHECKED
  ESC_MLP_CK(cudaMemcpyToSymbol(g_mlp_give_up, &wait, sizeof wait));
  clear_error();
  return ESC_OK;
#else
  (void)wait;
  return fail(ESC_EINVAL, "esc_debug_mlp_give_up: only in the checked build");
#endif
}

esc_status esc_mlp_forward(const uint16_t *x_bf16, uint64_t batch, const uint16_t *w_bf16, const float *params,
                           float *y, void *stream) {
  ESC_RANGE("esc_mlp_forward");
  if (batch == 0) return ESC_OK;
  if (!x_bf16 || !w_bf16 || !params || !y) return fail(ESC_EINVAL, "esc_mlp_forward: NULL argument");
  int grid = 0;
  ESC_MLP_CK(grid_for(batch, 2, &grid));
  mlp_forward_kernel<<<grid, kFwdThreads, FwdSmem::total, static_cast<cudaStream_t>(stream)>>>(
      x_bf16, batch, w_bf16, params, y);
  ESC_MLP_CK(cudaGetLastError());
  clear_error();
  return ESC_OK;
}

esc_status esc_mlp_grad(const uint16_t *x_bf16, const float *target, uint64_t batch, const uint16_t *w_bf16,
                        const float *params, float *grad, float *loss_sum, void *stream) {
  ESC_RANGE("esc_mlp_grad");
  if (batch == 0) return ESC_OK;
  if (!x_bf16 || !target || !w_bf16 || !params || !grad || !loss_sum)
    return fail(ESC_EINVAL, "esc_mlp_grad: NULL argument");
  int grid = 0;
  ESC_MLP_CK(grid_for(batch, 1, &grid));
  mlp_grad_kernel<<<grid, kGradThreads, GradSmem::total, static_cast<cudaStream_t>(stream)>>>(
      x_bf16, target, batch, w_bf16, params, grad, loss_sum);
  ESC_MLP_CK(cudaGetLastError());
  clear_error();
  return ESC_OK;
}

esc_status esc_mlp_adam(float *params, uint16_t *w_bf16, const float *grad, float *m, float *v, uint64_t n, float lr,
                        float beta1, float beta2, float eps, int32_t step, void *stream) {
  ESC_RANGE("esc_mlp_adam");
  if (!params || !w_bf16 || !grad || !m || !v || step < 1) return fail(ESC_EINVAL, "esc_mlp_adam: bad argument");
  const float bc1 = 1.0f - powf(beta1, (float)step);
  const float bc2 = 1.0f - powf(beta2, (float)step);
  adam_kernel<<<(int)std::min<uint64_t>((n + 255) / 256, 1024), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      params, w_bf16, grad, m, v, n, lr, beta1, beta2, eps, bc1, bc2);
  ESC_MLP_CK(cudaGetLastError());
  clear_error();
  return ESC_OK;
}

}  // extern "C"
