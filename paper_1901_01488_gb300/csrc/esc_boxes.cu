// The shared scan of many predicates by table lookup: count-only sub-queries of
// one table, answered in one pass whose cost per row hardly grows with the
// number of predicates.
//
// Interpreting every predicate on every row costs about 47 lane instructions
// per predicate and row, so that pass is bound by instruction issue (4.0e11
// predicate-rows/s).  Here each row looks its tests up instead:
//  * Host: a predicate's program becomes a few disjoint boxes, conjunctions of
//    signed tests (a OR b = a, or (NOT a) AND b), each test on one operand: a
//    column, or a udf(a, b, m), which is treated as a column of its values.
//    The predicate's count is the sum of its boxes' counts.
//  * An operand's tests change only at their bounds (cuts).  The sorted cuts
//    split its domain into intervals on which every test is constant;
//    build_kernel evaluates, for each operand and interval, the tests of all
//    boxes at one value of the interval: a row of bits, one per box.
//  * box_kernel finds each row's interval in every operand (a bucket of equal
//    width, then binary search among its cuts; the value itself for u8), ANDs
//    the operands' bit rows, 32 boxes per word, and counts the words vertically:
//    bit-sliced counters fed by a carry-save tree, two logic instructions per
//    adder.
// What bounds it: for many boxes, the table rows' traffic through L1 (a row of
// 2048 predicates is about 420 bytes per operand: 50 % of L1's throughput, 46 %
// of it hits, and the latency shows at 16 warps per SM); for few, the
// instructions that find the intervals (67 % of the issue slots).  Measured on
// the 8M-row skewed table, interpreted before and looked up now: 16 predicates
// 304 -> 121 us, 32 555 -> 168, 64 1446 -> 220, 256 5.45 ms -> 0.52, 2048 42.0
// ms -> 2.26.  Without buckets the first three take 138, 195 and 265 us, and on
// 20M rows 256 predicates 1.58 ms (1.29 with), 512 2.97 (2.24), 2048 7.29 (6.35).
// Predicates that do not decompose within the limits below are interpreted
// (shared_kernel in esc_scan.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <string>
#include <vector>

#include "esc_boxes.h"
#include "esc_internal.h"
#include "esc_ptx.cuh"

namespace esc {

namespace {

constexpr int kBoxThreads = 256;
constexpr int kBoxWarps = kBoxThreads / 32;
constexpr int kTile = 512;              // rows per tile of box_words_kernel: two per thread in its search phase
constexpr int kPlanes = 11;             // bit planes of a vertical counter
constexpr uint32_t kMaxPending = (1u << kPlanes) - 1 - 8;
constexpr uint32_t kCutSmem = 16 * 1024;    // cuts copied to shared memory up to this size
constexpr uint32_t kTableSmem = 40 * 1024;  // the same for the bit table
// Bucket tables (see `bucket_search`): at most this many bytes for all operands
// and buckets for one, and about this many buckets per cut.  (512 to 2048 and 4
// to 32: within 2 % of one another, except that the larger tables cost a
// resident block at 32 predicates, 169 -> 185 us.)
constexpr uint32_t kBucketBytes = 16 * 1024;
constexpr uint32_t kMaxBuckets = 1024;
constexpr uint32_t kBucketsPerCut = 8;
constexpr int kBoxStages = 2;           // tiles of columns in flight or in use

// How an operand's interval is found: the value itself (u8), or by searching
// 32- or 64-bit cuts (an i64 column whose cuts all fit 32 bits is searched
// with its values saturated to 32).
enum OperandKind : int32_t { OPD_U8 = 0, OPD_32 = 1, OPD_64 = 2 };

struct Operand {
  uint32_t a, b;          // byte offsets of the columns in a stage; b: a udf's second one, else ~0
  int32_t da, db;         // their esc_dtype
  int32_t kind;           // OperandKind of the value searched
  uint32_t ncuts;         // intervals: ncuts + 1
  uint32_t steps;         // binary-search steps; 2^steps - 1 padded cuts at least
  uint32_t cut_off;       // byte offset of the cuts
  uint32_t table_off;     // byte offset of interval 0's bit row
  // buckets of equal width (2^shift) over the cuts' values (kind OPD_32; bsteps ~0: none)
  uint32_t bsteps;        // binary-search steps left in a bucket
  uint32_t bucket_off;    // byte offset of the buckets
  int32_t base, top;      // one below the first cut; the last cut
  uint32_t shift;
  // udf: modulus, its remainder constants (below 2^16: M, K; else mult, sh1, sh2)
  uint32_t K;
  int32_t sh1, sh2;
  uint64_t d, M, mult;
#ifdef ESC_CHECKED
  uint32_t padded;        // cuts with their padding
  uint32_t nbuckets;
#endif
};

struct StageColumn {
  const uint8_t *data;
  uint32_t w, off;
};

struct BoxLaunch {
  Operand op[kMaxOperands];
  StageColumn col[kMaxRef];
  int32_t nop, ncol;
  uint32_t stage_bytes;
  uint32_t nopp;              // nop rounded up to a multiple of 4
  uint32_t nrows;
  uint32_t nboxes;
  uint32_t stride;            // bytes of a bit row
  uint32_t cut_bytes, table_bytes;
  uint32_t tile;              // rows per tile
  uint32_t lanes;             // lanes that share a row (power of two)
  uint32_t chunks;            // passes over a bit row: VEC * lanes words each
  uint32_t cuts_in_smem;
  uint32_t bucket_bytes;
  // byte offsets in shared memory (first the stages)
  uint32_t smem_offs, smem_cnt, smem_cut, smem_table, smem_bar, smem_bucket;
  const uint8_t *cuts;        // sorted, padded
  const uint8_t *buckets;     // u16 each
  uint8_t *table;
  const uint32_t *pred_of_box;
  const uint32_t *lane_ops;   // per 4 words of the bit row: operands their boxes test (bits)
  unsigned long long *counts;
  ScratchHdr *hdr;
};

// Build-time view: every box's signed tests, sorted by operand.
struct BuildArgs {
  const BoxTest *tests;
  const uint32_t *refs;       // test << 1 | negated
  const uint2 *box_ref;       // its range of refs
  const int64_t *pool;
};

[[maybe_unused]] __device__ __forceinline__ uint32_t width_of(int32_t dt) {
  return dt == ESC_U8 ? 1u : dt == ESC_U16 ? 2u : dt == ESC_I32 ? 4u : 8u;
}

__device__ __forceinline__ int64_t load_value(const uint8_t *p, int32_t dt, uint32_t row) {
  switch (dt) {
    case ESC_U8: return p[row];
    case ESC_U16: return reinterpret_cast<const uint16_t *>(p)[row];
    case ESC_I32: return reinterpret_cast<const int32_t *>(p)[row];
    default: return reinterpret_cast<const long long *>(p)[row];
  }
}

// x mod d for 32-bit x, 1 <= d < 2^32, M = ceil(2^64 / d) (Lemire, Kaser & Kurz 2019).
__device__ __forceinline__ uint32_t mod32(uint32_t x, uint64_t M, uint32_t d) {
  const uint64_t low = M * (uint64_t)x;
  const uint64_t u = (uint64_t)(uint32_t)(low >> 32) * d + __umulhi((uint32_t)low, d);
  return (uint32_t)(u >> 32);
}

// (a * b) mod d: the product wraps in 64 bits, the remainder truncates toward zero.
__device__ __forceinline__ int64_t udf_value(const Operand &o, int64_t a, int64_t b) {
  const int64_t p = (int64_t)((uint64_t)a * (uint64_t)b);
  const uint64_t n = p < 0 ? 0ull - (uint64_t)p : (uint64_t)p;
  uint64_t r;
  if (o.d < 65536u) {
    const uint32_t d = (uint32_t)o.d;
    uint32_t x = (uint32_t)n;
    if (n >> 32) x = mod32((uint32_t)(n >> 32), o.M, d) * o.K + mod32(x, o.M, d);  // below d^2 < 2^32
    r = mod32(x, o.M, d);
  } else {
    const uint64_t t = __umul64hi(o.mult, n);
    r = n - ((t + ((n - t) >> o.sh1)) >> o.sh2) * o.d;
  }
  return p < 0 ? -(int64_t)r : (int64_t)r;
}

// Whether value v passes a test (its sign aside).
__device__ __forceinline__ bool test_value(const BoxTest &t, const int64_t *pool, int64_t v) {
  if (t.op == OP_INSET) {
    if ((uint64_t)v >= 256u) return false;
    return ((uint64_t)pool[t.off + (v >> 6)] >> (v & 63)) & 1u;
  }
  if (t.op == OP_IN) {
    bool in = false;
    for (uint32_t k = 0; k < t.n; ++k) in = in || pool[t.off + k] == v;
    return in;
  }
  return t.lo <= v && v <= t.hi;
}

// Sorts an operand's cuts: each of them finds its place by counting those
// before it (a few thousand at most per operand, one launch for all; equal
// cuts keep their order and make empty intervals).  16 threads share a cut.
struct SortJob {
  uint32_t src;       // first of its cuts in the unsorted array
  uint32_t n, padded;
  uint32_t dst_off;   // byte offset of the sorted ones
  uint32_t wide;      // 64-bit cuts
};
constexpr uint32_t kSortCuts = 64;   // cuts per block
__global__ void __launch_bounds__(1024) sort_cuts_kernel(const int64_t *unsorted, const SortJob *jobs, uint8_t *cuts,
                                                         [[maybe_unused]] ScratchHdr *hdr) {
  __shared__ uint32_t rank[kSortCuts];
  const SortJob J = jobs[blockIdx.y];
  if (blockIdx.x * kSortCuts >= J.padded) return;   // uniform
  const uint32_t i = blockIdx.x * kSortCuts + threadIdx.x % kSortCuts, part = threadIdx.x / kSortCuts;
  if (threadIdx.x < kSortCuts) rank[threadIdx.x] = 0;
  __syncthreads();
  const int64_t *src = unsorted + J.src;
  const int64_t v = i < J.n ? src[i] : 0;
  if (i < J.n) {
    const uint32_t j0 = (uint32_t)((uint64_t)J.n * part / 16), j1 = (uint32_t)((uint64_t)J.n * (part + 1) / 16);
    uint32_t r = 0;
#pragma unroll 4
    for (uint32_t j = j0; j < j1; ++j) {
      const int64_t c = src[j];
      r += (c < v || (c == v && j < i)) ? 1u : 0u;
    }
    atomicAdd(&rank[threadIdx.x % kSortCuts], r);
  }
  __syncthreads();
  if (part != 0 || i >= J.padded) return;
  // padding past the last cut: the type's largest value
  const uint32_t at = i < J.n ? rank[threadIdx.x] : i;
  if (!ESC_INB(hdr, at < J.padded, 48, at)) return;
  if (J.wide) reinterpret_cast<int64_t *>(cuts + J.dst_off)[at] = i < J.n ? v : INT64_MAX;
  else reinterpret_cast<int32_t *>(cuts + J.dst_off)[at] = i < J.n ? (int32_t)v : INT32_MAX;
}

// Number of an operand's sorted cuts <= v (its interval of value v).
__device__ __forceinline__ uint32_t interval_of(const BoxLaunch &L, const Operand &o, int64_t v) {
  const uint8_t *cuts = L.cuts;
  if (o.kind == OPD_U8) return v < 0 ? 0u : (uint32_t)min(v, (int64_t)255);
  uint32_t pos = 0;
  for (uint32_t h = 1u << o.steps >> 1; h; h >>= 1) {
    if (!ESC_INB(L.hdr, pos + h <= o.padded, 44, pos + h)) return 0;
    const int64_t c = o.kind == OPD_64 ? reinterpret_cast<const int64_t *>(cuts + o.cut_off)[pos + h - 1]
                                       : (int64_t)reinterpret_cast<const int32_t *>(cuts + o.cut_off)[pos + h - 1];
    pos += c <= v ? h : 0u;
  }
  return min(pos, o.ncuts);
}

// The bit table: a warp makes one word (32 boxes, a lane each) of a run of an
// operand's intervals.  A box mostly has no or one range test of the operand:
// a run of intervals, found once; anything else is evaluated at each
// interval's first value.
constexpr int kBuildRun = 64;
__global__ void __launch_bounds__(256) build_kernel(const __grid_constant__ BoxLaunch L, const BuildArgs B) {
  const Operand &o = L.op[blockIdx.y];
  const uint32_t nint = o.kind == OPD_U8 ? 256u : o.ncuts + 1u;
  const uint32_t i0 = blockIdx.z * kBuildRun;
  if (i0 >= nint) return;
  const uint32_t word = blockIdx.x * 8u + (threadIdx.x >> 5), lane = threadIdx.x & 31u;
  if (word * 4u >= L.stride) return;
  const uint32_t box = word * 32u + lane;
  const bool real = box < L.nboxes;
  uint32_t r0 = 0, r1 = 0;   // the box's tests of this operand
  if (real) {
    const uint32_t e = B.box_ref[box].y;
    r0 = B.box_ref[box].x;
    while (r0 < e && B.tests[B.refs[r0] >> 1].operand < (uint32_t)blockIdx.y) ++r0;
    r1 = r0;
    while (r1 < e && B.tests[B.refs[r1] >> 1].operand == (uint32_t)blockIdx.y) ++r1;
  }
  bool general = r1 > r0 + 1;
  uint32_t a = 0, len = real ? ~0u : 0u, neg = 0;   // passes intervals a .. a + len - 1, or all others
  if (r1 == r0 + 1) {
    const BoxTest &t = B.tests[B.refs[r0] >> 1];
    neg = B.refs[r0] & 1u;
    if (t.op == OP_RANGE) {
      a = interval_of(L, o, t.lo);
      len = interval_of(L, o, t.hi) - a + 1u;
    } else {
      general = true;
    }
  }
  const bool any_general = __any_sync(FULL, general);
  const uint32_t i1 = min(i0 + kBuildRun, nint);
  for (uint32_t ib = i0; ib < i1; ib += 32) {
    uint32_t mine = 0;
    const uint32_t ie = min(ib + 32u, i1);
    for (uint32_t i = ib; i < ie; ++i) {
      bool in = (i - a < len) != (neg != 0);
      if (any_general) {
        int64_t v;   // a value of interval i: its first one, or the one before the first cut
        if (o.kind == OPD_U8) v = i;
        else if (o.ncuts == 0) v = 0;
        else if (o.kind == OPD_64) {
          const int64_t *c = reinterpret_cast<const int64_t *>(L.cuts + o.cut_off);
          v = i ? c[i - 1] : c[0] - 1;
        } else {
          const int32_t *c = reinterpret_cast<const int32_t *>(L.cuts + o.cut_off);
          v = i ? (int64_t)c[i - 1] : (int64_t)c[0] - 1;
        }
        if (general) {
          in = true;
          for (uint32_t r = r0; in && r < r1; ++r) {
            const uint32_t f = B.refs[r];
            in = test_value(B.tests[f >> 1], B.pool, v) != ((f & 1u) != 0);
          }
        }
      }
      const uint32_t w = __ballot_sync(FULL, in);
      if (lane == (i & 31u)) mine = w;
    }
    // interval ib + lane: ib is a multiple of 32
    const uint64_t at = (uint64_t)o.table_off + (uint64_t)(ib + lane) * L.stride + word * 4u;
    if (ib + lane < i1 && ESC_INB(L.hdr, at + 4 <= L.table_bytes, 40, at))
      *reinterpret_cast<uint32_t *>(L.table + at) = mine;
  }
}

// Numbers of sorted cuts <= v[k]: `steps` halvings of a padded array.
template <typename T, int R>
__device__ __forceinline__ void search([[maybe_unused]] const BoxLaunch &L, const Operand &o, const uint8_t *cuts,
                                       const T (&v)[R], uint32_t (&pos)[R]) {
  const T *cut = reinterpret_cast<const T *>(cuts + o.cut_off) - 1;
#pragma unroll
  for (int k = 0; k < R; ++k) pos[k] = 0;
  for (uint32_t h = 1u << o.steps >> 1; h; h >>= 1) {
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const uint32_t t = pos[k] + h;
      if (ESC_INB(L.hdr, t <= o.padded, 44, t) && cut[t] <= v[k]) pos[k] = t;
    }
  }
#pragma unroll
  for (int k = 0; k < R; ++k) pos[k] = min(pos[k], o.ncuts);   // padding equals the largest value
}

// The same with a table of buckets: the value's bucket gives the number of cuts
// before it (with buckets of one value: up to it), and the search goes on among
// the bucket's own cuts, `bsteps` halvings for the fullest one.  Later buckets'
// cuts lie above the value, so halvings past the bucket's end find nothing.
template <int R>
__device__ __forceinline__ void bucket_search([[maybe_unused]] const BoxLaunch &L, const Operand &o,
                                              const uint8_t *cuts, const uint8_t *buckets, const int32_t (&v)[R], uint32_t (&pos)[R]) {
  const int32_t *cut = reinterpret_cast<const int32_t *>(cuts + o.cut_off) - 1;
  const uint16_t *first = reinterpret_cast<const uint16_t *>(buckets + o.bucket_off);
  int32_t w[R];
#pragma unroll
  for (int k = 0; k < R; ++k) {
    w[k] = max(o.base, min(v[k], o.top));
    const uint32_t b = ((uint32_t)w[k] - (uint32_t)o.base) >> o.shift;
    pos[k] = ESC_INB(L.hdr, b < o.nbuckets, 43, b) ? first[b] : 0u;
  }
  for (uint32_t h = 1u << o.bsteps >> 1; h; h >>= 1) {
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const uint32_t t = pos[k] + h;
      if (ESC_INB(L.hdr, t <= o.padded, 44, t) && cut[t] <= w[k]) pos[k] = t;
    }
  }
#pragma unroll
  for (int k = 0; k < R; ++k) pos[k] = min(pos[k], o.ncuts);
}

template <int R>
__device__ __forceinline__ void search32(const BoxLaunch &L, const Operand &o, const uint8_t *cuts,
                                         const uint8_t *buckets, const int32_t (&v)[R], uint32_t (&pos)[R]) {
  if (o.bsteps != ~0u) bucket_search<R>(L, o, cuts, buckets, v, pos);
  else search<int32_t, R>(L, o, cuts, v, pos);
}

__device__ __forceinline__ int32_t saturate32(int64_t v) {
  return (int32_t)max((int64_t)INT32_MIN, min((int64_t)INT32_MAX, v));
}

// The intervals of operand o of R rows of a staged tile: rows row + k * kBoxThreads.
template <int R>
__device__ __forceinline__ void intervals(const BoxLaunch &L, const Operand &o, const uint8_t *stage, const uint8_t *cuts,
                                          const uint8_t *buckets, uint32_t row, uint32_t (&pos)[R]) {
  const uint8_t *a = stage + o.a;
#ifdef ESC_CHECKED
  const uint32_t rows = row + (R - 1) * kBoxThreads + 1;
  if (!ESC_INB(L.hdr, o.a + rows * width_of(o.da) <= L.stage_bytes, 45, o.a) ||
      (o.b != ~0u && !ESC_INB(L.hdr, o.b + rows * width_of(o.db) <= L.stage_bytes, 45, o.b))) {
    for (int k = 0; k < R; ++k) pos[k] = 0;
    return;
  }
#endif
  if (o.kind == OPD_U8) {
#pragma unroll
    for (int k = 0; k < R; ++k) pos[k] = a[row + k * kBoxThreads];
    return;
  }
  if (o.b == ~0u && o.da != ESC_I64) {
    int32_t v[R];
    if (o.da == ESC_I32) {
#pragma unroll
      for (int k = 0; k < R; ++k) v[k] = reinterpret_cast<const int32_t *>(a)[row + k * kBoxThreads];
    } else {
#pragma unroll
      for (int k = 0; k < R; ++k) v[k] = reinterpret_cast<const uint16_t *>(a)[row + k * kBoxThreads];
    }
    search32<R>(L, o, cuts, buckets, v, pos);
    return;
  }
  long long v[R];
#pragma unroll
  for (int k = 0; k < R; ++k) v[k] = load_value(a, o.da, row + k * kBoxThreads);
  if (o.b != ~0u) {
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = udf_value(o, v[k], load_value(stage + o.b, o.db, row + k * kBoxThreads));
  }
  if (o.kind == OPD_64) {
    search<long long, R>(L, o, cuts, v, pos);
  } else {
    int32_t w[R];
#pragma unroll
    for (int k = 0; k < R; ++k) w[k] = saturate32(v[k]);
    search32<R>(L, o, cuts, buckets, w, pos);
  }
}

template <int VEC>
struct Words {
  uint32_t w[VEC];
};

template <int VEC>
__device__ __forceinline__ void and_row(Words<VEC> &x, const uint8_t *p) {
  if constexpr (VEC == 1) {
    x.w[0] &= *reinterpret_cast<const uint32_t *>(p);
  } else if constexpr (VEC == 2) {
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    x.w[0] &= v.x;
    x.w[1] &= v.y;
  } else {
    const uint4 v = *reinterpret_cast<const uint4 *>(p);
    x.w[0] &= v.x;
    x.w[1] &= v.y;
    x.w[2] &= v.z;
    x.w[3] &= v.w;
  }
}

__device__ __forceinline__ uint32_t maj(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (a & c) | (b & c); }

// Adds a lane's vertical counters to the block's, box by box; lanes start at
// different bits, so those that hold the same word hit different counters.
template <int VEC>
__device__ __forceinline__ void flush_planes(uint32_t (&p)[VEC][kPlanes], uint32_t *cnt, uint32_t word0, uint32_t nboxes,
                                             uint32_t lane) {
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < kPlanes; ++k) any |= p[v][k];
    for (uint32_t j = 0; any != 0 && j < 32; ++j) {
      const uint32_t b = (j + lane) & 31u;
      if (!((any >> b) & 1u)) continue;
      uint32_t c = 0;
#pragma unroll
      for (int k = 0; k < kPlanes; ++k) c |= ((p[v][k] >> b) & 1u) << k;
      const uint32_t box = (word0 + v) * 32u + b;
      if (box < nboxes) atomicAdd(&cnt[box], c);
    }
#pragma unroll
    for (int k = 0; k < kPlanes; ++k) p[v][k] = 0;
  }
}

// Copies tile `tile`'s columns into a stage (warp 0): bulk copies, the last
// bytes of a ragged tile by hand.
__device__ __forceinline__ void issue_tile(const BoxLaunch &L, uint32_t tile, uint8_t *stage, uint64_t *full, uint32_t lane) {
  const uint32_t row0 = tile * L.tile, rows = min(L.tile, L.nrows - row0);
  uint32_t bulk = 0, tail = 0;
  const uint8_t *src = nullptr;
  uint8_t *dst = nullptr;
  if (lane < (uint32_t)L.ncol) {
    const StageColumn &c = L.col[lane];
    bulk = (rows * c.w) & ~15u;
    tail = rows * c.w - bulk;
    src = c.data + (size_t)row0 * c.w;
    dst = stage + c.off;
    if (!ESC_INB(L.hdr, c.off + rows * c.w <= L.stage_bytes, 42, c.off)) bulk = tail = 0;
  }
  if (__ballot_sync(FULL, tail != 0)) {
    for (uint32_t k = 0; k < tail; ++k) dst[bulk + k] = src[bulk + k];
    fence_proxy_async_smem();
  }
  const uint32_t tot = __reduce_add_sync(FULL, bulk);
  __syncwarp();
  if (lane == 0) mbar_arrive_expect_tx(full, tot);
  __syncwarp();
  if (bulk) bulk_load(dst, src, bulk, full);
}

// What both kernels share: a block's tiles (every gridDim.x-th), taken
// `passes` times, arrive in kBoxStages stages while the one before is worked
// on.  (Plain loads, one operand after the other, left the kernel waiting for
// memory: 299 us against 242 with the ring for 16 predicates on 8M rows.)
struct TileRing {
  uint8_t *stages;
  uint64_t *full;
  uint32_t mine, total;
  __device__ __forceinline__ uint32_t tile(uint32_t j) const { return blockIdx.x + (j % mine) * gridDim.x; }
  __device__ __forceinline__ void start(const BoxLaunch &L, uint8_t *sm, uint32_t passes) {
    stages = sm;
    full = reinterpret_cast<uint64_t *>(sm + L.smem_bar);
    const uint32_t ntiles = (L.nrows + L.tile - 1) / L.tile;   // grid <= ntiles
    mine = (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
    total = mine * passes;
    if (threadIdx.x == 0) {
      for (int s = 0; s < kBoxStages; ++s) mbar_init(&full[s], 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x < 32)
      for (uint32_t j = 0; j < kBoxStages && j < total; ++j) issue(L, j);
  }
  __device__ __forceinline__ void issue(const BoxLaunch &L, uint32_t j) const {   // warp 0
    issue_tile(L, tile(j), stages + j % kBoxStages * L.stage_bytes, &full[j % kBoxStages], threadIdx.x);
  }
  __device__ __forceinline__ bool wait(const BoxLaunch &L, uint32_t j) const {
    return mbar_wait(&full[j % kBoxStages], (j / kBoxStages) & 1u, L.hdr);
  }
  // Barrier after the stage's last use; then the copy of tile j + kBoxStages
  // goes into it.  False (for the whole block) when a warp gave up waiting: the
  // copies in flight, this tile's too, are waited for, bounded, and the block leaves.
  __device__ __forceinline__ bool release(const BoxLaunch &L, uint32_t j, bool ok) const {
    if (!__syncthreads_and(ok)) {
      for (uint32_t k = j; k < total && k < j + kBoxStages; ++k) wait(L, k);
      return false;
    }
    if (threadIdx.x < 32 && j + kBoxStages < total) issue(L, j + kBoxStages);
    return true;
  }
};

__device__ __forceinline__ void copy16(uint8_t *dst, const uint8_t *src, uint32_t bytes) {
  for (uint32_t i = threadIdx.x; i < bytes / 16; i += kBoxThreads)
    reinterpret_cast<uint4 *>(dst)[i] = reinterpret_cast<const uint4 *>(src)[i];
}

__device__ __forceinline__ void flush_counts(const BoxLaunch &L, const uint32_t *cnt) {
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < L.nboxes; i += kBoxThreads)
    if (cnt[i]) atomicAdd(&L.counts[L.pred_of_box[i]], (unsigned long long)cnt[i]);
}

// Adds two words to the vertical counters of one word of boxes.
__device__ __forceinline__ void ripple(uint32_t (&p)[kPlanes], uint32_t c, int at) {
#pragma unroll
  for (int k = 0; k < kPlanes; ++k) {
    if (k < at) continue;
    const uint32_t n = p[k] & c;
    p[k] ^= c;
    c = n;
  }
}

// Few boxes (at most VEC words): a thread keeps its rows' words in registers,
// kRows rows at a time; cuts and bit table in shared memory.  (With the rows'
// offsets passed through shared memory as below, and two rows a thread, 16
// predicates on 8M rows took 242 us, 653 lane instructions a row; this way
// 143 us and 403.)
constexpr int kRows = 4;
template <int VEC>
__global__ void __launch_bounds__(kBoxThreads, VEC == 4 ? 2 : 3) box_rows_kernel(const __grid_constant__ BoxLaunch L) {
  extern __shared__ __align__(128) uint8_t sm[];
  uint32_t *cnt = reinterpret_cast<uint32_t *>(sm + L.smem_cnt);
  TileRing ring;
  ring.start(L, sm, 1);
  for (uint32_t i = threadIdx.x; i < L.nboxes; i += kBoxThreads) cnt[i] = 0;
  copy16(sm + L.smem_cut, L.cuts, L.cut_bytes);
  copy16(sm + L.smem_table, L.table, L.table_bytes);
  copy16(sm + L.smem_bucket, L.buckets, L.bucket_bytes);
  const uint8_t *cuts = sm + L.smem_cut, *table = sm + L.smem_table;
  uint32_t p[VEC][kPlanes];
#pragma unroll
  for (int v = 0; v < VEC; ++v)
#pragma unroll
    for (int k = 0; k < kPlanes; ++k) p[v][k] = 0;
  uint32_t pending = 0;
  __syncthreads();
  for (uint32_t j = 0; j < ring.total; ++j) {
    const uint32_t row0 = ring.tile(j) * L.tile, rows = min(L.tile, L.nrows - row0);
    const uint8_t *stage = sm + j % kBoxStages * L.stage_bytes;
    const bool ok = ring.wait(L, j);
    Words<VEC> x[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k)
#pragma unroll
      for (int v = 0; v < VEC; ++v) x[k].w[v] = threadIdx.x + k * kBoxThreads < rows ? FULL : 0u;
    // (rows past the last one read what the stage holds; nothing counts them)
    for (int c = 0; c < L.nop; ++c) {
      const Operand &o = L.op[c];
      uint32_t pos[kRows];
      intervals<kRows>(L, o, stage, cuts, sm + L.smem_bucket, threadIdx.x, pos);
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        uint32_t off = o.table_off + pos[k] * (4u * VEC);
        if (!ESC_INB(L.hdr, off + 4u * VEC <= L.table_bytes, 41, off)) off = o.table_off;
        and_row<VEC>(x[k], table + off);
      }
    }
    if (!ring.release(L, j, ok)) return;
    if (pending > kMaxPending) {
      flush_planes<VEC>(p, cnt, 0, L.nboxes, threadIdx.x & 31u);
      pending = 0;
    }
    pending += kRows;
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      const uint32_t a = maj(p[v][0], x[0].w[v], x[1].w[v]);
      p[v][0] ^= x[0].w[v] ^ x[1].w[v];
      const uint32_t b = maj(p[v][0], x[2].w[v], x[3].w[v]);
      p[v][0] ^= x[2].w[v] ^ x[3].w[v];
      const uint32_t c = maj(p[v][1], a, b);
      p[v][1] ^= a ^ b;
      ripple(p[v], c, 2);
    }
  }
  flush_planes<VEC>(p, cnt, 0, L.nboxes, threadIdx.x & 31u);
  flush_counts(L, cnt);
}

// Many boxes.  Phase 1 of a tile: thread = row, the rows' table offsets into
// shared memory.  Phase 2: `lanes` lanes share a row, each 4 words (128 boxes)
// of its bit row, which comes from L1 and L2.  The first four operands have
// the largest tables; boxes are ordered by which of the four they test, and a
// lane skips those of the four that none of its boxes tests (2048 predicates
// on 20M rows: 7.6 ms without, 6.7 with).  Skipping further operands of a row
// once none of a lane's boxes is left saved traffic but cost more in
// instructions (9.4 ms).
__global__ void __launch_bounds__(kBoxThreads, 2) box_words_kernel(const __grid_constant__ BoxLaunch L) {
  extern __shared__ __align__(128) uint8_t sm[];
  uint32_t *offs = reinterpret_cast<uint32_t *>(sm + L.smem_offs);
  uint32_t *cnt = reinterpret_cast<uint32_t *>(sm + L.smem_cnt);
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  TileRing ring;
  ring.start(L, sm, L.chunks);
  for (uint32_t i = threadIdx.x; i < L.nboxes; i += kBoxThreads) cnt[i] = 0;
  copy16(sm + L.smem_bucket, L.buckets, L.bucket_bytes);
  const uint8_t *cuts = L.cuts;
  if (L.cuts_in_smem) {
    copy16(sm + L.smem_cut, L.cuts, L.cut_bytes);
    cuts = sm + L.smem_cut;
  }
  const uint32_t lanes = L.lanes, rows_per_step = 32u / lanes;
  const uint32_t sub = lane & (lanes - 1), rsub = lane / lanes;
  const uint32_t steps = kTile / (kBoxWarps * rows_per_step);
  const uint32_t nopp = L.nopp, nop = (uint32_t)L.nop;
  uint32_t p[4][kPlanes];
#pragma unroll
  for (int v = 0; v < 4; ++v)
#pragma unroll
    for (int k = 0; k < kPlanes; ++k) p[v][k] = 0;
  uint32_t pending = 0, word0 = 0, need = 0, lane_off = 0;
  bool live = false;
  __syncthreads();   // the copies above
  for (uint32_t j = 0; j < ring.total; ++j) {
    if (j % ring.mine == 0) {   // the next chunk of the bit rows
      if (live) flush_planes<4>(p, cnt, word0, L.nboxes, lane);
      pending = 0;
      word0 = (j / ring.mine * lanes + sub) * 4;
      live = word0 * 4u < L.stride &&   // a bit row may be shorter than the chunk
             ESC_INB(L.hdr, word0 / 4 < (L.nboxes + 127) / 128, 47, word0);
      lane_off = live ? word0 * 4u : 0u;
      need = live ? L.lane_ops[word0 / 4] : 0u;
    }
    const uint32_t row0 = ring.tile(j) * kTile;
    const uint32_t rows = min((uint32_t)kTile, L.nrows - row0);
    const uint8_t *stage = sm + j % kBoxStages * L.stage_bytes;
    const bool ok = ring.wait(L, j);
    for (int c = 0; c < L.nop; ++c) {
      const Operand &o = L.op[c];
      uint32_t pos[2];
      intervals<2>(L, o, stage, cuts, sm + L.smem_bucket, threadIdx.x, pos);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        uint32_t off = o.table_off + pos[k] * L.stride;
        if (!ESC_INB(L.hdr, (uint64_t)off + L.stride <= L.table_bytes, 41, off)) off = o.table_off;
        offs[(threadIdx.x + k * kBoxThreads) * nopp + c] = off;
      }
    }
    if (!ring.release(L, j, ok)) return;   // (also: the offsets are there)
    const bool n0 = need & 1u, n1 = need & 2u, n2 = need & 4u, n3 = need & 8u;
    constexpr int U = 8;   // rows per step of the carry-save tree
    for (uint32_t q = 0; q < steps; q += U) {
      if (pending > kMaxPending) {
        if (live) flush_planes<4>(p, cnt, word0, L.nboxes, lane);
        pending = 0;
      }
      pending += U;
      uint32_t tw[4], fo[4];
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        Words<4> x[2];
        const uint32_t *ro[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const uint32_t r = (warp * steps + q + u + k) * rows_per_step + rsub;
          const bool in = live && q + u + k < steps && r < rows && ESC_INB(L.hdr, r < (uint32_t)kTile, 46, r);
          ro[k] = &offs[(in ? r : 0u) * nopp];
#pragma unroll
          for (int v = 0; v < 4; ++v) x[k].w[v] = in ? FULL : 0u;
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const uint4 f = *reinterpret_cast<const uint4 *>(ro[k]);
          if (n0) and_row<4>(x[k], L.table + (f.x + lane_off));
          if (n1) and_row<4>(x[k], L.table + (f.y + lane_off));
          if (n2) and_row<4>(x[k], L.table + (f.z + lane_off));
          if (n3) and_row<4>(x[k], L.table + (f.w + lane_off));
        }
        uint32_t g = 4;
        for (; g + 4 <= nop; g += 4) {
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const uint4 f = *reinterpret_cast<const uint4 *>(ro[k] + g);
            and_row<4>(x[k], L.table + (f.x + lane_off));
            and_row<4>(x[k], L.table + (f.y + lane_off));
            and_row<4>(x[k], L.table + (f.z + lane_off));
            and_row<4>(x[k], L.table + (f.w + lane_off));
          }
        }
        for (; g < nop; ++g) {
#pragma unroll
          for (int k = 0; k < 2; ++k) and_row<4>(x[k], L.table + (ro[k][g] + lane_off));
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const uint32_t c2 = maj(p[v][0], x[0].w[v], x[1].w[v]);
          p[v][0] ^= x[0].w[v] ^ x[1].w[v];
          if (!(u & 2)) {
            tw[v] = c2;
            continue;
          }
          const uint32_t c4 = maj(p[v][1], tw[v], c2);
          p[v][1] ^= tw[v] ^ c2;
          if (!(u & 4)) {
            fo[v] = c4;
            continue;
          }
          const uint32_t c8 = maj(p[v][2], fo[v], c4);
          p[v][2] ^= fo[v] ^ c4;
          ripple(p[v], c8, 3);
        }
      }
    }
    __syncthreads();   // the offsets are used up
  }
  if (live) flush_planes<4>(p, cnt, word0, L.nboxes, lane);
  flush_counts(L, cnt);
}

// ------------------------------------------------------------------ host: boxes
// A box as two sets of the program's instructions: tests that hold, tests that fail.
struct Mask {
  uint64_t pos, neg;
};

struct Node {
  uint8_t kind;   // 0 test, 1 AND, 2 OR, 3 NOT, 4 TRUE, 5 FALSE
  int16_t a, b;
};

// The disjoint boxes of a subtree (of its complement when neg): their number, -1 if more than `cap`.
int expand(const Node *n, int at, bool neg, Mask *out, int cap) {
  const Node &x = n[at];
  switch (x.kind) {
    case 0:
      if (cap < 1) return -1;
      out[0] = neg ? Mask{0, 1ull << at} : Mask{1ull << at, 0};
      return 1;
    case 3: return expand(n, x.a, !neg, out, cap);
    case 4:
    case 5:
      if ((x.kind == 4) == neg) return 0;
      if (cap < 1) return -1;
      out[0] = Mask{0, 0};
      return 1;
    default: break;
  }
  Mask A[kMaxBoxes], B[kMaxBoxes];
  int k = 0;
  auto product = [&](int na, int nb) {
    for (int i = 0; i < na; ++i)
      for (int j = 0; j < nb; ++j) {
        const Mask m{A[i].pos | B[j].pos, A[i].neg | B[j].neg};
        if (m.pos & m.neg) continue;   // a test and its negation: empty
        if (k == cap) return false;
        out[k++] = m;
      }
    return true;
  };
  if ((x.kind == 1) != neg) {   // a AND b (NOT (a OR b) = NOT a AND NOT b)
    const int na = expand(n, x.a, neg, A, kMaxBoxes), nb = na < 0 ? -1 : expand(n, x.b, neg, B, kMaxBoxes);
    if (nb < 0 || !product(na, nb)) return -1;
  } else {                      // a OR b: a, or (NOT a) AND b
    const int na = expand(n, x.a, neg, out, cap);
    if (na < 0) return -1;
    k = na;
    const int nn = expand(n, x.a, !neg, A, kMaxBoxes), nb = nn < 0 ? -1 : expand(n, x.b, neg, B, kMaxBoxes);
    if (nb < 0 || !product(nn, nb)) return -1;
  }
  return k;
}

}  // namespace

int predicate_boxes(const esc_pred *p, uint64_t *pos, uint64_t *neg) {
  Node n[kMaxInstr];
  int16_t st[kMaxInstr];
  int sp = 0;
  for (int pc = 0; pc < p->ninstr; ++pc) {
    Node &x = n[pc];
    x = Node{0, -1, -1};
    switch (p->code[pc].op) {
      case OP_AND:
      case OP_OR:
        if (sp < 2) return -1;
        x = Node{(uint8_t)(p->code[pc].op == OP_AND ? 1 : 2), st[sp - 2], st[sp - 1]};
        sp -= 2;
        break;
      case OP_NOT:
        if (sp < 1) return -1;
        x = Node{3, st[sp - 1], -1};
        sp -= 1;
        break;
      case OP_TRUE: x.kind = 4; break;
      case OP_FALSE: x.kind = 5; break;
      case OP_JZ:
      case OP_JNZ: continue;   // skips work only
      default: break;
    }
    st[sp++] = (int16_t)pc;
  }
  if (sp != 1) return -1;
  Mask m[kMaxBoxes];
  const int k = expand(n, st[0], false, m, kMaxBoxes);
  for (int i = 0; i < k; ++i) {
    pos[i] = m[i].pos;
    neg[i] = m[i].neg;
  }
  return k;
}

namespace {

struct Box {
  uint32_t ref0, ref1;   // its tests in refs
  uint32_t pred;
};

struct HostOperand {
  int col, col2;      // table columns (col2 -1: the column itself)
  uint64_t m;         // udf modulus
  int64_t consts[6];  // udf: the program's constants (modulus, multiplier, shifts, 32-bit remainder)
  std::vector<int64_t> cuts;
};

uint32_t round16(uint64_t b) { return (uint32_t)((b + 15) & ~(uint64_t)15); }

}  // namespace

#ifdef ESC_CHECKED
std::atomic<uint32_t> g_shrink_table{0};   // esc_debug_shrink_table
#endif

// What a pass needs on the host; add_predicate adds to it.
struct BoxPlan {
  std::vector<HostOperand> ops;
  std::vector<BoxTest> tests;
  std::vector<uint32_t> refs;
  std::vector<Box> boxes;
  std::vector<int64_t> pool;
};

BoxPlan *new_box_plan() { return new BoxPlan; }
void free_box_plan(BoxPlan *p) { delete p; }

BoxFit add_predicate(BoxPlan *P, const esc_pred *p, uint32_t index) {
  uint64_t pos[kMaxBoxes], neg[kMaxBoxes];
  const int nb = predicate_boxes(p, pos, neg);
  if (nb < 0) return BOX_NEVER;
  if (P->boxes.size() + nb > (size_t)kMaxPassBoxes) return BOX_FULL;
  uint64_t used = 0;
  for (int i = 0; i < nb; ++i) used |= pos[i] | neg[i];
  // operands and tests of the instructions in use
  uint32_t test_of[kMaxInstr];
  const size_t ops0 = P->ops.size(), tests0 = P->tests.size(), pool0 = P->pool.size();
  for (int pc = 0; pc < p->ninstr; ++pc) {
    if (!((used >> pc) & 1u)) continue;
    const Instr &I = p->code[pc];
    HostOperand o{};
    o.col = p->ref_cols[I.ref];
    o.col2 = -1;
    if (I.op == OP_UDF) {
      o.col2 = p->ref_cols[I.ref2];
      if (o.col2 < o.col) std::swap(o.col, o.col2);   // the wrapped product commutes
      for (int k = 0; k < 6; ++k) o.consts[k] = p->pool[I.off + k];
      o.m = (uint64_t)o.consts[0];
    }
    size_t at = 0;
    while (at < P->ops.size() && !(P->ops[at].col == o.col && P->ops[at].col2 == o.col2 && P->ops[at].m == o.m)) ++at;
    if (at == P->ops.size()) {
      size_t udfs = 0;
      for (auto &x : P->ops) udfs += x.col2 >= 0;
      if (at >= (size_t)kMaxOperands || (o.col2 >= 0 && udfs >= (size_t)kMaxUdfOperands)) {
        P->ops.resize(ops0);   // (cuts already added to earlier operands only make empty intervals)
        P->tests.resize(tests0);
        P->pool.resize(pool0);
        return ops0 ? BOX_FULL : BOX_NEVER;
      }
      P->ops.push_back(std::move(o));
    }
    BoxTest bt{};
    bt.operand = (uint32_t)at;
    bt.op = I.op == OP_UDF ? (uint8_t)OP_RANGE : I.op;
    bt.lo = I.lo;
    bt.hi = I.hi;
    std::vector<int64_t> &cuts = P->ops[at].cuts;
    auto cut_value = [&](int64_t v) {
      cuts.push_back(v);
      if (v != INT64_MAX) cuts.push_back(v + 1);
    };
    if (I.op == OP_IN) {
      bt.off = (uint32_t)P->pool.size();
      bt.n = I.n;
      for (int k = 0; k < (int)I.n; ++k) {
        P->pool.push_back(p->pool[I.off + k]);
        cut_value(p->pool[I.off + k]);
      }
    } else if (I.op == OP_INSET) {
      bt.off = (uint32_t)P->pool.size();
      bt.n = I.n;
      for (int k = 0; k < 4; ++k) P->pool.push_back(p->pool[I.off + k]);
      for (int k = 0; k < (int)I.n; ++k) cut_value(p->pool[I.lo + k]);
    } else {
      if (I.lo != INT64_MIN) cuts.push_back(I.lo);
      if (I.hi != INT64_MAX) cuts.push_back(I.hi + 1);
    }
    test_of[pc] = (uint32_t)P->tests.size();
    P->tests.push_back(bt);
  }
  for (int i = 0; i < nb; ++i) {
    const size_t r0 = P->refs.size();
    for (uint64_t m = pos[i] | neg[i]; m; m &= m - 1) {
      const int pc = __builtin_ctzll(m);
      P->refs.push_back(test_of[pc] << 1 | (uint32_t)((neg[i] >> pc) & 1u));
    }
    P->boxes.push_back(Box{(uint32_t)r0, (uint32_t)P->refs.size(), index});
  }
  return BOX_ADDED;
}

namespace {

// Orders the boxes by which of the first four operands (those with the most
// cuts, whose bit rows come from L2) they test, so that a lane's 128 boxes
// mostly agree; lane_ops: the operands a lane's boxes test.
void sort_boxes(BoxPlan *P, std::vector<uint32_t> &lane_ops) {
  auto mask = [&](const Box &b) {
    uint32_t m = 0;
    for (uint32_t r = b.ref0; r < b.ref1; ++r) m |= 1u << P->tests[P->refs[r] >> 1].operand;
    return m;
  };
  std::vector<Box> sorted(P->boxes.size());
  std::vector<uint32_t> masks(P->boxes.size());
  size_t start[17] = {0};
  for (size_t b = 0; b < P->boxes.size(); ++b) {
    masks[b] = mask(P->boxes[b]);
    ++start[(masks[b] & 15u) + 1];
  }
  for (int k = 0; k < 16; ++k) start[k + 1] += start[k];
  for (size_t b = 0; b < P->boxes.size(); ++b) {
    const size_t at = start[masks[b] & 15u]++;
    sorted[at] = P->boxes[b];
    lane_ops[at / 128] |= masks[b];
  }
  P->boxes.swap(sorted);
}

// An operand's buckets, where they save at least two halvings (a bucket costs
// about as much as one): the smallest power-of-two width that gives at most
// `most` of them.  `cuts` in any order; appended to `out`.
void make_buckets(Operand &o, const std::vector<int64_t> &cuts, uint32_t most, std::vector<uint16_t> &out) {
  o.bsteps = ~0u;
  if (o.kind != OPD_32 || o.ncuts < 3 || o.ncuts > 65535 || most < 8) return;
  const auto mm = std::minmax_element(cuts.begin(), cuts.end());
  const int64_t base = *mm.first - 1, top = *mm.second;   // (cuts lie above the least 32-bit value)
  const uint64_t span = (uint64_t)(top - base);
  uint32_t shift = 0;
  while ((span >> shift) + 1 > most) ++shift;
  const uint32_t n = (uint32_t)(span >> shift) + 1;
  std::vector<uint32_t> before(n + 1, 0);   // cuts in buckets before each
  for (int64_t v : cuts) ++before[(size_t)((uint64_t)(v - base) >> shift) + 1];
  const uint32_t fullest = *std::max_element(before.begin(), before.end());
  uint32_t bsteps = 0;
  if (shift)
    while ((1ull << bsteps) - 1 < fullest) ++bsteps;
  if (bsteps + 2 > o.steps) return;
  for (uint32_t k = 0; k < n; ++k) before[k + 1] += before[k];
  o.bsteps = bsteps;
  o.base = (int32_t)base;
  o.top = (int32_t)top;
  o.shift = shift;
  o.bucket_off = (uint32_t)(out.size() * 2);
#ifdef ESC_CHECKED
  o.nbuckets = n;
#endif
  for (uint32_t k = 0; k < n; ++k) out.push_back((uint16_t)before[shift ? k : k + 1]);
}

}  // namespace

// (the blocks that run_boxes places, each for the most it can hold)
uint64_t box_scratch_bound(uint64_t n) {
  constexpr uint64_t kPredCuts = 2 * kMaxPool + 2 * kMaxInstr;   // a list's value makes two cuts, a range's bounds one each
  constexpr uint64_t kOthers = (uint64_t)kMaxOperands * 257;     // u8 operands; the interval below each one's cuts
  const uint64_t boxes = std::min<uint64_t>(n * kMaxBoxes, kMaxPassBoxes), words = (boxes + 31) / 32;
  // p predicates with cuts have as many boxes at least, and the more boxes the
  // fewer intervals fit the largest table
  uint64_t intervals = 0;
  for (uint64_t p = 0; p <= n; ++p)
    intervals = std::max(intervals, std::min(kOthers + kPredCuts * p, kMaxTableBytes / (4 * ((p + 31) / 32 + 3))));
  const uint64_t table = std::min(kMaxTableBytes, intervals * (words + 3) * 4);
  const uint64_t tests = n * kMaxInstr * sizeof(BoxTest), refs = n * kMaxBoxes * kMaxInstr * 4, pool = n * kMaxPool * 8;
  const uint64_t cuts = intervals * (8 + 16);   // unsorted; sorted and padded (to less than twice 8 bytes or 4 times 4)
  return table + tests + refs + pool + boxes * 13 + cuts + kBucketBytes + kMaxOperands * (sizeof(SortJob) + 32) + 16 * 256;
}

esc_status run_boxes(BoxPlan *P, const esc_table *t, int sms, unsigned long long *counts, ScratchHdr *hdr,
                     cudaStream_t st, bool *done) {
  *done = false;
  const uint32_t nboxes = (uint32_t)P->boxes.size();
  if (nboxes == 0) {   // every program is constant FALSE
    *done = true;
    return ESC_OK;
  }
  if (P->ops.empty()) return ESC_OK;   // no operand: left to the interpreter
  BoxLaunch L;
  std::memset(&L, 0, sizeof L);
  L.nop = (int32_t)P->ops.size();
  L.nopp = ((uint32_t)L.nop + 3u) & ~3u;
  L.nrows = (uint32_t)t->nrows;
  L.nboxes = nboxes;
  const uint32_t words = (nboxes + 31) / 32;
  // operands with the most cuts first: their tests leave the fewest boxes
  std::vector<uint32_t> order((size_t)L.nop), slot((size_t)L.nop);
  for (int c = 0; c < L.nop; ++c) order[c] = (uint32_t)c;
  std::stable_sort(order.begin(), order.end(),
                   [&](uint32_t x, uint32_t y) { return P->ops[x].cuts.size() > P->ops[y].cuts.size(); });
  for (int c = 0; c < L.nop; ++c) slot[order[c]] = (uint32_t)c;
  for (auto &x : P->tests) x.operand = slot[x.operand];
  for (auto &b : P->boxes)
    std::sort(P->refs.begin() + b.ref0, P->refs.begin() + b.ref1,
              [&](uint32_t x, uint32_t y) { return P->tests[x >> 1].operand < P->tests[y >> 1].operand; });
  std::vector<uint32_t> lane_ops((words + 3) / 4, 0u);
  sort_boxes(P, lane_ops);
  // intervals: sorted distinct cuts.  Few of them, or values of a small
  // domain, are sorted here (a 64K-entry set beats sorting many); the rest on
  // the GPU, where equal cuts stay.
  uint64_t intervals = 0, cut_bytes = 0;
  std::vector<SortJob> jobs;
  std::vector<int64_t> unsorted;
  std::vector<uint64_t> seen;
  auto column = [&](int col) {   // byte offset of a column in a stage
    const uint8_t *data = static_cast<const uint8_t *>(t->data[col]);
    for (int k = 0; k < L.ncol; ++k)
      if (L.col[k].data == data && L.col[k].w == (uint32_t)dtype_width(t->dtypes[col])) return L.col[k].off;
    StageColumn &c = L.col[L.ncol++];
    c = StageColumn{data, (uint32_t)dtype_width(t->dtypes[col]), L.stage_bytes};
    L.stage_bytes += c.w;   // (of one row; scaled to the tile below)
    return c.off;
  };
  size_t many = 0;
  for (auto &h : P->ops) many += h.cuts.size();
  const bool gpu_sort = many > 2048;
  uint32_t searched = 0;   // operands that may have buckets
  for (auto &h : P->ops) searched += h.col2 >= 0 || t->dtypes[h.col] != ESC_U8;
  uint32_t most_buckets = kMaxBuckets;
  while (most_buckets * searched * 2 > kBucketBytes) most_buckets /= 2;
  std::vector<uint16_t> buckets;
  std::vector<uint32_t> padded_cuts((size_t)L.nop);
  for (int c = 0; c < L.nop; ++c) {
    HostOperand &h = P->ops[order[c]];
    Operand &o = L.op[c];
    SortJob *job = nullptr;
    o.a = column(h.col);
    o.b = h.col2 >= 0 ? column(h.col2) : ~0u;
    o.da = t->dtypes[h.col];
    int64_t lo = INT32_MIN, hi = INT32_MAX;   // values the operand takes (32-bit search)
    if (h.col2 >= 0) {
      o.db = t->dtypes[h.col2];
      o.d = h.m;
      o.mult = (uint64_t)h.consts[1];
      o.sh1 = (int32_t)h.consts[2];
      o.sh2 = (int32_t)h.consts[3];
      o.M = (uint64_t)h.consts[4];
      o.K = (uint32_t)h.consts[5];
      o.kind = h.m <= (uint64_t)INT32_MAX ? OPD_32 : OPD_64;
      if (o.kind == OPD_32) {
        lo = 1 - (int64_t)h.m;
        hi = (int64_t)h.m - 1;
      }
    } else {
      o.kind = o.da == ESC_U8 ? OPD_U8 : o.da == ESC_I64 ? OPD_64 : OPD_32;
      if (o.da == ESC_U16) {
        lo = 0;
        hi = 65535;
      }
    }
    if (o.kind == OPD_U8) {
      h.cuts.clear();
    } else {
      if (o.kind == OPD_64 && h.col2 < 0 &&
          std::all_of(h.cuts.begin(), h.cuts.end(), [](int64_t v) { return v > INT32_MIN && v <= INT32_MAX; }))
        o.kind = OPD_32;
      if (o.kind == OPD_32)   // cuts past the last value separate nothing
        h.cuts.erase(std::remove_if(h.cuts.begin(), h.cuts.end(), [&](int64_t v) { return v > hi || v <= lo; }),
                     h.cuts.end());
      if (o.kind == OPD_32 && hi - lo < 65536 && h.cuts.size() > 256) {
        seen.assign(1024 + 1, 0);
        for (int64_t v : h.cuts) seen[(size_t)((v - lo) >> 6)] |= 1ull << ((v - lo) & 63);
        h.cuts.clear();
        for (size_t w = 0; w < seen.size(); ++w)
          for (uint64_t m = seen[w]; m; m &= m - 1) h.cuts.push_back(lo + (int64_t)(w * 64) + __builtin_ctzll(m));
      } else if (!gpu_sort || h.cuts.size() <= 64) {
        std::sort(h.cuts.begin(), h.cuts.end());
        h.cuts.erase(std::unique(h.cuts.begin(), h.cuts.end()), h.cuts.end());
      } else {
        jobs.push_back(SortJob{(uint32_t)unsorted.size(), (uint32_t)h.cuts.size(), 0, 0, 0});
        job = &jobs.back();
        unsorted.insert(unsorted.end(), h.cuts.begin(), h.cuts.end());
      }
    }
    o.ncuts = (uint32_t)h.cuts.size();
    while ((1ull << o.steps) - 1 < o.ncuts) ++o.steps;
    uint32_t per_cut = 8;
    while (per_cut < o.ncuts * kBucketsPerCut) per_cut *= 2;
    make_buckets(o, h.cuts, std::min(most_buckets, per_cut), buckets);
    // every halving reads inside the padding, also those that start at a bucket's first cut
    const uint32_t padded = std::max((1u << o.steps) - 1, o.bsteps == ~0u ? 0u : o.ncuts + (1u << o.bsteps) - 1);
    const uint32_t w = o.kind == OPD_64 ? 8u : 4u;
    padded_cuts[c] = padded;
#ifdef ESC_CHECKED
    o.padded = padded;
#endif
    o.cut_off = (uint32_t)cut_bytes;
    if (job) {
      job->padded = padded;
      job->dst_off = o.cut_off;
      job->wide = w == 8;
    }
    cut_bytes += o.kind == OPD_U8 ? 0 : round16((uint64_t)padded * w);
    o.table_off = (uint32_t)intervals;   // (in bit rows; scaled below)
    intervals += o.kind == OPD_U8 ? 256u : o.ncuts + 1u;
  }
  if (intervals * (words + 3) * 4 > kMaxTableBytes) return ESC_OK;   // too large to pay: the caller interprets
  L.cut_bytes = round16(cut_bytes);
  L.bucket_bytes = round16(buckets.size() * 2);
  // shared memory, and with it the kernel: rows in registers when the boxes
  // fit a thread's words and cuts and table fit beside the stages
  const uint32_t row_bytes = L.stage_bytes;
  uint32_t smem = 0;
  auto take = [&](uint64_t bytes) {
    const uint32_t at = smem;
    smem += round16(bytes);
    return at;
  };
  auto layout = [&](uint32_t tile) {
    L.tile = tile;
    L.stage_bytes = row_bytes * tile;
    smem = 0;
    take((uint64_t)kBoxStages * L.stage_bytes);
    L.smem_cnt = take((uint64_t)nboxes * 4);
    L.smem_bar = take(kBoxStages * 8);
  };
  layout(kRows * kBoxThreads);
  int vec = words <= 1 ? 1 : words <= 2 ? 2 : 4;
  uint64_t table_bytes = intervals * vec * 4;
  const bool by_row = words <= 4 && L.cut_bytes <= kCutSmem && table_bytes <= kTableSmem &&
                      smem + L.cut_bytes + table_bytes + L.bucket_bytes + 48 <= (uint64_t)kMaxBoxSmem;
  if (by_row) {
    L.smem_cut = take(L.cut_bytes);
    L.smem_table = take(table_bytes);
    L.smem_bucket = take(L.bucket_bytes);
  } else {
    vec = 4;
    L.lanes = 1;
    while (L.lanes < 32 && L.lanes * 4 < words) L.lanes *= 2;
    L.chunks = (words + 4 * L.lanes - 1) / (4 * L.lanes);
    table_bytes = intervals * ((words + 3) & ~3u) * 4;
    layout(kTile);
    L.smem_offs = take((uint64_t)kTile * L.nopp * 4);
    if (smem + L.bucket_bytes > (uint32_t)kMaxBoxSmem) {   // (16 i64 columns, 24 operands, 8192 boxes leave 12,272 bytes)
      L.bucket_bytes = 0;
      for (int c = 0; c < L.nop; ++c) L.op[c].bsteps = ~0u;
    }
    L.smem_bucket = take(L.bucket_bytes);
    if (L.cut_bytes <= kCutSmem && smem + L.cut_bytes <= (uint32_t)kMaxBoxSmem) {
      L.cuts_in_smem = 1;
      L.smem_cut = take(L.cut_bytes);
    }
  }
  L.stride = (words + vec - 1) / vec * vec * 4;
  L.table_bytes = (uint32_t)table_bytes;
  for (int k = 0; k < L.ncol; ++k) L.col[k].off *= L.tile;
  for (int c = 0; c < L.nop; ++c) {
    L.op[c].table_off *= L.stride;
    L.op[c].a *= L.tile;
    if (L.op[c].b != ~0u) L.op[c].b *= L.tile;
  }

  // one device block: uploaded arrays | cuts | table
  uint64_t at = 0;
  auto place = [&](uint64_t bytes) {
    const uint64_t a = at;
    at += (bytes + 255) & ~(uint64_t)255;
    return a;
  };
  const uint64_t a_tests = place(P->tests.size() * sizeof(BoxTest)), a_refs = place(P->refs.size() * 4 + 4),
                 a_box = place((uint64_t)nboxes * 8), a_pred = place((uint64_t)nboxes * 4),
                 a_lane = place(lane_ops.size() * 4),
                 a_pool = place(P->pool.size() * 8 + 8), a_jobs = place(jobs.size() * sizeof(SortJob) + 4),
                 a_uns = place(unsorted.size() * 8 + 8), a_buckets = place(buckets.size() * 2 + 16),
                 a_cuts = place(L.cut_bytes + 16), upload = at,
                 a_table = place(round16(table_bytes));
  HostStage stage(upload, st);   // (throws without host memory: before there is device memory to give back)
  void *mem = nullptr;
  esc_status s = alloc_async(&mem, at, st);
  if (s != ESC_OK) return s;
  uint8_t *dev = static_cast<uint8_t *>(mem);
  uint8_t *h = stage.data();
  auto put = [&](uint64_t a, const void *src, size_t bytes) {
    if (bytes) std::memcpy(h + a, src, bytes);
  };
  put(a_tests, P->tests.data(), P->tests.size() * sizeof(BoxTest));
  put(a_refs, P->refs.data(), P->refs.size() * 4);
  for (uint32_t b = 0; b < nboxes; ++b) {
    put(a_box + 8ull * b, &P->boxes[b], 8);   // ref0, ref1
    put(a_pred + 4ull * b, &P->boxes[b].pred, 4);
  }
  put(a_lane, lane_ops.data(), lane_ops.size() * 4);
  put(a_pool, P->pool.data(), P->pool.size() * 8);
  put(a_jobs, jobs.data(), jobs.size() * sizeof(SortJob));
  put(a_uns, unsorted.data(), unsorted.size() * 8);
  put(a_buckets, buckets.data(), buckets.size() * 2);
  for (int c = 0; c < L.nop; ++c) {   // cuts sorted here, padded (those sorted on the GPU are overwritten there)
    const Operand &o = L.op[c];
    if (o.kind == OPD_U8) continue;
    const std::vector<int64_t> &cuts = P->ops[order[c]].cuts;
    const uint32_t padded = padded_cuts[c];
    for (uint32_t k = 0; k < padded; ++k) {
      if (o.kind == OPD_64) {
        const int64_t v = k < o.ncuts ? cuts[k] : INT64_MAX;
        std::memcpy(h + a_cuts + o.cut_off + 8ull * k, &v, 8);
      } else {
        const int32_t v = k < o.ncuts ? (int32_t)cuts[k] : INT32_MAX;
        std::memcpy(h + a_cuts + o.cut_off + 4ull * k, &v, 4);
      }
    }
  }
  L.cuts = dev + a_cuts;
  L.table = dev + a_table;
  L.buckets = dev + a_buckets;
  L.lane_ops = reinterpret_cast<const uint32_t *>(dev + a_lane);
  L.pred_of_box = reinterpret_cast<const uint32_t *>(dev + a_pred);
  L.counts = counts;
  L.hdr = hdr;
  cudaError_t e = stage.copy_to(dev);
  if (e == cudaSuccess && !jobs.empty()) {
    uint32_t most = 0;
    for (auto &j : jobs) most = std::max(most, j.padded);
    sort_cuts_kernel<<<dim3((most + kSortCuts - 1) / kSortCuts, (unsigned)jobs.size()), 1024, 0, st>>>(
        reinterpret_cast<const int64_t *>(dev + a_uns), reinterpret_cast<const SortJob *>(dev + a_jobs), dev + a_cuts,
        hdr);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    uint32_t most = 1;
    for (int c = 0; c < L.nop; ++c) most = std::max(most, L.op[c].kind == OPD_U8 ? 256u : L.op[c].ncuts + 1u);
    const BuildArgs B{reinterpret_cast<const BoxTest *>(dev + a_tests), reinterpret_cast<const uint32_t *>(dev + a_refs),
                      reinterpret_cast<const uint2 *>(dev + a_box), reinterpret_cast<const int64_t *>(dev + a_pool)};
    build_kernel<<<dim3((L.stride / 4 + 7) / 8, (unsigned)L.nop, (most + kBuildRun - 1) / kBuildRun), 256, 0, st>>>(L, B);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    if (by_row) L.table_bytes = round16(table_bytes);   // what the kernel copies
#ifdef ESC_CHECKED
    L.table_bytes -= std::min(g_shrink_table.load(), L.table_bytes / 16) * 16;
#endif
    const uint32_t fit = std::max<uint32_t>(1, (227u * 1024) / (smem + 1024));
    const uint32_t ctas = std::min<uint32_t>(fit, vec == 4 ? 2 : 3);
    const uint32_t grid = std::min<uint32_t>((uint32_t)sms * ctas, (L.nrows + L.tile - 1) / L.tile);
    const void *fn = !by_row ? reinterpret_cast<const void *>(box_words_kernel)
                     : vec == 1 ? reinterpret_cast<const void *>(box_rows_kernel<1>)
                     : vec == 2 ? reinterpret_cast<const void *>(box_rows_kernel<2>)
                                : reinterpret_cast<const void *>(box_rows_kernel<4>);
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxBoxSmem);
    void *args[] = {&L};
    if (e == cudaSuccess) e = cudaLaunchKernel(fn, dim3(grid), dim3(kBoxThreads), args, smem, st);
  }
  cudaFreeAsync(mem, st);
  if (e != cudaSuccess) return fail(ESC_ECUDA, std::string("shared scan by table lookup: ") + cudaGetErrorString(e));
  *done = true;
  return ESC_OK;
}

}  // namespace esc

extern "C" esc_status esc_debug_shrink_table(uint32_t chunks) {
#ifdef ESC_CHECKED
  esc::g_shrink_table.store(chunks);
  esc::clear_error();
  return ESC_OK;
#else
  (void)chunks;
  return esc::fail(ESC_EINVAL, "esc_debug_shrink_table: only in the checked build");
#endif
}
