// Exact semi-join cardinalities over dense keys: the COUNT(*) foreign-key
// join queries of the paper's overhead experiments (Sec. 3.1: lineitem joined
// with a filtered orders / part / supplier table) generalised to a star
// schema.  One pass over the fact table's foreign-key columns: a row matches in
// dimension d when 0 <= fk_d < D_d and bit fk_d of bitmap_d is set, and for
// every dimension subset S,
//   count(S) = |{ rows that match in all of S }|.
//
// Kernel shape: persistent grid of one block per SM (shared memory sized to the
// bitmaps it holds, the rest of the SM's on-chip memory left to L1); a warp
// streams 256 rows per step, 512 consecutive bytes per non-allocating load of a
// foreign-key column, 8 rows a lane.  The kernel is specialised on how many
// bitmaps sit in shared memory (dimensions are ordered smallest bitmap first,
// so the shared ones come first): each probe is then a fixed sequence -- clamp
// the word index, load, two funnel shifts that append the key's bit to the
// lane's bits of that dimension.  Every 32 rows the subsets' bits are ANDed and
// counted (15 popcounts for four dimensions).
// What bounds it: L1's data pipe (it was 92 % busy with 32 bytes per lane and
// load, which read every sector twice) for large bitmaps, HBM next.  Measured
// at 120M rows, before (each lane 8 consecutive rows, 16 byte counters per
// thread, 512 threads) and now: dimensions of 2M, 200K, 30K and 2,556 rows 373
// -> 320 us a call, one of 2M 200 -> 149, 900K and 30K 209 -> 162, 8M and 2M
// 714 -> 712.  By threads per block: four dimensions 512 / 640 / 768 / 1024:
// 360 / 329 / 320 / 328; one: 183 / 161 / 151 / 149.  Holding part of a large
// bitmap in shared memory did not help (a gather there costs what one in L1
// does).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>

#include "esc_internal.h"
#include "esc_ptx.cuh"

namespace esc {

constexpr uint32_t kSjWarpRows = 256;   // rows a warp takes per step: 8 per lane
// Threads of a block (one per SM; measured above): more where few dimensions leave registers.
constexpr uint32_t sj_threads(int ndims) { return ndims <= 2 ? 1024 : 768; }
constexpr int kSjMaxDims = 4;
constexpr uint32_t kSjSmemBitmapBytes = 96 * 1024;  // shared copies of the smaller bitmaps

struct SjParams {
  const int32_t *fk[kSjMaxDims];       // in probe order
  const uint32_t *bitmap[kSjMaxDims];
  uint32_t dim_rows[kSjMaxDims];
  uint32_t smem_off[kSjMaxDims];       // word offset in shared memory (the first NS dimensions)
  uint32_t words[kSjMaxDims];
  int32_t ndims;
  uint32_t nrows;
  unsigned long long *hist;            // 16 subset counts, zeroed
  ScratchHdr *hdr;                     // launch header (zeroed): blocks done, the checked build's findings
  HostResult *result;                  // hist and hdr are a call slot: the last block reports here and clears them
  unsigned long long seq;              // for result
  uint32_t smem_words;                 // shared-memory words the launch has (checked build)
};

__device__ __forceinline__ int4 ld_stream(const int32_t *p) {
  int4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// The word that holds bit `key` of a bitmap of `rows` bits; a word whose bit
// is 0 when key is out of range (negative keys wrap to large unsigned values).
// A shared-memory copy ends with a zero word at index `wlast` and has the bits
// past `rows` cleared, so clamping the word index is the whole bounds test
// there; a bitmap read in place is tested explicitly.
__device__ __forceinline__ uint32_t probe_word(const uint32_t *bm, uint32_t key, uint32_t rows, uint32_t wlast,
                                               bool shared) {
  if (shared) return bm[min(key >> 5, wlast)];
  const uint32_t w = __ldg(&bm[min(key >> 5, wlast)]);
  return key < rows ? w : 0u;
}

// The same, in the checked build: the word index is tested against the
// bitmap's words (in shared memory: its copy and the zero word).
__device__ __forceinline__ uint32_t probe_word_checked(const uint32_t *bm, uint32_t key, uint32_t rows, uint32_t wlast,
                                                       bool shared, uint32_t words, ScratchHdr *hdr) {
  const uint32_t wi = min(key >> 5, wlast);
  if (!ESC_INB(hdr, wi < (shared ? words + 1 : words), 32, wi)) return 0u;
  return probe_word(bm, key, rows, wlast, shared);
}

// A thread's rows as bits: bits[d] collects the rows' matches in dimension d,
// 32 rows at most; count() adds, for every subset of the dimensions, the rows
// that match all of it.
template <int ND, int NS>
struct RowBits {
  uint32_t bits[ND] = {};
  uint32_t n[1 << ND] = {};   // by subset (0: unused)

  __device__ __forceinline__ void row(const SjParams &P, const uint32_t *const (&bm)[ND], const uint32_t (&wmax)[ND],
                                      const int32_t (&k)[ND]) {
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const uint32_t key = (uint32_t)k[d];
#ifdef ESC_CHECKED
      const uint32_t w = probe_word_checked(bm[d], key, P.dim_rows[d], wmax[d], d < NS, P.words[d], P.hdr);
#else
      const uint32_t w = probe_word(bm[d], key, P.dim_rows[d], wmax[d], d < NS);
#endif
      // the key's bit to the top of the word, and from there into the collected ones
      bits[d] = __funnelshift_l(__funnelshift_l(w, w, ~key), bits[d], 1);
    }
  }
  __device__ __forceinline__ void count() {
    uint32_t s[1 << ND];
#pragma unroll
    for (int v = 1; v < (1 << ND); ++v) {
      const int low = v & -v, rest = v ^ low;   // the subset without its first dimension
      const int d = low == 1 ? 0 : low == 2 ? 1 : low == 4 ? 2 : 3;
      s[v] = rest ? s[rest] & bits[d] : bits[d];
      n[v] += __popc(s[v]);
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) bits[d] = 0;
  }
};

template <int ND, int NS>
__global__ void __launch_bounds__(sj_threads(ND), 1) semijoin_kernel(const __grid_constant__ SjParams P) {
  extern __shared__ __align__(16) uint32_t sbm[];
  __shared__ unsigned int bins[16];
#pragma unroll
  for (int d = 0; d < NS; ++d) {
    // the words (bits past the last row cleared) and a zero word
    const uint32_t tail = P.dim_rows[d] & 31u;
    for (uint32_t w = threadIdx.x; w <= P.words[d]; w += blockDim.x) {
      uint32_t x = w < P.words[d] ? P.bitmap[d][w] : 0u;
      if (w + 1 == P.words[d] && tail) x &= (1u << tail) - 1u;
      if (ESC_INB(P.hdr, P.smem_off[d] + w < P.smem_words, 31, P.smem_off[d] + w)) sbm[P.smem_off[d] + w] = x;
    }
  }
  if (threadIdx.x < 16) bins[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t *bm[ND];
  uint32_t wmax[ND];
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    bm[d] = d < NS ? sbm + P.smem_off[d] : P.bitmap[d];
    wmax[d] = d < NS ? P.words[d] : P.words[d] - 1u;  // shared: the zero word; global: words >= 1
  }

  RowBits<ND, NS> R;
  // A warp's loads are 512 consecutive bytes: lane l takes rows 4l .. 4l + 3 of
  // either half of the warp's 256 rows.
  const uint32_t nchunks = P.nrows / kSjWarpRows;
  const uint32_t stride = gridDim.x * (blockDim.x / 32);
  uint32_t steps = 0;
  for (uint32_t ch = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); ch < nchunks; ch += stride) {
    const uint32_t r0 = ch * kSjWarpRows + 4u * (threadIdx.x & 31u);
    if (ESC_INB(P.hdr, (uint64_t)r0 + 132 <= P.nrows, 30, r0)) {
      int4 v[ND][2];
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int q = 0; q < 2; ++q) v[d][q] = ld_stream(P.fk[d] + (size_t)r0 + 128 * q);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        int32_t k0[ND], k1[ND], k2[ND], k3[ND];
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          k0[d] = v[d][q].x;
          k1[d] = v[d][q].y;
          k2[d] = v[d][q].z;
          k3[d] = v[d][q].w;
        }
        R.row(P, bm, wmax, k0);
        R.row(P, bm, wmax, k1);
        R.row(P, bm, wmax, k2);
        R.row(P, bm, wmax, k3);
      }
    }
    if ((++steps & 3u) == 0) R.count();   // 32 rows
  }
  R.count();
  // ragged tail: rows nchunks*256 .. nrows-1, one per thread of block 0
  if (blockIdx.x == 0) {
    const uint32_t r = nchunks * kSjWarpRows + threadIdx.x;   // nrows <= 2^32 - 2^16: no overflow
    if (r < P.nrows) {
      int32_t k[ND];
#pragma unroll
      for (int d = 0; d < ND; ++d) k[d] = P.fk[d][r];
      R.row(P, bm, wmax, k);
    }
    R.count();
  }
#pragma unroll
  for (int v = 1; v < (1 << ND); ++v) {
    const uint32_t t = __reduce_add_sync(0xffffffffu, R.n[v]);
    if ((threadIdx.x & 31) == 0 && t) atomicAdd(&bins[v], t);
  }
  __syncthreads();
  if (threadIdx.x < 16 && bins[threadIdx.x]) atomicAdd(&P.hist[threadIdx.x], (unsigned long long)bins[threadIdx.x]);
  if (P.result && threadIdx.x < 32) {
    __threadfence();
    __syncwarp();
    uint32_t last = 0;
    if (threadIdx.x == 0) last = atomicAdd(&P.hdr->blocks_done, 1u) == gridDim.x - 1u;
    if (__shfl_sync(0xffffffffu, last, 0)) {
      __threadfence();
      if (threadIdx.x < 16) {
        P.result->hist[threadIdx.x] = atomicAdd(&P.hist[threadIdx.x], 0ull);
        P.hist[threadIdx.x] = 0;
      }
      if (threadIdx.x == 0) {
        P.result->status = 0;   // (the release build's kernel raises none)
        *P.hdr = ScratchHdr{};
      }
      __threadfence_system();   // the slot is clear before the host can know
      __syncwarp();
      if (threadIdx.x == 0) *(volatile unsigned long long *)&P.result->seq = P.seq;
    }
  }
}

template <int ND, int NS>
cudaError_t launch_semijoin(const SjParams &P, size_t smem, int sms, cudaStream_t st) {
  static std::once_flag once[64];
  static cudaError_t attr[64];
  int dev = 0;
  cudaGetDevice(&dev);
  std::call_once(once[dev & 63], [&] {
    attr[dev & 63] = cudaFuncSetAttribute(semijoin_kernel<ND, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)kSjSmemBitmapBytes);
    // as much L1 as the launch leaves: a bitmap probed in place (too large for
    // shared memory) is then mostly served from L1 (its hot words: Zipf keys)
    if (attr[dev & 63] == cudaSuccess)
      attr[dev & 63] = cudaFuncSetAttribute(semijoin_kernel<ND, NS>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                            (int)cudaSharedmemCarveoutMaxL1);
  });
  if (attr[dev & 63] != cudaSuccess) return attr[dev & 63];
  constexpr uint32_t threads = sj_threads(ND);
  const uint32_t chunks = P.nrows / kSjWarpRows;
  const int grid = std::max(1, std::min<int>(sms, (int)((chunks + threads / 32 - 1) / (threads / 32))));
  semijoin_kernel<ND, NS><<<grid, threads, smem, st>>>(P);
  return cudaGetLastError();
}

template <int ND>
cudaError_t launch_nd(const SjParams &P, int ns, size_t smem, int sms, cudaStream_t st) {
  switch (ns) {
    case 0: return launch_semijoin<ND, 0>(P, smem, sms, st);
    case 1: return launch_semijoin<ND, (ND >= 1 ? 1 : 0)>(P, smem, sms, st);
    case 2: return launch_semijoin<ND, (ND >= 2 ? 2 : 0)>(P, smem, sms, st);
    case 3: return launch_semijoin<ND, (ND >= 3 ? 3 : 0)>(P, smem, sms, st);
    default: return launch_semijoin<ND, ND>(P, smem, sms, st);
  }
}

// Stream-ordered allocation from the library's device pool (esc_scan.cu).
esc_status alloc_async(void **p, size_t bytes, cudaStream_t st);

}  // namespace esc

using namespace esc;

extern "C" esc_status esc_semijoin_counts(const esc_table *fact, const char *const *fk_cols, int32_t ndims,
                                          const uint32_t *const *dev_bitmaps, const uint64_t *dim_rows,
                                          uint64_t *subset_counts, void *stream) {
  ESC_RANGE("esc_semijoin_counts");
  if (!fact || !fk_cols || !dev_bitmaps || !dim_rows || !subset_counts)
    return fail(ESC_EINVAL, "esc_semijoin_counts: NULL argument");
  if (ndims < 1 || ndims > kSjMaxDims) return fail(ESC_EINVAL, "esc_semijoin_counts: ndims must be 1..4");
  SjParams P;
  std::memset(&P, 0, sizeof P);
  P.ndims = ndims;
  P.nrows = (uint32_t)fact->nrows;
  const int32_t *fk[kSjMaxDims];
  uint32_t words[kSjMaxDims];
  for (int d = 0; d < ndims; ++d) {
    if (!fk_cols[d]) return fail(ESC_EINVAL, "esc_semijoin_counts: NULL column name");
    int c = -1;
    for (size_t i = 0; i < fact->names.size(); ++i)
      if (fact->names[i] == fk_cols[d]) c = (int)i;
    if (c < 0) return fail(ESC_EINVAL, std::string("esc_semijoin_counts: unknown column ") + fk_cols[d]);
    if (fact->dtypes[c] != ESC_I32) return fail(ESC_ETYPE, "esc_semijoin_counts: foreign keys must be i32");
    for (int e = 0; e < d; ++e)
      if (fk[e] == fact->data[c]) return fail(ESC_EINVAL, "esc_semijoin_counts: repeated foreign-key column");
    if (dim_rows[d] >= (1ull << 32)) return fail(ESC_EINVAL, "esc_semijoin_counts: dimension too large");
    if (dim_rows[d] > 0 && !dev_bitmaps[d]) return fail(ESC_EINVAL, "esc_semijoin_counts: NULL bitmap");
    fk[d] = static_cast<const int32_t *>(fact->data[c]);
    words[d] = (uint32_t)((dim_rows[d] + 31) / 32);
  }
  // probe order: smallest bitmap first; a prefix of them goes to shared memory
  int order[kSjMaxDims] = {0, 1, 2, 3};
  std::stable_sort(order, order + ndims, [&](int a, int b) { return words[a] < words[b]; });
  uint32_t smem_words = 0;
  int ns = 0;
  for (int i = 0; i < ndims; ++i) {
    const int d = order[i];
    P.fk[i] = fk[d];
    P.bitmap[i] = dev_bitmaps[d];
    P.dim_rows[i] = (uint32_t)dim_rows[d];
    P.words[i] = words[d];
    P.smem_off[i] = ~0u;
    // shared copy: the words and a zero word (an empty dimension is that word alone)
    if (ns == i && (uint64_t)(smem_words + words[d] + 1) * 4 <= kSjSmemBitmapBytes) {
      P.smem_off[i] = smem_words;
      smem_words += (words[d] + 1 + 3) & ~3u;
      ++ns;
    }
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // a call slot, or scratch from the library's device pool (memory stays
  // reserved between calls): 16 counts, then the launch header
  void *mem = nullptr;
  SlotRef slot;
  const bool in_slot = take_slot(st, &slot);
  cudaError_t e = cudaSuccess;
  if (in_slot) {
    if (inject_alloc_failure()) {
      give_slot(slot);
      return fail(ESC_ENOMEM, "device scratch allocation: injected failure (esc_debug_fail_allocs)");
    }
    P.hist = slot.dev->hist;
    P.hdr = &slot.dev->hdr;
    P.result = slot.host_dev;
    P.seq = slot.seq;
  } else {
    if (esc_status as = alloc_async(&mem, 16 * 8 + sizeof(ScratchHdr), st); as != ESC_OK) return as;
    e = cudaMemsetAsync(mem, 0, 16 * 8 + sizeof(ScratchHdr), st);
    P.hist = static_cast<unsigned long long *>(mem);
    P.hdr = reinterpret_cast<ScratchHdr *>(static_cast<uint8_t *>(mem) + 16 * 8);
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = (size_t)std::max<uint32_t>(smem_words, 4) * 4;
  P.smem_words = (uint32_t)(smem / 4);
  if (e == cudaSuccess) {
    switch (ndims) {
      case 1: e = launch_nd<1>(P, ns, smem, sms, st); break;
      case 2: e = launch_nd<2>(P, ns, smem, sms, st); break;
      case 3: e = launch_nd<3>(P, ns, smem, sms, st); break;
      default: e = launch_nd<4>(P, ns, smem, sms, st); break;
    }
  }
  struct {
    unsigned long long h[16];
    ScratchHdr hdr;
  } back;
  unsigned long long *h = back.h;
  if (e == cudaSuccess && !in_slot) e = cudaMemcpyAsync(&back, mem, sizeof back, cudaMemcpyDeviceToHost, st);
  if (mem) cudaFreeAsync(mem, st);
  if (e == cudaSuccess && !(in_slot && poll_slot(slot))) e = cudaStreamSynchronize(st);
  // (after a failure the slot stays taken: its launch may still be running)
  if (e != cudaSuccess) return fail(ESC_ECUDA, std::string("esc_semijoin_counts: ") + cudaGetErrorString(e));
  if (in_slot) {
    std::memcpy(back.h, slot.host->hist, sizeof back.h);
    back.hdr.status = slot.host->status;
    give_slot(slot);
  }
  if (back.hdr.status != 0) return device_status(back.hdr, "esc_semijoin_counts");
  // subsets are in probe order (bit i = dimension order[i]): back to the caller's bits
  subset_counts[0] = fact->nrows;
  for (uint32_t v = 1; v < (1u << ndims); ++v) {
    uint32_t S = 0;
    for (int i = 0; i < ndims; ++i) S |= ((v >> i) & 1u) << order[i];
    subset_counts[S] = h[v];
  }
  clear_error();
  return ESC_OK;
}
