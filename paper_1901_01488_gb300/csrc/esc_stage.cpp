// Pool of pinned host blocks (see esc_stage.h).
#include "esc_stage.h"

#include <mutex>
#include <new>

#include "esc_internal.h"

namespace esc {

struct StageBlock {
  uint8_t *mem = nullptr;
  cudaEvent_t copied = nullptr;
  bool busy = false;   // held by a call
};

namespace {

// Copies up to 64 KB from ordinary memory do not wait for the stream.
constexpr size_t kInlineBytes = (size_t)64 << 10;
constexpr int kSmall = 8, kLarge = 4, kDevices = 64;
constexpr size_t kSmallBytes = (size_t)256 << 10, kLargeBytes = (size_t)4 << 20;

std::mutex g_mu;
struct Pool {
  StageBlock small[kSmall], large[kLarge];
} g_pool[kDevices];

StageBlock *acquire(size_t bytes, cudaStream_t st) {
  if (bytes <= kInlineBytes || bytes > kLargeBytes) return nullptr;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return nullptr;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return nullptr;
  const bool is_small = bytes <= kSmallBytes;
  RelaxedCapture relaxed;
  std::lock_guard<std::mutex> lk(g_mu);
  StageBlock *b = is_small ? g_pool[dev].small : g_pool[dev].large;
  const int n = is_small ? kSmall : kLarge;
  for (int i = 0; i < n; ++i) {
    if (b[i].busy) continue;
    if (b[i].mem) {
      const cudaError_t e = cudaEventQuery(b[i].copied);
      if (e != cudaSuccess) {
        if (e == cudaErrorNotReady) cudaGetLastError();
        continue;
      }
    } else {
      void *p = nullptr;
      if (cudaEventCreateWithFlags(&b[i].copied, cudaEventDisableTiming) != cudaSuccess ||
          cudaHostAlloc(&p, is_small ? kSmallBytes : kLargeBytes, cudaHostAllocPortable) != cudaSuccess) {
        cudaGetLastError();
        if (b[i].copied) cudaEventDestroy(b[i].copied);
        b[i].copied = nullptr;
        return nullptr;
      }
      b[i].mem = static_cast<uint8_t *>(p);
    }
    b[i].busy = true;
    return &b[i];
  }
  return nullptr;
}

}  // namespace

HostStage::HostStage(size_t bytes, cudaStream_t st) : bytes_(bytes), st_(st) {
  if (inject_host_failure()) throw std::bad_alloc();
  block_ = acquire(bytes, st);
  if (!block_) own_.reset(new uint8_t[bytes ? bytes : 1]);
  data_ = block_ ? block_->mem : own_.get();
}

HostStage::~HostStage() {
  if (!block_) return;
  std::lock_guard<std::mutex> lk(g_mu);
  block_->busy = false;
}

cudaError_t HostStage::copy_to(void *dev) {
  const cudaError_t e = cudaMemcpyAsync(dev, data_, bytes_, cudaMemcpyHostToDevice, st_);
  if (e != cudaSuccess || !block_) return e;
  const cudaError_t r = cudaEventRecord(block_->copied, st_);
  if (r != cudaSuccess) cudaStreamSynchronize(st_);   // the block must not be reused before the copy
  return r;
}

}  // namespace esc
