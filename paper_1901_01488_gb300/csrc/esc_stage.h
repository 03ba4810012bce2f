// Host memory from which a call's arrays are copied to the device without
// waiting for the stream: an asynchronous copy of more than 64 KB from
// pageable memory returns only after the work before it has run, so that
// calls could not overlap.  Pinned blocks come from a pool per device, bounded
// (8 of 256 KB, 4 of 4 MB), each reused once the copy it served has completed
// (an event).  Without a free block, for arrays up to 64 KB or larger than a
// block, and while the stream is being captured, the memory is ordinary.
#pragma once
#include <cuda_runtime.h>

#include <stddef.h>
#include <stdint.h>

#include <memory>

namespace esc {

// Event and allocation calls are refused to every thread while one captures a
// stream in global mode; these touch no capturing stream.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

struct StageBlock;

class HostStage {
 public:
  HostStage(size_t bytes, cudaStream_t st);
  ~HostStage();
  HostStage(const HostStage &) = delete;
  HostStage &operator=(const HostStage &) = delete;
  uint8_t *data() { return data_; }
  // Enqueues the copy of all bytes to `dev`; the host memory may not change after it.
  cudaError_t copy_to(void *dev);

 private:
  size_t bytes_;
  cudaStream_t st_;
  StageBlock *block_ = nullptr;
  std::unique_ptr<uint8_t[]> own_;
  uint8_t *data_;
};

}  // namespace esc
