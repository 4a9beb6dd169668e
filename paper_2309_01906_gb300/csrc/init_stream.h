// init_stream.h — device state that is ready before its first use on any stream.
#pragma once

#include <cuda_runtime.h>

namespace hp {

// Clears and fills fresh device memory on a stream of its own; after wait() it is
// ready for every stream.  cudaMemset, and cudaMemcpy from pageable memory, are
// queued on the legacy stream and may still be pending when they return, behind
// whatever the program has queued there, and streams created non-blocking (a
// user's first run may be on one) do not wait for it.
class InitStream {
 public:
  ~InitStream() {
    if (s_) cudaStreamDestroy(s_);
  }
  cudaError_t zero(void* p, size_t bytes) {
    const cudaError_t e = open();
    return e == cudaSuccess ? cudaMemsetAsync(p, 0, bytes, s_) : e;
  }
  cudaError_t upload(void* dst, const void* src, size_t bytes) {
    const cudaError_t e = open();
    return e == cudaSuccess ? cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, s_) : e;
  }
  cudaError_t wait() { return s_ ? cudaStreamSynchronize(s_) : cudaSuccess; }

 private:
  cudaError_t open() { return s_ ? cudaSuccess : cudaStreamCreateWithFlags(&s_, cudaStreamNonBlocking); }
  cudaStream_t s_ = nullptr;
};

}  // namespace hp
