// init_stream.h — device state that is ready before its first use on any stream.
#pragma once

#include <cuda_runtime.h>

namespace hp {

// the current device's stream for such work, or nullptr (api.cu)
cudaStream_t init_stream();

// Clears and fills fresh device memory.  cudaMemset, and cudaMemcpy from pageable
// memory, are queued on the legacy stream and may still be pending when they
// return, behind whatever the program has queued there, and streams created
// non-blocking (a user's first run may be on one) do not wait for it.  So the work
// goes to the stream of the first run, which later runs are ordered after; when
// there is none, or it is being captured (the work would wait for a replay), to a
// stream for such work, one per device and process, that wait() waits for (a new
// nest's first run: 96 us on the run's stream, 115 on one created for it).
class InitStream {
 public:
  explicit InitStream(const cudaStream_t* run) : run_(run) {}   // the first run's stream, or nullptr
  InitStream(const InitStream&) = delete;
  InitStream& operator=(const InitStream&) = delete;
  cudaError_t zero(void* p, size_t bytes) {
    const cudaError_t e = open();
    return e == cudaSuccess ? cudaMemsetAsync(p, 0, bytes, s_) : e;
  }
  cudaError_t upload(void* dst, const void* src, size_t bytes) {
    const cudaError_t e = open();
    return e == cudaSuccess ? cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, s_) : e;
  }
  cudaError_t wait() { return own_ ? cudaStreamSynchronize(s_) : cudaSuccess; }

 private:
  cudaError_t open() {
    if (open_) return cudaSuccess;
    if (run_) {
      cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
      if (cudaStreamIsCapturing(*run_, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
        s_ = *run_;
        open_ = true;
        return cudaSuccess;
      }
      cudaGetLastError();
    }
    s_ = init_stream();
    open_ = own_ = s_ != nullptr;
    return open_ ? cudaSuccess : cudaErrorMemoryAllocation;
  }
  const cudaStream_t* run_;
  cudaStream_t s_ = nullptr;
  bool open_ = false, own_ = false;
};

}  // namespace hp
