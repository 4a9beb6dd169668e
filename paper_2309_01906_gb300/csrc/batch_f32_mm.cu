// batch_f32_mm.cu — the persistent batched kernel for FP32 max / min.
#include "batch_kernels.cuh"

namespace hp {
cudaError_t launch_batch_mm(int combo, const BatchLaunch& b, cudaStream_t st) {
  return combo == 2 ? launch_batch_op<OpF32Max>(b, st) : launch_batch_op<OpF32Min>(b, st);
}
int batch_mm_blocks_per_sm(int combo) {
  return combo == 2 ? batch_blocks_per_sm<OpF32Max>() : batch_blocks_per_sm<OpF32Min>();
}
}  // namespace hp
