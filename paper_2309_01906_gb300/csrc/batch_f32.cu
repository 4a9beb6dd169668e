// batch_f32.cu — the persistent batched kernel for plain FP32 sums, and the FP32 dispatch.
#include "batch_kernels.cuh"

namespace hp {
// batch_f32_comp.cu, batch_f32_mm.cu (units of their own: they compile in parallel)
cudaError_t launch_batch_comp(const BatchLaunch& b, cudaStream_t st);
int batch_comp_blocks_per_sm();
cudaError_t launch_batch_mm(int combo, const BatchLaunch& b, cudaStream_t st);
int batch_mm_blocks_per_sm(int combo);

cudaError_t launch_batch_fp(int combo, const BatchLaunch& b, cudaStream_t st) {
  switch (combo) {
    case 0: return launch_batch_op<OpF32Sum>(b, st);
    case 1: return launch_batch_comp(b, st);
    default: return launch_batch_mm(combo, b, st);
  }
}
int batch_fp_blocks_per_sm(int combo) {
  switch (combo) {
    case 0: return batch_blocks_per_sm<OpF32Sum>();
    case 1: return batch_comp_blocks_per_sm();
    default: return batch_mm_blocks_per_sm(combo);
  }
}
}  // namespace hp
