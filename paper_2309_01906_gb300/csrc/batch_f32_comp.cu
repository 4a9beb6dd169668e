// batch_f32_comp.cu — the persistent batched kernel for compensated FP32 sums.
#include "batch_kernels.cuh"

namespace hp {
cudaError_t launch_batch_comp(const BatchLaunch& b, cudaStream_t st) { return launch_batch_op<OpF32Comp>(b, st); }
int batch_comp_blocks_per_sm() { return batch_blocks_per_sm<OpF32Comp>(); }
}  // namespace hp
