// resident_f32_comp.cu — the resident serving kernel for compensated FP32 sums.
#include "resident_kernels.cuh"

namespace hp {
cudaError_t launch_resident_comp(const ResidentSource& src, int grid, cudaStream_t st) {
  return launch_resident_op<OpF32Comp>(src, grid, st);
}
int resident_comp_blocks_per_sm() { return resident_blocks_per_sm<OpF32Comp>(); }
}  // namespace hp
