// resident_f32_mm.cu — the resident serving kernel for FP32 max / min.
#include "resident_kernels.cuh"

namespace hp {
cudaError_t launch_resident_mm(int combo, const ResidentSource& src, int grid, cudaStream_t st) {
  return combo == 2 ? launch_resident_op<OpF32Max>(src, grid, st) : launch_resident_op<OpF32Min>(src, grid, st);
}
int resident_mm_blocks_per_sm(int combo) {
  return combo == 2 ? resident_blocks_per_sm<OpF32Max>() : resident_blocks_per_sm<OpF32Min>();
}
}  // namespace hp
