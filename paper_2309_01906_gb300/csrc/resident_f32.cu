// resident_f32.cu — the resident serving kernel for plain FP32 sums, and the FP32 dispatch.
#include "resident_kernels.cuh"

namespace hp {
// resident_f32_comp.cu, resident_f32_mm.cu (units of their own: they compile in parallel)
cudaError_t launch_resident_comp(const ResidentSource& src, int grid, cudaStream_t st);
int resident_comp_blocks_per_sm();
cudaError_t launch_resident_mm(int combo, const ResidentSource& src, int grid, cudaStream_t st);
int resident_mm_blocks_per_sm(int combo);

cudaError_t launch_resident_fp(int combo, const ResidentSource& src, int grid, cudaStream_t st) {
  switch (combo) {
    case 0: return launch_resident_op<OpF32Sum>(src, grid, st);
    case 1: return launch_resident_comp(src, grid, st);
    default: return launch_resident_mm(combo, src, grid, st);
  }
}
int resident_fp_blocks_per_sm(int combo) {
  switch (combo) {
    case 0: return resident_blocks_per_sm<OpF32Sum>();
    case 1: return resident_comp_blocks_per_sm();
    default: return resident_mm_blocks_per_sm(combo);
  }
}
}  // namespace hp
