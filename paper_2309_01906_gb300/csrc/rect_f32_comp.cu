// rect_f32_comp.cu — rectangular executor instantiated for compensated FP32 sums.
#include "rect_launch.cuh"

namespace hp {
hp_status launch_rect_f32_comp(const NestPlan& np, LaunchCfg& cfg, const RectArgs& a) {
  return launch_rect<OpF32Comp>(np, cfg, a);
}
}  // namespace hp
