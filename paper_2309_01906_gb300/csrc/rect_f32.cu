// rect_f32.cu — rectangular executor instantiated for plain FP32 sums.
#include "rect_launch.cuh"

namespace hp {
hp_status launch_rect_f32_sum(const NestPlan& np, LaunchCfg& cfg, const RectArgs& a) {
  return launch_rect<OpF32Sum>(np, cfg, a);
}
}  // namespace hp
