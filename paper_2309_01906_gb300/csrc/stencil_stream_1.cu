// stencil_stream_1.cu — streamed stencil kernels of radius 1.
#include "stencil_stream.cuh"

namespace hp {
HP_STREAM_RADIUS(1)
}  // namespace hp
