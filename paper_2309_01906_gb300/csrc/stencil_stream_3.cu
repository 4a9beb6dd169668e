// stencil_stream_3.cu — streamed stencil kernels of radius 3.
#include "stencil_stream.cuh"

namespace hp {
HP_STREAM_RADIUS(3)
}  // namespace hp
