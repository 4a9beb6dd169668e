// stencil_stream_2.cu — streamed stencil kernels of radius 2.
#include "stencil_stream.cuh"

namespace hp {
HP_STREAM_RADIUS(2)
}  // namespace hp
