// stencil_stream_4.cu — streamed stencil kernels of radius 4.
#include "stencil_stream.cuh"

namespace hp {
HP_STREAM_RADIUS(4)
}  // namespace hp
