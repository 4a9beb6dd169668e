// stencil_stream.h — host interface of the register-streamed stencil kernels
// (stencil_stream.cuh), one translation unit per radius.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace hp {

struct StreamArgs {
  const float* in;
  float* out;
  uint32_t ny, nx;
  uint32_t S;                 // rows per strip
  uint32_t n_xt;              // column groups
  uint64_t n_tasks;           // column groups x strips
  float c[81];
};

// Is there a streamed kernel of radius R and T steps?  Its partial sums take
// 8 R T registers per thread, so radius 4 ends at 5 steps (6: 18 TFLOP/s, the
// tiled kernel's rate).
constexpr bool stream_has(int R, int T) { return R >= 1 && R <= 3 ? T >= 1 && T <= 8 : R == 4 && T >= 1 && T <= 5; }

// One aligned step of radius 1 stays tiled.
constexpr bool stream_has(int R, int T, bool vec) { return stream_has(R, T) && !(vec && R == 1 && T == 1); }

// CTAs of the kernel that fit on an SM (0 if none; CUDA error in *e)
int stream_occupancy(int R, int T, bool vec, cudaError_t* e);

// columns stored by one warp (more at the array's edges), and column groups of a row
int stream_columns(int R, int T);
int64_t stream_groups(int64_t nx, int R, int T);

// rows per strip for an ny x nx array when `ctas` CTAs fit on each of `sms` SMs
uint32_t stream_strip_rows(int64_t ny, int64_t nx, int R, int T, int ctas, int sms);

constexpr int kStreamWarps = 4;     // warps per CTA

// a.S is set; fills the geometry and launches
cudaError_t stream_launch(int R, int T, bool vec, StreamArgs a, cudaStream_t st);

// per radius (stencil_stream_<R>.cu): the kernel's launch and occupancy
#define HP_STREAM_DECL(R)                                                                       \
  cudaError_t stream_launch_r##R(int T, bool vec, const StreamArgs& a, unsigned grid, cudaStream_t st); \
  int stream_occupancy_r##R(int T, bool vec, cudaError_t* e);
HP_STREAM_DECL(1)
HP_STREAM_DECL(2)
HP_STREAM_DECL(3)
HP_STREAM_DECL(4)
#undef HP_STREAM_DECL

}  // namespace hp
