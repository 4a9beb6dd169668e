// stencil_stream.cuh — stencil steps streamed through the registers of a warp.
//
// A warp owns 128 adjacent columns (a float4 per lane) and walks down a strip of
// rows.  Every step of the nest keeps, per lane, the 2R partial sums of the
// output rows it has begun; a new input row advances each of them by one row of
// the window and completes one output row, which is at once the next step's
// input row.  So all T steps run in one pass over the rows, no step's values
// leave the registers, and the columns a lane lacks come from its neighbours by
// shuffle.  The outer R*T columns of the 128 are the ghost zone: they are
// computed from values the warp does not have, and only the others are stored.
// At the array's own edges one float4 is ghost zone enough, since what lies
// outside is known to be 0 at every step, so the first group starts 4 columns
// before the array (8000 x 116, radius 3, 8 steps: one group instead of two).
// Likewise a strip starts R*T rows early.  Points outside the array are 0 at
// every step.  Each point of each step is the same FP32 FMA chain as in the
// tiled kernel (row-major over the window, from 0), so the bits are equal.
//
// Rows arrive through a ring of D stages per warp filled by cp.async (absent
// rows and columns are zero-filled by the copy), D - 2 rows ahead.
//
// What bounds it: HBM up to 36 FMAs per point (16384^2, radius 1: 2 and 3 steps
// 357 us, 6.0 TB/s; radius 2, one step 351 us against 536 tiled), instruction issue
// beyond (radius 1: 4 steps 439 us = 44 TFLOP/s against 1024 us tiled, 8 steps 916
// against 2408; radius 4, one step: 720 us = 60 TFLOP/s against 1261 tiled; 4 steps of
// radius 1 use 0.80 of the issue slots and keep the FMA pipe active 0.61 of the
// time).  The tiled kernel reads each window row from shared memory, 2R + 1 loads a point.
// Packed FP32x2 FMAs over two strips per warp measured no faster than scalar
// ones (4 steps 483 us) and were left out.  128 columns per warp: a narrower
// group would spend more of its lanes on ghost columns (4 steps of radius 1: 8
// of 128).  Plain stores beat streaming ones by 2%.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "stencil_stream.h"

namespace hp {

constexpr int kStreamCols = 128;    // columns per warp

// ghost columns on each side of a warp's 128: whole float4s.  One step needs
// none: the ring's rows carry the neighbours' R columns.
__host__ __device__ constexpr int stream_ghost(int R, int T) { return T == 1 ? 0 : (R * T + 3) / 4 * 4; }

namespace stream {

struct True { static constexpr bool value = true; };
struct False { static constexpr bool value = false; };

__device__ __forceinline__ uint32_t saddr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
// copies that read nothing and write zeros when !valid
__device__ __forceinline__ void copy16(uint32_t dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy4(uint32_t dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}

}  // namespace stream

// VEC: rows are whole 16-byte groups (nx % 4 == 0, aligned bases); otherwise
// rows are copied and stored 4 bytes per lane, adjacent lanes on adjacent
// columns, and turned through the ring and one more stage
template <int R, int T, bool VEC, int D, int MINB>
__global__ void __launch_bounds__(32 * kStreamWarps, MINB)
    stencil_stream_kernel(const __grid_constant__ StreamArgs a) {
  constexpr int W = 2 * R + 1, H = R * T, HX = stream_ghost(R, T), XW = kStreamCols - 2 * HX;
  constexpr int RB = T == 1 ? 4 : 0;                    // ring columns on each side of the 128
  constexpr int RW = kStreamCols + 2 * RB;
  constexpr int STAGES = D + (VEC ? 0 : 1);
  __shared__ __align__(16) float ring[kStreamWarps][STAGES][RW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t task = blockIdx.x * static_cast<uint64_t>(kStreamWarps) + warp;
  if (task >= a.n_tasks) return;
  const uint32_t st = static_cast<uint32_t>(task / a.n_xt), xt = static_cast<uint32_t>(task - static_cast<uint64_t>(st) * a.n_xt);
  const uint32_t ny = a.ny, nx = a.nx, S = a.S;
  const uint32_t y0 = st * S;                           // first row of the strip
  constexpr int EX = T == 1 ? 0 : 4;                    // ghost columns at the array's edge
  const uint32_t gx0 = xt * XW - EX;                    // column of lane 0 (mod 2^32: negative columns are >= nx)
  const int c_lo = xt == 0 ? EX : HX, c_hi = xt + 1 == a.n_xt ? kStreamCols : kStreamCols - HX;   // columns stored
  const uint32_t gx = gx0 + 4 * lane;
  const int n_it = static_cast<int>(min(S, ny - y0)) + 2 * H;
  const int64_t pitch = a.nx;
  float (*const rg)[RW] = ring[warp];

  // ---- ring: row `it` is global row y0 - H + it
  uint32_t fy = y0 - H;                                 // next row to copy
  const uint32_t fx = VEC ? gx : gx0 + lane;            // first column this lane copies
  const float* fp = a.in + static_cast<int64_t>(static_cast<int32_t>(fy)) * pitch + static_cast<int32_t>(fx);
  const bool fx_in = fx < nx;
  auto issue = [&](int stage) {
    const bool row_in = fy < ny;
    const float* row = fp;
    float* dst = &rg[stage][RB];
    if constexpr (VEC) {
      const bool in = row_in && fx_in;
      stream::copy16(stream::saddr(dst + 4 * lane), in ? row : a.in, in);
      if constexpr (T == 1) {
        if (lane < 2) {   // the 4 columns before (lane 0) and after (lane 1) the 128
          const bool side_in = row_in && (lane ? gx0 + kStreamCols : gx0 - 4) < nx;
          stream::copy16(stream::saddr(dst + (lane ? kStreamCols : -4)),
                         side_in ? row + (lane ? kStreamCols - 4 : -4) : a.in, side_in);
        }
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const bool in = row_in && fx + 32 * k < nx;
        stream::copy4(stream::saddr(dst + lane + 32 * k), in ? row + 32 * k : a.in, in);
      }
      if constexpr (T == 1) {
        if (lane < 8) {   // columns -4 .. -1 (lanes 0-3) and 128 .. 131 (lanes 4-7)
          const int off = lane < 4 ? -4 : kStreamCols - 4;
          const bool side_in = row_in && fx + off < nx;
          stream::copy4(stream::saddr(dst + lane + off), side_in ? row + off : a.in, side_in);
        }
      }
    }
    ++fy;
    fp += pitch;
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < D - 1; ++s) issue(s);

  // ---- partial sums: A[s][j] has had 2R - j rows of its window
  float A[T][2 * R][4];
#pragma unroll
  for (int s = 0; s < T; ++s)
#pragma unroll
    for (int j = 0; j < 2 * R; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) A[s][j][i] = 0.0f;

  const bool store_lane = 4 * lane >= c_lo && 4 * lane < c_hi && gx < nx;
  float* op = a.out + static_cast<int64_t>(y0) * pitch + static_cast<int32_t>(VEC ? gx : gx0 + lane);
  int stage = 0, refill = D - 1;
  bool col_in[4];                                       // a 16-byte group is inside the array or outside
#pragma unroll
  for (int i = 0; i < 4; ++i) col_in[i] = gx + i < nx;

  auto walk = [&](auto masked) {
    for (int it = 0; it < n_it; ++it) {
      asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 2) : "memory");
      if constexpr (!VEC || T == 1) __syncwarp();
      float v[4], w[4 + 2 * R];
      {
        const float* src = &rg[stage][RB + 4 * lane];
        const float4 q = *reinterpret_cast<const float4*>(src);
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
        if constexpr (T == 1) {   // the neighbours' columns from the ring
          const float4 l = *reinterpret_cast<const float4*>(src - 4), r = *reinterpret_cast<const float4*>(src + 4);
          const float lv[4] = {l.x, l.y, l.z, l.w}, rv[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
          for (int i = 0; i < R; ++i) {
            w[i] = lv[4 - R + i];
            w[4 + R + i] = rv[i];
          }
        }
      }
      issue(refill);      // the stage read one iteration ago
      refill = stage;
      stage = stage + 1 == D ? 0 : stage + 1;
#pragma unroll
      for (int s = 0; s < T; ++s) {
        if constexpr (T > 1) {
#pragma unroll
          for (int i = 0; i < R; ++i) {
            w[i] = __shfl_up_sync(0xffffffffu, v[4 - R + i], 1);
            w[4 + R + i] = __shfl_down_sync(0xffffffffu, v[i], 1);
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) w[R + i] = v[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float o = A[s][0][i];
#pragma unroll
          for (int dx = 0; dx < W; ++dx) o = __fmaf_rn(a.c[2 * R * W + dx], w[i + dx], o);
          v[i] = o;
        }
#pragma unroll
        for (int j = 0; j < 2 * R; ++j) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float o = j + 1 < 2 * R ? A[s][j + 1 < 2 * R ? j + 1 : 0][i] : 0.0f;
#pragma unroll
            for (int dx = 0; dx < W; ++dx) o = __fmaf_rn(a.c[(2 * R - 1 - j) * W + dx], w[i + dx], o);
            A[s][j][i] = o;
          }
        }
        if constexpr (decltype(masked)::value) {
          if (s + 1 < T) {   // the zero ghost surface stays zero at every step
            const bool row_in = y0 - H + it - (s + 1) * R < ny;
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = row_in && col_in[VEC ? 0 : i] ? v[i] : 0.0f;
          }
        }
      }
      if (it >= 2 * H) {
        if constexpr (VEC) {
          if (store_lane) *reinterpret_cast<float4*>(op) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
          __syncwarp();
          *reinterpret_cast<float4*>(&rg[D][4 * lane]) = make_float4(v[0], v[1], v[2], v[3]);
          __syncwarp();
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int c = lane + 32 * k;
            if (c >= c_lo && c < c_hi && gx0 + c < nx) op[32 * k] = rg[D][c];
          }
        }
        op += pitch;
      }
    }
  };
  // One step needs no masks.  With radius 1 the 4 selects a step are a tenth of
  // its work, so strips whose ghost zones stay inside the array skip them; with
  // wider windows they cost less than a second copy of the loop (registers, and
  // instruction cache where both run on one SM).
  if constexpr (T == 1) {
    walk(stream::False{});
  } else if constexpr (R == 1) {
    const bool inside = gx0 < nx && gx0 + kStreamCols <= nx && y0 >= H && ny - y0 >= S + H;
    if (inside) walk(stream::False{});
    else walk(stream::True{});
  } else {
    walk(stream::True{});
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Registers grow with the partial sums (8 R T) and the window; the CTAs per SM
// that each kernel is compiled for were swept one up and one down at 16384^2
// with strips of one length (e.g. radius 1: 4 steps 6 CTAs 443 us, 7 CTAs 450, 8 CTAs
// 487; 8 steps 3 CTAs 989 us, 4 CTAs 1011; radius 2: 4 steps 3 CTAs 1191 us, 4 CTAs 1265).
constexpr int stream_blocks(int R, int T) {
  const int q = 8 * R * T + 4 * R;
  return T == 1 ? (R <= 2 ? 8 : R == 3 ? 6 : 7) : q <= 20 ? 8 : q <= 36 ? 6 : q <= 44 ? 5 : q <= 60 ? 4 : q <= 104 ? 3 : 2;
}
// ring stages: fewer warps keep more rows in flight each
constexpr int stream_depth(int R, int T) { return 8 * R * T + 4 * R <= 44 ? 6 : 8; }

template <int R, int T, bool VEC>
constexpr auto stream_kernel() {
  return stencil_stream_kernel<R, T, VEC, stream_depth(R, T), stream_blocks(R, T)>;
}

// the kernel of radius R for a run-time step count (0 when there is none)
template <int R, bool VEC, int T = 1>
auto stream_pick(int t) -> void (*)(const StreamArgs) {
  if constexpr (stream_has(R, T)) {
    if constexpr (stream_has(R, T, VEC)) {
      if (t == T) return stream_kernel<R, T, VEC>();
    }
    return stream_pick<R, VEC, T + 1>(t);
  }
  return nullptr;
}

#define HP_STREAM_RADIUS(R)                                                                              \
  cudaError_t stream_launch_r##R(int T, bool vec, const StreamArgs& a, unsigned grid, cudaStream_t st) { \
    auto k = vec ? stream_pick<R, true>(T) : stream_pick<R, false>(T);                                   \
    if (!k) return cudaErrorInvalidValue;                                                                \
    k<<<grid, 32 * kStreamWarps, 0, st>>>(a);                                                            \
    return cudaPeekAtLastError();                                                                        \
  }                                                                                                      \
  int stream_occupancy_r##R(int T, bool vec, cudaError_t* e) {                                           \
    auto k = vec ? stream_pick<R, true>(T) : stream_pick<R, false>(T);                                   \
    int n = 0;                                                                                           \
    *e = k ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 32 * kStreamWarps, 0)                  \
           : cudaErrorInvalidValue;                                                                      \
    return n;                                                                                            \
  }

}  // namespace hp
