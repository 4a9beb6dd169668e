// stencil_stream.cu — geometry and dispatch of the register-streamed stencil kernels.
#include "stencil_stream.cuh"

#include <algorithm>
#include <cmath>

namespace hp {

int stream_columns(int R, int T) { return kStreamCols - 2 * stream_ghost(R, T); }

// the last group's last lane lies outside the array (one step: no ghost zone)
int64_t stream_groups(int64_t nx, int R, int T) {
  const int64_t cols = stream_columns(R, T), over = T == 1 ? nx : nx - (kStreamCols - 8) + cols;
  return std::max<int64_t>(1, (over + cols - 1) / cols);
}

// A strip of S rows costs S + 2 R T row steps and about 8 more until its ring is
// full, times the CTAs an SM runs at once plus half of one for the latency of
// each step.  Fewer than `busy` CTAs of an SM take as long as that many: 24 warps
// where memory decides (16384^2, radius 1, 4 steps: 18 warps per SM took 524 us,
// 28 took 454), about one per scheduler where a row step is hundreds of FMAs
// (266 x 1848, radius 2, 7 steps: 39 us in strips that fill 12 warps, 27 in
// longer ones that fill 4, 29 tiled); an underfull last wave costs that share of
// a whole one.  Over 220 drawn sizes and radii this line took 1.13 times less
// than 24 warps for all.  Longer strips than 288 rows measured slower than their
// row steps (16384^2, radius 2, one step: 386 us with 512 rows, 347 to 356 with
// 96 to 288).
uint32_t stream_strip_rows(int64_t ny, int64_t nx, int R, int T, int ctas, int sms) {
  const int64_t n_xt = stream_groups(nx, R, T);
  const int64_t per_wave = static_cast<int64_t>(kStreamWarps) * sms;   // warps of one CTA on each SM
  const double fmas = static_cast<double>(T) * (2 * R + 1) * (2 * R + 1);
  const double busy = std::min<double>(ctas, std::min(24.0, 2.0 + 200.0 / fmas) / kStreamWarps);
  double best = 0.0;
  uint32_t pick = 4;
  for (int64_t S = 4; S <= 288; S += S < 64 ? 4 : 16) {
    const int64_t tasks = n_xt * ((ny + S - 1) / S);
    const double w = static_cast<double>(tasks) / (static_cast<double>(ctas) * per_wave);   // waves
    const double n = w <= 1.0 ? std::max<double>(static_cast<double>((tasks + per_wave - 1) / per_wave), busy)
                              : ctas * w + busy * (std::ceil(w) - w);
    const double cost = (n + 0.5) * static_cast<double>(std::min(S, ny) + 2 * R * T + 8);
    if (S == 4 || cost < best) {
      best = cost;
      pick = static_cast<uint32_t>(S);
    }
    if (S >= ny) break;
  }
  return pick;
}

int stream_occupancy(int R, int T, bool vec, cudaError_t* e) {
  switch (R) {
    case 1: return stream_occupancy_r1(T, vec, e);
    case 2: return stream_occupancy_r2(T, vec, e);
    case 3: return stream_occupancy_r3(T, vec, e);
    default: return stream_occupancy_r4(T, vec, e);
  }
}

cudaError_t stream_launch(int R, int T, bool vec, StreamArgs a, cudaStream_t st) {
  a.n_xt = static_cast<uint32_t>(stream_groups(a.nx, R, T));
  a.n_tasks = static_cast<uint64_t>(a.n_xt) * ((static_cast<uint64_t>(a.ny) + a.S - 1) / a.S);
  const uint64_t ctas = (a.n_tasks + kStreamWarps - 1) / kStreamWarps;
  if (ctas > 0x7fffffffull) return cudaErrorInvalidConfiguration;
  const unsigned grid = static_cast<unsigned>(ctas);
  switch (R) {
    case 1: return stream_launch_r1(T, vec, a, grid, st);
    case 2: return stream_launch_r2(T, vec, a, grid, st);
    case 3: return stream_launch_r3(T, vec, a, grid, st);
    default: return stream_launch_r4(T, vec, a, grid, st);
  }
}

}  // namespace hp
