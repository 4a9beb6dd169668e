// stencil_stream.cu — geometry and dispatch of the register-streamed stencil kernels.
#include "stencil_stream.cuh"

#include <algorithm>
#include <cmath>

namespace hp {

int stream_columns(int R, int T) { return kStreamCols - 2 * stream_ghost(R, T); }

// A strip of S rows costs S + 2 R T row steps and about 8 more until its ring is
// full.  `busy` of the resident warps saturate an SM (about 24: at 16384^2,
// radius 1, 4 steps, 18 warps per SM took 524 us, 28 took 454), so an underfull
// last wave costs that share of a whole one.  Longer strips than 288
// rows measured slower than their row steps (16384^2, radius 2, one step: 386 us
// with 512 rows, 347 to 356 with 96 to 288).
uint32_t stream_strip_rows(int64_t ny, int64_t nx, int R, int T, int ctas, int sms) {
  const int64_t cols = stream_columns(R, T), n_xt = (nx + cols - 1) / cols;
  const double resident = static_cast<double>(ctas) * kStreamWarps * sms, busy = std::min(1.0, 24.0 * sms / resident);
  double best = 0.0;
  uint32_t pick = 4;
  for (int64_t S = 4; S <= 288; S += S < 64 ? 4 : 16) {
    const double w = static_cast<double>(n_xt) * static_cast<double>((ny + S - 1) / S) / resident;
    const double waves = w <= 1.0 ? std::max(w, busy) : w + busy * (std::ceil(w) - w);
    const double cost = waves * static_cast<double>(std::min(S, ny) + 2 * R * T + 8);
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
  const uint64_t cols = static_cast<uint64_t>(stream_columns(R, T));
  a.n_xt = static_cast<uint32_t>((a.nx + cols - 1) / cols);
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
