// narrow.cu — nests on 8- and 16-bit integers with a SIMD-in-register level.
//
// App. A: besides the SIMT lanes, CUDA offers SIMD intrinsics on integers that
// treat a 32-bit register as two 16-bit or four 8-bit lanes; Sec. 3.8: a level
// can be split below the lanes.  Here every 32-bit register of a thread's
// 128-bit load is such a level: sums and int8 dot products go through
// __dp4a / __dp2a_lo into an int32 accumulator (exact modulo 2^32), maxima and
// minima through packed running registers of two 16-bit lanes (an int8 word is
// widened to two such) whose sub-lanes are folded once at the end.  Warps combine with
// the warp-reduce instructions (__reduce_add/max/min_sync), CTAs in shared
// memory, grid parts after a ticket.  Integer results do not depend on the
// order, so threads take 16-byte pieces cyclically (coalesced), rows that start
// or end off a 16-byte boundary give their ends to single-element loads, and
// short rows share a warp (narrow_rows_kernel).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <sstream>
#include <string>

#include "api_internal.h"

namespace hp {

constexpr int kNarThreads = 256;

// Teams of up to 256 threads are compiled for 8 resident CTAs per SM (32
// registers): a streaming fold needs the bytes in flight of 2048 threads to
// keep HBM busy.  Larger CTA teams (sub_width up to 32 warps) take a 1024-thread
// variant.
constexpr int kNarMinBlocks = 8;
constexpr int kNarDotBlocks = 6;   // CTA teams of the dot product: 40 registers (16384 x 65536: 152 us, with 8 CTAs 164)


namespace {
int64_t ceil_div64(int64_t a, int64_t b) { return (a + b - 1) / b; }
int64_t gcd64(int64_t a, int64_t b) { return b == 0 ? a : gcd64(b, a % b); }
}  // namespace

hp_status plan_narrow(int depth, const int64_t* extents, const hp_level_map* map, hp_red_op op, int red_level,
                      hp_prec prec, hp_body body, NarrowPlan* out, std::string* why) {
  auto bad = [&](const std::string& m) {
    *why = m;
    return HP_EINVAL;
  };
  if (prec != HP_I8 && prec != HP_I16) return bad("not an 8- or 16-bit nest");
  if (op != HP_RED_SUM && op != HP_RED_MAX && op != HP_RED_MIN) return bad("HP_I8 / HP_I16 reduce with SUM, MAX or MIN");
  if (body != HP_BODY_LOAD && body != HP_BODY_DOT_BCAST) return bad("HP_I8 / HP_I16 take body LOAD or DOT_BCAST");
  if (body == HP_BODY_DOT_BCAST && (prec != HP_I8 || op != HP_RED_SUM))
    return bad("DOT_BCAST on narrow integers: HP_I8 with SUM (int8 x int8 products)");
  if (depth < 1 || depth > HP_MAX_DEPTH) return bad("depth must be in [1, HP_MAX_DEPTH]");
  if (!extents) return bad("extents is NULL");
  if (red_level < 0 || red_level >= depth) return bad("red_level must be in [0, depth - 1] (something is reduced)");
  NarrowPlan p;
  p.depth = depth;
  p.red_level = red_level;
  p.op = op;
  p.prec = prec;
  p.body = body;
  p.esize = prec == HP_I8 ? 1 : 2;
  int64_t O = 1, R = 1, inner = 1;
  for (int l = 0; l < depth; ++l) {
    if (extents[l] < 0) return bad("extents must be >= 0");
    p.ext[l] = extents[l];
    if (l < red_level) O *= extents[l];
    else R *= extents[l];
    if (l > red_level) inner *= std::max<int64_t>(extents[l], 1);
    if (O > (int64_t(1) << 40) || R > (int64_t(1) << 40)) return bad("nest too large");
  }
  if (O * std::max<int64_t>(R, 1) > (int64_t(1) << 42)) return bad("nest too large (2^42 iterations)");
  p.O = O;
  p.R = R;
  bool all_auto = map == nullptr;
  if (map) {
    all_auto = true;
    for (int l = 0; l < depth; ++l)
      if (map[l].hw != HP_HW_AUTO) all_auto = false;
  }
  p.auto_map = all_auto;
  int red_hw, sub = 0;
  int64_t tile = 0;
  const int64_t bytes = R * p.esize;
  if (all_auto) {
    red_hw = bytes <= 16384 ? HP_HW_WARP : ((O >= 304 || bytes <= (int64_t(1) << 18)) ? HP_HW_CTA : HP_HW_GRID);
  } else {
    for (int l = 0; l < red_level; ++l)
      if (map[l].hw != HP_HW_GRID) return bad("narrow-integer nests keep their output levels on GRID");
    red_hw = map[red_level].hw;
    sub = map[red_level].sub_width;
    tile = map[red_level].tile;
    for (int l = red_level; l < depth; ++l)
      if (map[l].hw != red_hw) return bad("the reduced levels of a narrow-integer nest share one hardware level");
    if (red_hw != HP_HW_WARP && red_hw != HP_HW_CTA && red_hw != HP_HW_GRID)
      return bad("narrow-integer nests put their reduced levels on WARP, CTA or GRID");
    if (red_hw == HP_HW_CTA && (sub < 0 || sub > 32)) return bad("CTA sub_width must be in [0, 32]");
    if (tile < 0) return bad("tile must be >= 0");
  }
  const int64_t piece = 16 / p.esize;   // elements of one 128-bit load
  if (red_hw == HP_HW_WARP) {
    p.team = 0;
    p.W = 1;
    p.G = 1;
    p.part = R;
  } else {
    p.team = 1;
    p.W = (red_hw == HP_HW_CTA && sub > 0) ? sub : 8;
    if (red_hw == HP_HW_GRID) {
      int64_t part;
      if (tile > 0) {
        part = tile * inner;
      } else {
        // one wave of the CTAs that fit on an SM
        const int64_t want = std::max<int64_t>(1, (body == HP_BODY_DOT_BCAST ? kNarDotBlocks : kNarMinBlocks) * 152 / std::max<int64_t>(O, 1));
        part = std::max<int64_t>(65536, ceil_div64(R, want));
        const int64_t step = (R % piece == 0) ? inner * piece / gcd64(inner, piece) : inner;   // whole pieces
        part = ceil_div64(part, step) * step;
      }
      p.part = std::max<int64_t>(1, part);
      p.G = R > 0 ? ceil_div64(R, p.part) : 1;
      if (p.G > (int64_t(1) << 30)) return bad("too many grid parts");
    } else {
      p.G = 1;
      p.part = R;
    }
  }
  for (int l = 0; l < depth; ++l)
    p.map[l] = {l < red_level ? HP_HW_GRID : red_hw, l >= red_level && red_hw == HP_HW_CTA ? p.W : 0,
                l == red_level && red_hw == HP_HW_GRID ? p.part / inner : 0};
  *out = p;
  return HP_OK;
}

namespace {
// which kernel takes the rows of a warp team (row_kernel)
enum RowKernel { ROW_WARP, ROW_SHARED, ROW_ELEMENTS };
RowKernel row_kernel(const NarrowPlan& p, bool ragged, int sms);
}  // namespace

std::string describe_narrow(const NarrowPlan& p) {
  static const char* hw[] = {"grid", "cluster", "cta", "warp", "subwarp", "lane", "seq", "auto"};
  static const char* ops[] = {"sum", "max", "min"};
  static const char* kRowNames[] = {"warp", "rows", "elements"};
  std::ostringstream s;
  s << "{\"kind\":\"narrow\",\"prec\":\"" << (p.prec == HP_I8 ? "i8" : "i16") << "\",\"op\":\"" << ops[p.op]
    << "\",\"body\":\"" << (p.body == HP_BODY_LOAD ? "load" : "dot_bcast") << "\",\"depth\":" << p.depth
    << ",\"red_level\":" << p.red_level << ",\"extents\":[";
  for (int l = 0; l < p.depth; ++l) s << (l ? "," : "") << p.ext[l];
  s << "],\"map\":[";
  for (int l = 0; l < p.depth; ++l)
    s << (l ? "," : "") << "{\"hw\":\"" << hw[p.map[l].hw] << "\",\"sub_width\":" << p.map[l].sub_width
      << ",\"tile\":" << p.map[l].tile << "}";
  s << "],\"auto_map\":" << (p.auto_map ? "true" : "false") << ",\"team\":\"" << (p.team ? "block" : "warp")
    << "\",\"outputs\":" << p.O << ",\"reduced\":" << p.R << ",\"warps\":" << p.W << ",\"grid_parts\":" << p.G
    << ",\"part\":" << p.part << ",\"vec\":" << 16 / p.esize << ",\"simd\":" << 4 / p.esize << ",\"kernel\":\"narrow_"
    << (p.team ? "block" : kRowNames[row_kernel(p, p.R % (16 / p.esize) != 0, 152)]) << "\"}";
  return s.str();
}

namespace {

struct NarArgs {
  const void* a;
  const void* w;     // DOT_BCAST: broadcast operand over the reduced levels
  int32_t* out;
  int32_t* part;
  int32_t* tickets;
  int64_t O, R, G, part_len;
  int32_t W;
};

// the larger (OP 1) or smaller (OP 2) of each signed 16-bit half: one instruction from sm_90 on
template <int OP>
__device__ __forceinline__ uint32_t minmax16(uint32_t a, uint32_t b) {
  uint32_t r;
  if constexpr (OP == 1) asm("max.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  else asm("min.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// A thread's running value.  Sums: an int32.  Maxima and minima: packed 16-bit
// lanes.  A 16-bit comparison is decided by the high byte first, so the high
// byte of the larger of two 16-bit values is the larger of their high bytes:
// int8 lanes 1 and 3 of a word fold as they stand, lanes 0 and 2 after a shift by
// 8 (3 instructions per word; __vmaxs4 is emulated on this GPU: 65536 x 4099
// int8, 40 us against 47).
// E: int8_t or int16_t; OP: 0 sum, 1 max, 2 min
template <class E, int OP>
struct NarrowOp {
  static constexpr bool kI8 = sizeof(E) == 1;
  static constexpr int32_t ident() { return OP == 0 ? 0 : (OP == 1 ? (kI8 ? -128 : -32768) : (kI8 ? 127 : 32767)); }
  // the identity in every sub-lane of a word of input
  static constexpr uint32_t packed_ident() {
    return OP == 0 ? 0u
                   : OP == 1 ? (kI8 ? 0x80808080u : 0x80008000u) : (kI8 ? 0x7f7f7f7fu : 0x7fff7fffu);
  }
  struct Run {
    int32_t sum = 0;
    uint32_t hi = OP == 1 ? 0x80008000u : 0x7fff7fffu, lo = hi;   // lo: int8 lanes 0 and 2
  };
  // one 32-bit register of the input: 4 (2) sub-lanes
  __device__ static __forceinline__ void fold_word(uint32_t x, uint32_t wv, Run& r, bool dot) {
    if constexpr (OP == 0) {
      if constexpr (kI8) r.sum = __dp4a(static_cast<int>(x), dot ? static_cast<int>(wv) : 0x01010101, r.sum);
      else r.sum = __dp2a_lo(static_cast<int>(x), 0x0101, r.sum);
    } else {
      r.hi = minmax16<OP>(r.hi, x);
      if constexpr (kI8) r.lo = minmax16<OP>(r.lo, x << 8);
    }
  }
  __device__ static __forceinline__ void fold_piece(const uint4& q, const uint4& w, Run& r, bool dot) {
    fold_word(q.x, w.x, r, dot);
    fold_word(q.y, w.y, r, dot);
    fold_word(q.z, w.z, r, dot);
    fold_word(q.w, w.w, r, dot);
  }
  __device__ static __forceinline__ int32_t value(const Run& r) {
    if constexpr (OP == 0) {
      return r.sum;
    } else {
      const uint32_t p = kI8 ? minmax16<OP>(r.hi, r.lo) : r.hi;
      const int32_t a = static_cast<int32_t>(p) >> (kI8 ? 24 : 16);
      const int32_t b = static_cast<int32_t>(p << 16) >> (kI8 ? 24 : 16);
      return combine(a, b);
    }
  }
  __device__ static __forceinline__ int32_t combine(int32_t a, int32_t b) {
    if constexpr (OP == 0) return static_cast<int32_t>(static_cast<uint32_t>(a) + static_cast<uint32_t>(b));
    else if constexpr (OP == 1) return max(a, b);
    else return min(a, b);
  }
  __device__ static __forceinline__ int32_t warp_reduce(int32_t v) {
    if constexpr (OP == 0) return __reduce_add_sync(0xffffffffu, v);
    else if constexpr (OP == 1) return __reduce_max_sync(0xffffffffu, v);
    else return __reduce_min_sync(0xffffffffu, v);
  }
};

// bytes s .. s + 15 of the 32 bytes (x, y)
__device__ __forceinline__ uint4 shift_bytes(uint4 x, uint4 y, uint32_t s) {
  uint32_t v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
  if (s & 8u) {
#pragma unroll
    for (int i = 0; i < 6; ++i) v[i] = v[i + 2];
  }
  if (s & 4u) {
#pragma unroll
    for (int i = 0; i < 5; ++i) v[i] = v[i + 1];
  }
  const uint32_t b = 8u * (s & 3u);
  return make_uint4(__funnelshift_r(v[0], v[1], b), __funnelshift_r(v[1], v[2], b), __funnelshift_r(v[2], v[3], b),
                    __funnelshift_r(v[3], v[4], b));
}

// This thread's share of elements [lo, hi) of one output (a = the output's
// first element): whole 16-byte pieces cyclically over the T threads of the
// team.  RAGGED: the elements before the first and after the last 16-byte
// boundary go to single loads, one per thread, and a broadcast operand that
// starts off the pieces' boundary is read as two aligned pieces and shifted
// (pieces whose two would reach outside w join the single loads).  Rows of
// 65541 int8, 268 MB: 466 us as single loads, 39 so (HBM's rate); the dot
// product 465 and 47.
template <class E, int OP, bool DOT, bool RAGGED>
__device__ __forceinline__ int32_t fold_range(const E* __restrict__ a, const E* __restrict__ w, int64_t lo, int64_t hi,
                                              int64_t R, int64_t t, int64_t T) {
  using Op = NarrowOp<E, OP>;
  constexpr int64_t kP = 16 / sizeof(E);   // elements per 128-bit piece
  typename Op::Run run;
  int32_t acc = Op::ident();               // the single elements
  uint32_t ws = 0;                         // offset of w's pieces from a 16-byte boundary
  if constexpr (RAGGED) {
    int64_t head = static_cast<int64_t>((16u - (reinterpret_cast<uintptr_t>(a + lo) & 15u)) & 15u) / static_cast<int64_t>(sizeof(E));
    if (head > hi - lo) head = hi - lo;
    int64_t body = (hi - lo - head) / kP * kP;
    if constexpr (DOT) {
      ws = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(w + lo + head) & 15u);
      if (ws != 0 && body > 0 && lo + head < kP) {
        head += kP;
        body -= kP;
      }
      if (ws != 0 && body > 0 && lo + head + body + kP > R) body -= kP;
    }
    const int64_t first_end = lo + head, tail = lo + head + body;
    for (int64_t x = t; x < (hi - lo) - body; x += T) {   // at most 15 + 16 elements on either side
      const int64_t e = x < head ? lo + x : tail + (x - head);
      const int32_t v = static_cast<int32_t>(a[e]);
      if constexpr (OP == 0) {
        acc = static_cast<int32_t>(static_cast<uint32_t>(acc) +
                                   static_cast<uint32_t>(DOT ? v * static_cast<int32_t>(w[e]) : v));
      } else {
        acc = Op::combine(acc, v);
      }
    }
    lo = first_end;
    hi = tail;
  }
  const uint4* ap = reinterpret_cast<const uint4*>(a + lo) + t;
  const uint4* wq = DOT ? reinterpret_cast<const uint4*>(w + lo - ws) + t : nullptr;
  const int64_t pieces = (hi - lo) / kP;
  int64_t n = t < pieces ? (pieces - t + T - 1) / T : 0;   // pieces of this thread
  auto fold = [&](const uint4& q, const uint4& r) { Op::fold_piece(q, r, run, DOT); };
  if (DOT && RAGGED && ws != 0) {
    for (; n >= 2; n -= 2, ap += 2 * T, wq += 2 * T) {
      const uint4 q0 = __ldcs(ap), q1 = __ldcs(ap + T);
      const uint4 x0 = __ldg(wq), y0 = __ldg(wq + 1), x1 = __ldg(wq + T), y1 = __ldg(wq + T + 1);
      fold(q0, shift_bytes(x0, y0, ws));
      fold(q1, shift_bytes(x1, y1, ws));
    }
    if (n > 0) {
      const uint4 q = __ldcs(ap);
      fold(q, shift_bytes(__ldg(wq), __ldg(wq + 1), ws));
    }
  } else {
    for (; n >= 4; n -= 4, ap += 4 * T, wq += 4 * T) {       // four pieces in flight
      uint4 q[4], r[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        q[u] = __ldcs(ap + u * T);
        if constexpr (DOT) r[u] = __ldg(wq + u * T);
        else r[u] = make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) fold(q[u], r[u]);
    }
    if (n > 0) {   // the last one to three, in flight together
      uint4 q[3], r[3];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int64_t at = u < n ? u * T : 0;
        q[u] = __ldcs(ap + at);
        if constexpr (DOT) r[u] = __ldg(wq + at);
        else r[u] = make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (u < n) fold(q[u], r[u]);
    }
  }
  return RAGGED ? Op::combine(acc, Op::value(run)) : Op::value(run);
}

template <class E, int OP, bool DOT, bool RAGGED>
__global__ void __launch_bounds__(kNarThreads, RAGGED ? (DOT ? 5 : 6) : kNarMinBlocks) narrow_warp_kernel(NarArgs g) {
  using Op = NarrowOp<E, OP>;
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (kNarThreads / 32);
  for (int64_t o = static_cast<int64_t>(blockIdx.x) * (kNarThreads / 32) + (threadIdx.x >> 5); o < g.O; o += warps) {
    const E* a = static_cast<const E*>(g.a) + o * g.R;
    const E* w = static_cast<const E*>(g.w);
    int32_t v = fold_range<E, OP, DOT, RAGGED>(a, w, 0, g.R, g.R, lane, 32);
    v = Op::warp_reduce(v);
    if (lane == 0) g.out[o] = v;
  }
}

// a warp per row, one element per lane and load: ragged rows of a few hundred
// elements, too few for the shared-warp kernel's start to pay (row_kernel)
template <class E, int OP, bool DOT>
__global__ void __launch_bounds__(kNarThreads, kNarMinBlocks) narrow_elements_kernel(NarArgs g) {
  using Op = NarrowOp<E, OP>;
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (kNarThreads / 32);
  const E* w = static_cast<const E*>(g.w);
  for (int64_t o = static_cast<int64_t>(blockIdx.x) * (kNarThreads / 32) + (threadIdx.x >> 5); o < g.O; o += warps) {
    const E* a = static_cast<const E*>(g.a) + o * g.R;
    int32_t v = Op::ident();
    for (int64_t x = lane; x < g.R; x += 32) {
      const int32_t e = static_cast<int32_t>(a[x]);
      v = Op::combine(v, DOT ? e * static_cast<int32_t>(w[x]) : e);
    }
    v = Op::warp_reduce(v);
    if (lane == 0) g.out[o] = v;
  }
}

template <class E, int OP, bool DOT, bool RAGGED, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == kNarThreads ? (RAGGED ? (DOT ? 5 : 6) : DOT ? kNarDotBlocks : kNarMinBlocks) : 1)
    narrow_block_kernel(NarArgs g) {
  using Op = NarrowOp<E, OP>;
  __shared__ int32_t wp[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t items = g.O * g.G;
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int64_t o = item / g.G, pg = item - o * g.G;
    const int64_t lo = pg * g.part_len, hi = std::min<int64_t>(lo + g.part_len, g.R);
    const E* a = static_cast<const E*>(g.a) + o * g.R;
    int32_t v = fold_range<E, OP, DOT, RAGGED>(a, static_cast<const E*>(g.w), lo, hi, g.R, threadIdx.x, blockDim.x);
    v = Op::warp_reduce(v);
    if (lane == 0) wp[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      int32_t r = wp[0];
      for (int q = 1; q < g.W; ++q) r = Op::combine(r, wp[q]);
      if (g.G == 1) {
        g.out[o] = r;
      } else {
        g.part[item] = r;
        __threadfence();   // publish the part before taking the ticket
        if (atomicAdd(&g.tickets[o], 1) == g.G - 1) {
          __threadfence();
          const volatile int32_t* pp = g.part + o * g.G;
          int32_t s = pp[0];
          for (int64_t q = 1; q < g.G; ++q) s = Op::combine(s, pp[q]);
          g.out[o] = s;
          g.tickets[o] = 0;   // ready for the next run
        }
      }
    }
    __syncthreads();   // wp is rewritten by the next item
  }
}

// Short rows: L lanes per row (short_lanes), 32 / L rows per warp and kShortRows
// such sets in flight.  A row's first and last granule may hold
// neighbouring rows' bytes: they are replaced by the identity (0 in a sum) with
// masks from shared memory.  The dot product's w sits in shared memory in 16
// copies, copy s shifted by s bytes, so that any alignment reads whole pieces.
// Bound by instructions per granule (masks, shifts), by HBM for whole granules:
// int8 sums of 268 MB, before (a warp per row, an element per load off 16-byte
// boundaries) and now: 64-byte rows 376 and 44 us (6.5 TB/s), 333 bytes 109 and
// 48, 500 bytes 125 and 54, 1000 bytes 118 and 45.
constexpr int kShortBytes = 1024;             // rows off 16-byte boundaries
constexpr int kShortAligned = 512;             // rows of whole granules (a warp per row of 1024 bytes reads 6.2 TB/s)
constexpr int kShortRows = 4;
constexpr int kShortW = kShortBytes + 48;   // one shifted copy of w, with the 16 bytes before and after it

// a granule that reaches outside the array [first, last): its valid bytes [lo, hi) one by one
__device__ __noinline__ uint4 granule_bytes(const unsigned char* p, int lo, int hi) {
  uint32_t v[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (i >= lo && i < hi) v[i >> 2] |= static_cast<uint32_t>(p[i]) << (8 * (i & 3));
  return make_uint4(v[0], v[1], v[2], v[3]);
}

template <class E, int OP, bool DOT, bool RAGGED>
__global__ void __launch_bounds__(kNarThreads, 4) narrow_rows_kernel(NarArgs g, int L) {
  using Op = NarrowOp<E, OP>;
  __shared__ __align__(16) uint32_t masks[RAGGED ? 256 : 1][4];   // bytes [lo, hi) of a granule: entry 16 lo + hi - 1
  __shared__ __align__(16) uint32_t wcopy[DOT ? (RAGGED ? 16 : 1) : 1][DOT ? kShortW / 4 : 4];
  const int tid = threadIdx.x;
  if constexpr (RAGGED) {
    for (int i = tid; i < 256 * 4; i += kNarThreads) {
      const int word = i & 3, lo = i >> 6, hi = ((i >> 2) & 15) + 1;
      uint32_t m = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * word + k >= lo && 4 * word + k < hi) m |= 0xffu << (8 * k);
      masks[i >> 2][word] = m;
    }
  }
  if constexpr (DOT) {
    const int n = static_cast<int>(g.R);
    const unsigned char* wb = static_cast<const unsigned char*>(g.w);
    constexpr int kWords = kShortW / 4;
    for (int i = tid; i < (RAGGED ? 16 : 1) * kWords; i += kNarThreads) {
      const int c = i / kWords, j = i - c * kWords;
      uint32_t v = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int e = 4 * j + k + c - 16;                    // element of w at this byte
        if (e >= 0 && e < n) v |= static_cast<uint32_t>(wb[e]) << (8 * k);
      }
      wcopy[c][j] = v;
    }
  }
  __syncthreads();
  const int lane = tid & 31, sub = lane & (L - 1), set = 32 / L;
  const int row_bytes = static_cast<int>(g.R) * static_cast<int>(sizeof(E));
  const int max_granules = RAGGED ? (row_bytes + 30) / 16 : row_bytes / 16;
  const int64_t per_warp = static_cast<int64_t>(set) * kShortRows;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * (kNarThreads / 32) * per_warp;
  int off[kShortRows];                                       // this lane's rows, in bytes from the warp's first
#pragma unroll
  for (int u = 0; u < kShortRows; ++u) off[u] = (u * set + lane / L) * row_bytes;
  for (int64_t base = (static_cast<int64_t>(blockIdx.x) * (kNarThreads / 32) + (tid >> 5)) * per_warp; base < g.O;
       base += stride) {
    const unsigned char* const first = static_cast<const unsigned char*>(g.a) + base * row_bytes;
    const int skew0 = static_cast<int>(reinterpret_cast<uintptr_t>(first) & 15u);
    const int64_t left = g.O - base;
    const bool ends = base == 0 || left <= per_warp + 15;    // a granule may reach outside the array
    typename Op::Run run[kShortRows];
    for (int j = sub; j < max_granules; j += L) {
      uint4 q[kShortRows];
      int lo[kShortRows], hi[kShortRows];                    // valid bytes of the granule
#pragma unroll
      for (int u = 0; u < kShortRows; ++u) {
        const int skew = RAGGED ? (skew0 + off[u]) & 15 : 0;
        const int at = off[u] - skew + 16 * j;
        lo[u] = RAGGED && j == 0 ? skew : 0;
        hi[u] = RAGGED ? min(16, row_bytes + skew - 16 * j) : 16;
        if (ends && u * set + lane / L >= left) hi[u] = 0;
        constexpr uint32_t id = Op::packed_ident();
        q[u] = make_uint4(id, id, id, id);
        if (hi[u] > 0) {
          if (RAGGED && ends && (lo[u] > 0 || hi[u] < 16) &&
              ((base == 0 && at < 0) || at + 16 > left * row_bytes))
            q[u] = granule_bytes(first + at, lo[u], hi[u]);
          else
            q[u] = __ldcs(reinterpret_cast<const uint4*>(first + at));
        }
      }
#pragma unroll
      for (int u = 0; u < kShortRows; ++u) {
        if constexpr (RAGGED) {
          const uint4 m = *reinterpret_cast<const uint4*>(masks[16 * lo[u] + max(hi[u], 1) - 1]);
          constexpr uint32_t id = Op::packed_ident();
          q[u] = make_uint4((q[u].x & m.x) | (id & ~m.x), (q[u].y & m.y) | (id & ~m.y), (q[u].z & m.z) | (id & ~m.z),
                            (q[u].w & m.w) | (id & ~m.w));
        }
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if constexpr (DOT) {
          // the granule's first byte is element 16 j - skew; copies start 16 bytes before element 0
          const int x = 16 * j + 16 - (RAGGED ? (skew0 + off[u]) & 15 : 0);
          r = *reinterpret_cast<const uint4*>(&wcopy[RAGGED ? x & 15 : 0][(x >> 4) * 4]);
        }
        Op::fold_piece(q[u], r, run[u], DOT);
      }
    }
#pragma unroll
    for (int u = 0; u < kShortRows; ++u) {
      int32_t v = Op::value(run[u]);
      for (int m = L >> 1; m >= 1; m >>= 1) v = Op::combine(v, __shfl_xor_sync(0xffffffffu, v, m));
      const int row = u * set + lane / L;
      if (sub == 0 && row < left) g.out[base + row] = v;
    }
  }
}

template <class K>
int nar_blocks(K kernel, int threads, int sms) {
  int per = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0);
  return std::max(1, per) * sms;
}

// CTAs for `items` work items when `resident` fit at once: the fewest waves,
// with the items spread evenly over them (no short last wave)
int64_t balanced_grid(int64_t items, int64_t resident) {
  if (items <= resident) return std::max<int64_t>(items, 1);
  const int64_t waves = ceil_div64(items, resident);
  return ceil_div64(items, waves);
}

// lanes per short row: the fewest idle lane slots over at most four rounds of
// granules, counting the reduction and the store as 2 log2 L + 6 of the about 40
// instructions that a granule takes (500-byte rows: 16 lanes 102 us, 32 lanes,
// half of them idle in the second round, 112)
int short_lanes(int granules) {
  int best = 32, cost = 1 << 30;
  for (int lg = 5; lg >= 0; --lg) {
    const int L = 1 << lg, rounds = (granules + L - 1) / L;
    if (rounds > 4) break;
    const int c = L * (40 * rounds + 2 * lg + 6);
    if (c < cost) {
      cost = c;
      best = L;
    }
  }
  return best;
}

// Which kernel takes the rows of a warp team?  The shared-warp kernel
// (narrow_rows_kernel) folds the most rows per second, but its start (tables in
// shared memory, several rounds of granules per lane) costs about a microsecond,
// two and a half with the tables of a ragged dot product, which only many rows
// earn back.  Device times of 1000 and 30,000 rows, the shared-warp kernel / a warp
// per row: 64 bytes 2.7 / 1.4 and 2.7 / 4.4 us, 16 bytes 1.6 / 1.4 and 1.6 / 4.3; ragged
// 1000 bytes 3.9 / 1.8 and 6.8 / 9.8; ragged 100 bytes, with a warp per row by elements,
// 3.6 / 1.4 and 3.6 / 4.5, dot product 5.8 / 1.5 and 5.8 / 5.3.
RowKernel row_kernel(const NarrowPlan& p, bool ragged, int sms) {
  const int64_t bytes = p.R * p.esize;
  if (p.R < 1 || bytes > (ragged ? kShortBytes : kShortAligned)) return ROW_WARP;
  if (!ragged) return p.O > (bytes <= 32 ? 20 : bytes <= 256 ? 80 : 100) * static_cast<int64_t>(sms) ? ROW_SHARED : ROW_WARP;
  // beyond about 12 elements per lane whole pieces beat single elements; a warp per row fills
  // the SMs once with 48 to 64 rows each
  if (p.R > 384) return p.O > 80 * static_cast<int64_t>(sms) ? ROW_SHARED : ROW_WARP;
  // the start against what a thousand rows take longer by elements (measured lines, us)
  const bool dot = p.body == HP_BODY_DOT_BCAST;
  const double start = dot ? 3.4 : bytes <= 16 ? 0.95 : 1.8;
  const double elements = 0.09 + (dot ? 0.0003 : 0.00015) * p.R, shared = (dot ? 0.00029 : 0.00017) * bytes;
  return p.O / 1000.0 * (elements - shared) * (152.0 / sms) > start ? ROW_SHARED : ROW_ELEMENTS;
}

template <class E, int OP, bool DOT, bool RAGGED>
cudaError_t launch_narrow(const NarrowPlan& p, const NarArgs& g, int sms, cudaStream_t st) {
  const RowKernel rows = p.team == 0 ? row_kernel(p, RAGGED, sms) : ROW_WARP;
  if (rows == ROW_SHARED) {
    const int bytes = static_cast<int>(p.R) * p.esize;
    const int L = short_lanes(RAGGED ? (bytes + 30) / 16 : bytes / 16);
    auto k = narrow_rows_kernel<E, OP, DOT, RAGGED>;
    const int64_t need = ceil_div64(p.O, static_cast<int64_t>(kNarThreads / L) * kShortRows);
    k<<<static_cast<int>(balanced_grid(need, nar_blocks(k, kNarThreads, sms))), kNarThreads, 0, st>>>(g, L);
  } else if (p.team == 0) {
    const int64_t need = ceil_div64(p.O, kNarThreads / 32);
    auto k = narrow_warp_kernel<E, OP, DOT, RAGGED>;
    if constexpr (RAGGED) {
      if (rows == ROW_ELEMENTS) k = narrow_elements_kernel<E, OP, DOT>;
    }
    k<<<static_cast<int>(balanced_grid(need, nar_blocks(k, kNarThreads, sms))), kNarThreads, 0, st>>>(g);
  } else {
    const int threads = 32 * p.W;
    if (threads <= kNarThreads) {
      auto k = narrow_block_kernel<E, OP, DOT, RAGGED, kNarThreads>;
      const int grid = static_cast<int>(balanced_grid(p.O * p.G, nar_blocks(k, threads, sms)));
      k<<<grid, threads, 0, st>>>(g);
    } else {
      auto k = narrow_block_kernel<E, OP, DOT, RAGGED, 1024>;
      const int grid = static_cast<int>(balanced_grid(p.O * p.G, nar_blocks(k, threads, sms)));
      k<<<grid, threads, 0, st>>>(g);
    }
  }
  return cudaPeekAtLastError();
}

template <class E, int OP, bool DOT>
cudaError_t launch_narrow_v(const NarrowPlan& p, const NarArgs& g, bool vec, int sms, cudaStream_t st) {
  return vec ? launch_narrow<E, OP, DOT, false>(p, g, sms, st) : launch_narrow<E, OP, DOT, true>(p, g, sms, st);
}

}  // namespace

hp_status narrow_prepare(hp_nest* n, InitStream& init) {
  const NarrowPlan& p = n->nar;
  if (p.G > 1 && p.O > 0) {
    n->part_bytes = static_cast<size_t>(p.O * p.G) * sizeof(int32_t);
    cudaError_t e = cudaMalloc(&n->part, n->part_bytes);
    if (e != cudaSuccess) return fail(HP_ENOMEM, "cudaMalloc (narrow parts)");
    if ((e = cudaMalloc(&n->tickets, sizeof(int32_t) * p.O)) != cudaSuccess)
      return fail(HP_ENOMEM, "cudaMalloc (narrow tickets)");
    if ((e = init.zero(n->tickets, sizeof(int32_t) * p.O)) != cudaSuccess)
      return fail(HP_ECUDA, std::string("clear tickets: ") + cudaGetErrorString(e));
  }
  return HP_OK;
}

hp_status run_narrow(hp_nest* n, const void* const* in_dev, void* out_dev, cudaStream_t st) {
  const NarrowPlan& p = n->nar;
  if (p.O == 0) return HP_OK;
  if (!out_dev) return fail(HP_EINVAL, "out is NULL");
  const bool dot = p.body == HP_BODY_DOT_BCAST;
  if (p.R > 0 && (!in_dev || !in_dev[0] || (dot && !in_dev[1]))) return fail(HP_EINVAL, "missing input");
  NarArgs g;
  g.a = p.R > 0 ? in_dev[0] : nullptr;
  g.w = (p.R > 0 && dot) ? in_dev[1] : nullptr;
  g.out = static_cast<int32_t*>(out_dev);
  g.part = static_cast<int32_t*>(n->part);
  g.tickets = n->tickets;
  g.O = p.O;
  g.R = p.R;
  g.G = p.G;
  g.part_len = std::max<int64_t>(p.part, 1);
  g.W = p.W;
  const int64_t piece = 16 / p.esize;
  const bool vec = p.R % piece == 0 && g.part_len % piece == 0 && reinterpret_cast<uintptr_t>(g.a) % 16 == 0 &&
                   (!dot || reinterpret_cast<uintptr_t>(g.w) % 16 == 0);
  cudaError_t e;
  const int sms = n->sms;
  if (p.prec == HP_I8) {
    if (dot) e = launch_narrow_v<int8_t, 0, true>(p, g, vec, sms, st);
    else if (p.op == HP_RED_SUM) e = launch_narrow_v<int8_t, 0, false>(p, g, vec, sms, st);
    else if (p.op == HP_RED_MAX) e = launch_narrow_v<int8_t, 1, false>(p, g, vec, sms, st);
    else e = launch_narrow_v<int8_t, 2, false>(p, g, vec, sms, st);
  } else {
    if (p.op == HP_RED_SUM) e = launch_narrow_v<int16_t, 0, false>(p, g, vec, sms, st);
    else if (p.op == HP_RED_MAX) e = launch_narrow_v<int16_t, 1, false>(p, g, vec, sms, st);
    else e = launch_narrow_v<int16_t, 2, false>(p, g, vec, sms, st);
  }
  if (e != cudaSuccess) return fail(HP_ECUDA, std::string("narrow launch: ") + cudaGetErrorString(e));
  return HP_OK;
}

}  // namespace hp
