// csr.cu — ragged (CSR) nests: out[i] = OP_{e in [off[i], off[i+1])} val[e] * x[col[e]]
// and the count histogram hist[b] = #{e : col[e] >> shift == b}.
//
// The inner level is ragged, so its binding to hardware is chosen per row
// (Sec. 3.3: a region compiled for several candidate levels, one picked at run
// time; Sec. 3.8: sub-warp partitions for short rows).  Each run bins the rows
// by length into classes, and one persistent kernel takes units of them from a
// work counter (csr_work_kernel), the longest rows first:
//   class 0  len <= 4      one thread per row            (SEQ)
//   class 1  len <= 64     a group of 8 lanes per row     (SUBWARP(8))
//   class 2  len <= 2048   a warp per row                 (WARP)
//   class 3  len <= 16384  a CTA of 256 threads per row   (CTA)
//   class 4  longer        chunks of 16384 entries, a CTA per chunk writing
//                          its partial to the chunk's slot; a second pass
//                          folds each row's partials (GRID, two-pass;
//                          double-float for compensated sums).
// Within a class, lane t of a row's team folds entries start + t + k*L (L the
// team's lanes) into 4 accumulators (k mod 4), then the team combines them in
// a fixed tree; the tree depends on the row's length only, never on which
// team ran it or where the row sits in the class list, so results are
// reproducible although the class lists are filled with atomics.
// The histogram is counted in shared memory per CTA and flushed with 64-bit
// integer atomics (exact in any order), fused into the same sweep or alone.
// An explicit map for the entry level (SEQ, SUBWARP(w), WARP, CTA) puts every
// row into that one class instead.
// The x gathers are random 4-byte reads that L1 almost never serves again, so
// they are cached in L2 only (__ldcg): no L1 line fills for single use.
#include <cuda_runtime.h>

#include <algorithm>
#include <new>
#include <sstream>
#include <string>

#include "accum.cuh"
#include "api_internal.h"
#include "csr_sequence.h"

namespace hp {

constexpr int kCsrClasses = 5;
#ifndef HP_CSR_LIMIT1
#define HP_CSR_LIMIT1 64                                  // longest row of an 8-lane team (32: 6.44 ms, 64: 6.40, 128: 6.42 on the Zipf workload)
#endif
#ifndef HP_CSR_LIMIT2
#define HP_CSR_LIMIT2 2048                                // longest row of a warp team (1024: 6.42 ms, 2048: 6.37, 4096: 6.37)
#endif
#ifndef HP_CSR_LIMIT3
#define HP_CSR_LIMIT3 16384                               // longest row of a CTA team
#endif
#ifndef HP_CSR_CHUNK
#define HP_CSR_CHUNK 16384                                // entries per chunk of a longer row
#endif
constexpr int64_t kCsrLimit0 = 4, kCsrLimit1 = HP_CSR_LIMIT1, kCsrLimit2 = HP_CSR_LIMIT2, kCsrLimit3 = HP_CSR_LIMIT3;  // class bounds (inclusive)
constexpr int64_t kCsrChunk = HP_CSR_CHUNK;
static_assert(kCsrLimit3 >= kCsrChunk, "split rows must be longer than one chunk (bounds the chunk slots)");
constexpr int kCsrThreads = 256;                          // every kernel's CTA
// rows of one unit of work, by class: a chunk, a row, up to kCsrWarpRows rows per
// warp, up to kCsrTeamRows rows per 8-lane team, 8 rows per thread
constexpr int kCsrUnit0 = 8 * kCsrThreads, kCsrWarps = kCsrThreads / 32, kCsrTeams = kCsrThreads / 8;
// fewer where the CTAs would not get a unit each (rows of 64: 300 rows 22 and 11 us in
// a graph) or, when the nest's rows are long enough to hide a unit's claim, 8 each
// (rows of 2000, 4 rows per warp and now: 5000 rows, 157 units for 760 CTAs, 119 and 56 us;
// 50,000, whose 1562 units leave a last wave nearly empty, 446 and 379; rows of 100, 8 units
// each: 57 and 61)
constexpr int kCsrWarpRows = 4, kCsrTeamRows = 8;
constexpr int64_t kCsrLongRows = 512;   // entries per row, on average
// up to this many chunk slots the last CTA of the work kernel folds the long
// rows' partials; beyond, a kernel of its own does (25,000 rows would take one
// CTA about 200 us)
constexpr int64_t kCsrTailChunks = 1024;
constexpr int kCsrHistSmemMax = 12288;                   // bins counted in shared memory
#ifndef HP_CSR_GROUPS
#define HP_CSR_GROUPS 2                                   // 128-bit groups of col / val loaded before their folds
#endif
#ifndef HP_CSR_MIN_BLOCKS
#define HP_CSR_MIN_BLOCKS 5                               // resident CTAs per SM the wide-team kernels' registers allow (48 registers)
#endif

// Device counters.  They are zero between runs: the work kernel's last CTA
// clears them, so that a run needs no clearing launch of its own (csr_sequence.h
// has the runs that fail half-way).  Runs of one nest that overlap, which is not
// allowed, spoil each other's counts; every list position, row id and slot taken
// from them is bounded all the same and the run is flagged.
enum CsrCounter { kCntRows = 0 /* .. 4: rows per class */, kCntChunks = 5, kCntUnit = 6, kCntDone = 7,
                  kCntSlots = 8 /* chunk slots of the run, for the combine kernel; not cleared */, kCsrCounters = 16 };

struct CsrState {
  int64_t* counters = nullptr;
  int32_t* rows01 = nullptr;     // row ids: class 0 from the front, class 1 from the back
  int32_t* rows23 = nullptr;     // class 2 from the front, class 3 from the back
  int32_t* chunk_row = nullptr;  // per chunk slot: row id
  int32_t* chunk_idx = nullptr;  // per chunk slot: chunk index within its row
  int32_t* chunk_cnt = nullptr;  // per chunk slot: chunks of its row
  void* part = nullptr;          // per chunk slot: partial accumulator
  int64_t max_chunks = 0;
  int grid = 0;                  // CTAs of the persistent kernel
  bool dirty = false;            // counters left by a failed run (csr_enqueue)
};

// ---------------------------------------------------------------- planning
hp_status plan_csr(int depth, int64_t n_rows, const hp_level_map* map, hp_red_op op, int red_level, hp_prec prec,
                   hp_body body, const void* body_params, CsrPlan* out, std::string* why) {
  auto bad = [&](const std::string& s) {
    *why = s;
    return HP_EINVAL;
  };
  if (depth != 2) return bad("CSR nests have depth 2 (rows, entries)");
  if (n_rows < 0 || n_rows >= (int64_t(1) << 31)) return bad("CSR n_rows must be in [0, 2^31)");
  if (!body_params) return bad("CSR nests need hp_csr_params");
  const hp_csr_params* cp = static_cast<const hp_csr_params*>(body_params);
  if (cp->nnz < 0) return bad("CSR nnz must be >= 0");
  if (cp->n_cols < 0 || cp->n_cols >= (int64_t(1) << 31)) return bad("CSR n_cols must be in [0, 2^31)");
  if (op == HP_RED_HIST_COUNT || cp->fuse_hist) {
    if (cp->n_bins < 1 || cp->n_bins >= (int64_t(1) << 31)) return bad("histogram n_bins must be in [1, 2^31)");
    if (cp->hist_shift < 0 || cp->hist_shift > 30) return bad("histogram shift must be in [0, 30]");
  }
  if (op == HP_RED_HIST_COUNT) {
    if (red_level != 0) return bad("a count histogram reduces over all levels (red_level 0)");
    if (cp->fuse_hist) return bad("fuse_hist applies to SUM / MAX / MIN nests");
  } else {
    if (op != HP_RED_SUM && op != HP_RED_MAX && op != HP_RED_MIN) return bad("unknown reduction op");
    if (red_level != 1) return bad("CSR nests reduce the entries of each row (red_level 1)");
    if (body != HP_BODY_CSR_GATHER) return bad("CSR nests take the CSR_GATHER body");
    if (prec != HP_F32 && prec != HP_F32_COMP) return bad("CSR nests compute in FP32 (plain or compensated)");
  }
  CsrPlan p;
  p.n_rows = n_rows;
  p.nnz = cp->nnz;
  p.n_cols = cp->n_cols;
  p.hist_shift = cp->hist_shift;
  p.fuse_hist = cp->fuse_hist;
  p.n_bins = cp->n_bins;
  p.op = op;
  p.prec = prec;
  p.fixed_class = -1;
  if (map) {
    if (map[0].hw != HP_HW_GRID && map[0].hw != HP_HW_AUTO) return bad("CSR rows are bound to the grid");
    const int hw = map[1].hw;
    if (hw == HP_HW_AUTO) p.fixed_class = -1;
    else if (hw == HP_HW_SEQ || hw == HP_HW_LANE) p.fixed_class = 0;
    else if (hw == HP_HW_SUBWARP) {
      if (map[1].sub_width != 8 && map[1].sub_width != 0) return bad("CSR sub-warp rows use groups of 8 lanes");
      p.fixed_class = 1;
    } else if (hw == HP_HW_WARP) p.fixed_class = 2;
    else if (hw == HP_HW_CTA) p.fixed_class = 3;
    else if (hw == HP_HW_GRID) p.fixed_class = 4;
    else return bad("CSR entries bind to SEQ, SUBWARP(8), WARP, CTA, GRID or AUTO");
  }
  *out = p;
  return HP_OK;
}

std::string describe_csr(const CsrPlan& p) {
  std::ostringstream s;
  s << "{\"kind\":\"csr\",\"rows\":" << p.n_rows << ",\"nnz\":" << p.nnz << ",\"cols\":" << p.n_cols
    << ",\"op\":" << static_cast<int>(p.op) << ",\"fuse_hist\":" << p.fuse_hist << ",\"bins\":" << p.n_bins
    << ",\"shift\":" << p.hist_shift << ",\"fixed_class\":" << p.fixed_class
    << ",\"class_limits\":[" << kCsrLimit0 << "," << kCsrLimit1 << "," << kCsrLimit2 << "," << kCsrLimit3
    << "],\"chunk\":" << kCsrChunk << "}";
  return s.str();
}

// ---------------------------------------------------------------- device code
namespace {

__device__ __forceinline__ int row_class(int64_t len, int fixed) {
  if (fixed >= 0) return fixed;
  if (len <= kCsrLimit0) return 0;
  if (len <= kCsrLimit1) return 1;
  if (len <= kCsrLimit2) return 2;
  if (len <= kCsrLimit3) return 3;
  return 4;
}

__device__ __forceinline__ int64_t n_chunks_of(int64_t len) { return len > 0 ? (len + kCsrChunk - 1) / kCsrChunk : 1; }

__device__ __forceinline__ void zero_hist(long long* hist, int64_t n_bins) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n_bins; i += stride) hist[i] = 0;
}
__global__ void csr_zero_kernel(long long* hist, int64_t n_bins) { zero_hist(hist, n_bins); }

// where row k of class c sits in the row lists
__device__ __forceinline__ int64_t list_at(int c, int64_t k, int64_t n_rows) { return (c & 1) ? n_rows - 1 - k : k; }

// Binning: row ids into their class's list (tile by tile: warp ballots give
// each row its rank, one global add per block and class reserves the tile's
// range) and chunk slots of long rows.  Two classes share a list from its two
// ends, so no counting pass has to place them.  Also clears the fused histogram.
__global__ void __launch_bounds__(kCsrThreads) csr_bin_kernel(const int64_t* __restrict__ off, int64_t n_rows, int fixed,
                                                              int64_t* counters, int32_t* rows01, int32_t* rows23,
                                                              int32_t* chunk_row, int32_t* chunk_idx,
                                                              int32_t* chunk_cnt, int64_t max_chunks, int32_t* err,
                                                              long long* hist, int64_t n_bins) {
  constexpr int kWarps = kCsrThreads / 32;
  __shared__ int wpos[kWarps][kCsrClasses];
  __shared__ long long bbase[kCsrClasses];
  grid_launch_dependents();   // the work kernel clears its shared histogram meanwhile
  if (hist) zero_hist(hist, n_bins);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t tile = blockIdx.x * static_cast<int64_t>(blockDim.x); tile < n_rows; tile += stride) {
    const int64_t i = tile + threadIdx.x;
    int c = -1;
    int64_t len = 0;
    if (i < n_rows) {
      len = off[i + 1] - off[i];
      c = row_class(len, fixed);
    }
    int rank = 0;
#pragma unroll
    for (int k = 0; k < kCsrClasses; ++k) {
      const unsigned m = __ballot_sync(0xffffffffu, c == k);
      if (lane == 0) wpos[warp][k] = __popc(m);
      if (c == k) rank = __popc(m & lt_mask);
    }
    __syncthreads();
    if (threadIdx.x < kCsrClasses) {
      int tot = 0;
      for (int w = 0; w < kWarps; ++w) {
        const int v = wpos[w][threadIdx.x];
        wpos[w][threadIdx.x] = tot;
        tot += v;
      }
      bbase[threadIdx.x] =
          tot ? static_cast<long long>(atomicAdd(reinterpret_cast<unsigned long long*>(&counters[kCntRows + threadIdx.x]),
                                                 static_cast<unsigned long long>(tot)))
              : 0;
    }
    __syncthreads();
    if (c >= 0 && c < 4) {
      const int64_t k = bbase[c] + wpos[warp][c] + rank;
      if (k < n_rows) (c < 2 ? rows01 : rows23)[list_at(c, k, n_rows)] = static_cast<int32_t>(i);
      else atomicExch(err, 2);           // counters of another run
    }
    if (c == 4) {
      const int64_t nc = n_chunks_of(len);
      const unsigned long long base =
          atomicAdd(reinterpret_cast<unsigned long long*>(&counters[kCntChunks]), static_cast<unsigned long long>(nc));
      if (static_cast<int64_t>(base) + nc > max_chunks) {  // offsets disagree with the declared nnz
        atomicExch(err, 2);
      } else {
        for (int64_t k = 0; k < nc; ++k) {
          chunk_row[base + k] = static_cast<int32_t>(i);
          chunk_idx[base + k] = static_cast<int32_t>(k);
          chunk_cnt[base + k] = static_cast<int32_t>(nc);
        }
      }
    }
    __syncthreads();  // wpos / bbase are reused by the next tile
  }
}

struct CsrArgs {
  const int64_t* off;
  const int32_t* col;
  const float* val;
  const float* x;
  float* y;
  long long* hist;      // fused histogram (global), or nullptr
  int32_t* err;         // device error word: 2 = offsets or columns outside the declared sizes
  int64_t nnz;
  int64_t n_cols;
  int shift;
  int64_t n_bins;
  int smem_bins;        // bins counted in shared memory (0: count straight into global memory)
};

__device__ __forceinline__ void hist_add(const CsrArgs& a, int* sh, int32_t c) {
  const int64_t b = static_cast<int64_t>(c) >> a.shift;
  if (b < a.n_bins) {
    if (a.smem_bins) atomicAdd(&sh[b], 1);
    else atomicAdd(reinterpret_cast<unsigned long long*>(&a.hist[b]), 1ull);
  }
}

// fold entries s + t, s + t + L, ... < e into 4 accumulators (entry k goes to acc[(k / L) % 4])
template <class Op, bool HIST>
__device__ __forceinline__ void csr_fold(const CsrArgs& a, int* sh, int64_t s, int64_t e, int t, int L,
                                         typename Op::Acc (&acc)[4]) {
  if (s < 0 || e > a.nnz || s > e) {  // offsets outside [0, nnz]: flag, fold nothing
    if (t == 0) atomicExch(a.err, 2);
    return;
  }
  for (int64_t b = s + t; b < e; b += 4 * static_cast<int64_t>(L)) {
    int32_t c[4];
    float v[4];
    bool ok[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t idx = b + static_cast<int64_t>(u) * L;
      ok[u] = idx < e;
      c[u] = ok[u] ? __ldcs(a.col + idx) : 0;
      v[u] = ok[u] ? __ldcs(a.val + idx) : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (ok[u]) {
        if (static_cast<uint32_t>(c[u]) < static_cast<uint64_t>(a.n_cols)) {
          Op::add_prod(acc[u], v[u], __ldcg(a.x + c[u]));
          if constexpr (HIST) hist_add(a, sh, c[u]);
        } else {
          atomicExch(a.err, 2);
        }
      }
    }
  }
}

template <class Op, bool HIST>
__device__ __forceinline__ void csr_fold_one(const CsrArgs& a, int* sh, int64_t idx, typename Op::Acc& acc) {
  const int32_t c = __ldcs(a.col + idx);
  const float v = __ldcs(a.val + idx);
  if (static_cast<uint32_t>(c) < static_cast<uint64_t>(a.n_cols)) {
    Op::add_prod(acc, v, __ldcg(a.x + c));
    if constexpr (HIST) hist_add(a, sh, c);
  } else {
    atomicExch(a.err, 2);
  }
}

template <class Op, bool HIST>
__device__ __forceinline__ void csr_fold_group(const CsrArgs& a, int* sh, const int4& c, const float4& v,
                                               typename Op::Acc (&acc)[4]) {
  const int32_t cc[4] = {c.x, c.y, c.z, c.w};
  const float vv[4] = {v.x, v.y, v.z, v.w};
  float xv[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
    xv[u] = (static_cast<uint32_t>(cc[u]) < static_cast<uint64_t>(a.n_cols)) ? __ldcg(a.x + cc[u]) : 0.0f;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (static_cast<uint32_t>(cc[u]) < static_cast<uint64_t>(a.n_cols)) {
      Op::add_prod(acc[u], vv[u], xv[u]);
      if constexpr (HIST) hist_add(a, sh, cc[u]);
    } else {
      atomicExch(a.err, 2);
    }
  }
}

// Entries [s, e) for wide teams: the 16-byte-aligned middle is read as 128-bit
// groups of col and val (lane t takes groups g0 + t, g0 + t + L, ...,
// HP_CSR_GROUPS at a time so that 4 x HP_CSR_GROUPS gathers of x are in
// flight; the fold order does not depend on it), the unaligned head and tail
// (< 4 entries each) by lanes 0..3 into their first and second accumulators.
// The tree depends only on (s, e), so a row's result is reproducible.
template <class Op, bool HIST>
__device__ __forceinline__ void csr_fold_vec(const CsrArgs& a, int* sh, int64_t s, int64_t e, int t, int L,
                                             typename Op::Acc (&acc)[4]) {
  if (s < 0 || e > a.nnz || s > e) {
    if (t == 0) atomicExch(a.err, 2);
    return;
  }
  const int64_t g0 = (s + 3) >> 2, g1 = e >> 2;
  if (g0 >= g1) {
    csr_fold<Op, HIST>(a, sh, s, e, t, L, acc);
    return;
  }
  if (t < 4 * g0 - s) csr_fold_one<Op, HIST>(a, sh, s + t, acc[0]);
  if (t < e - 4 * g1) csr_fold_one<Op, HIST>(a, sh, 4 * g1 + t, acc[1]);
  const int4* col4 = reinterpret_cast<const int4*>(a.col);
  const float4* val4 = reinterpret_cast<const float4*>(a.val);
  constexpr int K = HP_CSR_GROUPS;
  for (int64_t g = g0 + t; g < g1; g += K * static_cast<int64_t>(L)) {
    int4 c[K];
    float4 v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      c[k] = make_int4(0, 0, 0, 0);
      v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (g + k * static_cast<int64_t>(L) < g1) {
        c[k] = __ldcs(col4 + g + k * static_cast<int64_t>(L));
        v[k] = __ldcs(val4 + g + k * static_cast<int64_t>(L));
      }
    }
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (g + k * static_cast<int64_t>(L) < g1) csr_fold_group<Op, HIST>(a, sh, c[k], v[k], acc);
  }
}

template <class Op>
__device__ __forceinline__ typename Op::Acc fold4(const typename Op::Acc (&acc)[4]) {
  return Op::combine(Op::combine(acc[0], acc[1]), Op::combine(acc[2], acc[3]));
}

template <class Op>
__device__ __forceinline__ typename Op::Acc team_reduce(typename Op::Acc a, int width) {
  for (int m = width >> 1; m >= 1; m >>= 1) a = Op::combine(a, Op::shfl_xor(a, m, width));
  return a;
}

__device__ __forceinline__ void hist_init(int* sh, int bins) {
  for (int i = threadIdx.x; i < bins; i += blockDim.x) sh[i] = 0;
  __syncthreads();
}

__device__ __forceinline__ void hist_flush(const CsrArgs& a, int* sh) {
  __syncthreads();
  for (int i = threadIdx.x; i < a.smem_bins; i += blockDim.x)
    if (sh[i]) atomicAdd(reinterpret_cast<unsigned long long*>(&a.hist[i]), static_cast<unsigned long long>(sh[i]));
}

// CTA-wide fold of one entry range; the result is valid in thread 0.  One
// barrier: callers alternate between the two halves of their warp-partial
// buffer, so that the next range's partials never overwrite the ones thread 0
// may still be reading.
template <class Op, bool HIST>
__device__ __forceinline__ typename Op::Acc cta_fold(const CsrArgs& a, int* sh, int64_t s, int64_t e,
                                                     typename Op::Acc* wsh) {
  typename Op::Acc acc[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) acc[u] = Op::ident();
  csr_fold_vec<Op, HIST>(a, sh, s, e, threadIdx.x, blockDim.x, acc);
  typename Op::Acc r = team_reduce<Op>(fold4<Op>(acc), 32);
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) wsh[warp] = r;
  __syncthreads();
  if (threadIdx.x == 0) {
    r = wsh[0];
    for (int w = 1; w < nw; ++w) r = Op::combine(r, wsh[w]);
  }
  return r;
}

// a long row's partials (the second pass of Sec. 2's recursive reduction at
// grid level): the thread of the row's first slot folds them with the grid-part
// combine (combine_parts), a fixed tree per row
template <class Op>
__device__ __forceinline__ void combine_slot(int64_t k, int64_t n_slots, float* y, const int32_t* chunk_row,
                                             const int32_t* chunk_idx, const int32_t* chunk_cnt,
                                             const typename Op::Acc* part) {
  if (chunk_idx[k] != 0) return;
  const int n = chunk_cnt[k];
  if (n < 1 || k + n > n_slots) return;   // a row the binning could not place whole (flagged there)
  y[chunk_row[k]] = combine_parts<Op>(part + k, n, nullptr);
}
template <class Op>
__global__ void csr_split_combine_kernel(float* __restrict__ y, const int64_t* counters,
                                         const int32_t* __restrict__ chunk_row, const int32_t* __restrict__ chunk_idx,
                                         const int32_t* __restrict__ chunk_cnt, const typename Op::Acc* __restrict__ part) {
  const int64_t n_slots = counters[kCntSlots];
  for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < n_slots;
       k += static_cast<int64_t>(gridDim.x) * blockDim.x)
    combine_slot<Op>(k, n_slots, y, chunk_row, chunk_idx, chunk_cnt, part);
}

struct CsrLists {
  int64_t* counters;
  const int32_t* rows01;
  const int32_t* rows23;
  const int32_t* chunk_row;
  const int32_t* chunk_idx;
  const int32_t* chunk_cnt;
  int64_t n_rows, max_chunks;
  int tail_combine;           // 1: the last CTA folds the long rows' partials
  uint32_t units;             // of the warp class, per CTA, that its rows per warp leave
};

// All classes in one persistent kernel: units are taken from a counter, chunks
// of the longest rows first, single-thread rows last, so one class's waits are
// filled with another's gathers and only the last units leave SMs idle.  (One
// kernel per class ran them one after the other, each with its own tail and its
// own flush of the histogram: 6.37 ms for 4.2 M rows, and nine launches, 61 us,
// for 300.)  The next unit is claimed before the current one is folded.
template <class Op, bool HIST>
__global__ void __launch_bounds__(kCsrThreads, HP_CSR_MIN_BLOCKS) csr_work_kernel(const CsrArgs a, const CsrLists l,
                                                                                typename Op::Acc* part) {
  using Acc = typename Op::Acc;
  extern __shared__ int sh_hist[];
  __shared__ Acc wsh[2][kCsrThreads / 32];
  __shared__ uint32_t s_unit, s_first[kCsrClasses], s_rows[3], s_per[3], s_end;   // s_per: rows per team and unit
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned long long* const claim = reinterpret_cast<unsigned long long*>(&l.counters[kCntUnit]);
  if constexpr (HIST) {
    if (a.smem_bins) hist_init(sh_hist, a.smem_bins);
  }
  grid_wait();   // the binning
  if (tid == 0) s_unit = static_cast<uint32_t>(atomicAdd(claim, 1ull));
  // the classes' sizes and their first units, longest rows first (fewer than 2^32
  // units: rows and chunks are below 2^31); in shared memory, to spare registers
  if (tid == 0) {
    const int64_t slots = l.counters[kCntChunks] < l.max_chunks ? l.counters[kCntChunks] : l.max_chunks;
    for (int c = 0; c < 3; ++c) s_rows[c] = static_cast<uint32_t>(min(l.counters[c], l.n_rows));
    s_first[4] = 0;
    s_first[3] = static_cast<uint32_t>(slots);
    s_first[2] = s_first[3] + static_cast<uint32_t>(min(l.counters[3], l.n_rows));
    for (int c = 2; c >= 1; --c) {
      const uint32_t teams = c == 2 ? kCsrWarps : kCsrTeams;
      uint32_t per = c == 2 ? kCsrWarpRows : kCsrTeamRows;
      while (per > 1 && s_rows[c] < (c == 2 ? l.units : 1) * gridDim.x * (teams * per)) per /= 2;
      s_per[c] = per;
      s_first[c - 1] = s_first[c] + (s_rows[c] + teams * per - 1) / (teams * per);
    }
    s_end = s_first[0] + (s_rows[0] + kCsrUnit0 - 1) / kCsrUnit0;
  }
  __syncthreads();
  int buf = 0;
  while (true) {
    const uint32_t u = s_unit;
    __syncthreads();   // every thread has read it
    if (u >= s_end) break;
    uint32_t next = 0;
    if (tid == 0) next = static_cast<uint32_t>(atomicAdd(claim, 1ull));
    if (u < s_first[2]) {      // a chunk of a long row, or a row of the CTA class
      int64_t s, e;
      int32_t row;
      const bool chunk = u < s_first[3];
      if (chunk) {
        row = l.chunk_row[u];
        s = a.off[row] + l.chunk_idx[u] * kCsrChunk;
        e = a.off[row + 1];
        if (s + kCsrChunk < e) e = s + kCsrChunk;
      } else {
        row = l.rows23[list_at(3, u - s_first[3], l.n_rows)];
        s = a.off[row];
        e = a.off[row + 1];
      }
      const Acc r = cta_fold<Op, HIST>(a, sh_hist, s, e, wsh[buf]);
      buf ^= 1;
      if (tid == 0) {
        if (chunk) part[u] = r;
        else a.y[row] = Op::finish(r);
      }
    } else if (u < s_first[1]) {   // `per` rows per warp; lane i reads the i-th one's place
      const uint32_t per = s_per[2], k0 = ((u - s_first[2]) * kCsrWarps + warp) * per;
      const int n = k0 >= s_rows[2] ? 0 : static_cast<int>(min(s_rows[2] - k0, per));
      int32_t id = 0;
      int64_t s = 0, e = 0;
      if (lane < n) {
        id = l.rows23[list_at(2, k0 + lane, l.n_rows)];
        s = a.off[id];
        e = a.off[id + 1];
      }
      for (int i = 0; i < n; ++i) {
        Acc acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = Op::ident();
        csr_fold_vec<Op, HIST>(a, sh_hist, __shfl_sync(0xffffffffu, s, i), __shfl_sync(0xffffffffu, e, i), lane, 32, acc);
        const Acc r = team_reduce<Op>(fold4<Op>(acc), 32);
        if (lane == i) a.y[id] = Op::finish(r);
      }
    } else if (u < s_first[0]) {   // 8 lanes per row, 4 `per` rows per warp
      const uint32_t per = s_per[1], k0 = ((u - s_first[1]) * kCsrWarps + warp) * (4 * per);
      int32_t id = -1;
      int64_t s = 0, e = 0;
      if (lane < 4 * per && k0 + lane < s_rows[1]) {
        id = l.rows01[list_at(1, k0 + lane, l.n_rows)];
        s = a.off[id];
        e = a.off[id + 1];
      }
      for (int i = 0; i < static_cast<int>(per); ++i) {
        const int src = 4 * i + (lane >> 3);
        const int32_t row = __shfl_sync(0xffffffffu, id, src);
        const int64_t rs = __shfl_sync(0xffffffffu, s, src), re = __shfl_sync(0xffffffffu, e, src);
        Acc acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = Op::ident();
        if (row >= 0) csr_fold<Op, HIST>(a, sh_hist, rs, re, lane & 7, 8, acc);
        const Acc r = team_reduce<Op>(fold4<Op>(acc), 8);
        if (row >= 0 && (lane & 7) == 0) a.y[row] = Op::finish(r);
      }
    } else {               // a thread per row
      const uint32_t k0 = (u - s_first[0]) * kCsrUnit0 + tid;
      for (int i = 0; i < kCsrUnit0 / kCsrThreads; ++i) {
        const uint32_t k = k0 + i * kCsrThreads;
        if (k >= s_rows[0]) break;
        const int32_t row = l.rows01[list_at(0, k, l.n_rows)];
        Acc acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = Op::ident();
        csr_fold<Op, HIST>(a, sh_hist, a.off[row], a.off[row + 1], 0, 1, acc);
        a.y[row] = Op::finish(fold4<Op>(acc));
      }
    }
    if (tid == 0) s_unit = next;
    __syncthreads();
  }
  if constexpr (HIST) {
    if (a.smem_bins) hist_flush(a, sh_hist);
  }
  // the last CTA to get here clears the counters for the next run
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(reinterpret_cast<unsigned long long*>(&l.counters[kCntDone]), 1ull) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();   // the partials of every CTA are visible
  if (l.tail_combine)
    for (int64_t k = tid; k < s_first[3]; k += kCsrThreads)
      combine_slot<Op>(k, s_first[3], a.y, l.chunk_row, l.chunk_idx, l.chunk_cnt, part);
  if (tid == 0) l.counters[kCntSlots] = s_first[3];
  if (tid <= kCntDone) l.counters[tid] = 0;
}

// standalone count histogram over all entries
__global__ void __launch_bounds__(256) csr_hist_kernel(const int32_t* __restrict__ col, int64_t nnz, int shift,
                                                       int64_t n_bins, int smem_bins, long long* hist) {
  extern __shared__ int sh_hist[];
  if (smem_bins) hist_init(sh_hist, smem_bins);
  CsrArgs a{};
  a.hist = hist;
  a.shift = shift;
  a.n_cols = 0;
  a.n_bins = n_bins;
  a.smem_bins = smem_bins;
  const int64_t n4 = nnz / 4;
  const int4* col4 = reinterpret_cast<const int4*>(col);
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n4;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int4 c = __ldcs(col4 + i);
    hist_add(a, sh_hist, c.x);
    hist_add(a, sh_hist, c.y);
    hist_add(a, sh_hist, c.z);
    hist_add(a, sh_hist, c.w);
  }
  for (int64_t i = n4 * 4 + blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < nnz;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    hist_add(a, sh_hist, __ldcs(col + i));
  if (smem_bins) hist_flush(a, sh_hist);
}

inline hp_status cuda_fail(cudaError_t e, const char* what) {
  return fail(HP_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// the attribute belongs to the kernel (shared by every nest): always the
// largest histogram any nest counts in shared memory
template <class K>
hp_status set_smem(K kernel, size_t dyn) {
  if (dyn == 0) return HP_OK;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(kCsrHistSmemMax * sizeof(int)));
  return e == cudaSuccess ? HP_OK : cuda_fail(e, "CSR kernel shared memory");
}

// one run of a nest with entries (csr_enqueue)
template <class Op, bool HIST>
struct CsrRun {
  hp_nest* n;
  const CsrArgs& a;
  cudaStream_t st;
  size_t dyn() const { return HIST ? static_cast<size_t>(a.smem_bins) * sizeof(int) : 0; }
  hp_status prepare() { return set_smem(csr_work_kernel<Op, HIST>, dyn()); }
  hp_status clear() {
    const cudaError_t e = cudaMemsetAsync(n->cs->counters, 0, kCsrCounters * sizeof(int64_t), st);
    return e == cudaSuccess ? HP_OK : HP_ECUDA;   // the message stays the failed launch's
  }
  hp_status bin() {
    const CsrPlan& p = n->csr;
    const CsrState& cs = *n->cs;
    // enough CTAs for the rows and for the histogram's bins, which it clears (100 rows, 2^24
    // bins: 2057 us with the rows' one CTA)
    const int64_t most = std::max<int64_t>(p.n_rows, a.hist ? p.n_bins : 0);
    const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((most + kCsrThreads - 1) / kCsrThreads, 8 * n->sms)));
    csr_bin_kernel<<<grid, kCsrThreads, 0, st>>>(a.off, p.n_rows, p.fixed_class, cs.counters, cs.rows01, cs.rows23,
                                                 cs.chunk_row, cs.chunk_idx, cs.chunk_cnt, cs.max_chunks, n->err, a.hist,
                                                 p.n_bins);
    const cudaError_t e = cudaPeekAtLastError();
    return e == cudaSuccess ? HP_OK : cuda_fail(e, "CSR binning launch");
  }
  hp_status work() {
    const CsrState& cs = *n->cs;
    const bool tail = cs.max_chunks <= kCsrTailChunks;
    const CsrLists l{cs.counters, cs.rows01, cs.rows23, cs.chunk_row, cs.chunk_idx, cs.chunk_cnt,
                     n->csr.n_rows, cs.max_chunks, tail ? 1 : 0, n->csr.nnz >= kCsrLongRows * n->csr.n_rows ? 8u : 1u};
    typename Op::Acc* part = static_cast<typename Op::Acc*>(cs.part);
    const cudaError_t w = launch_dependent(csr_work_kernel<Op, HIST>, cs.grid, kCsrThreads, dyn(), st, a, l, part);
    if (w != cudaSuccess) return cuda_fail(w, "CSR work kernel launch");
    if (!tail) {
      const int cgrid = static_cast<int>(std::min<int64_t>((cs.max_chunks + 255) / 256, 4 * n->sms));
      csr_split_combine_kernel<Op><<<cgrid, 256, 0, st>>>(a.y, cs.counters, cs.chunk_row, cs.chunk_idx, cs.chunk_cnt, part);
    }
    const cudaError_t e = cudaPeekAtLastError();
    return e == cudaSuccess ? HP_OK : cuda_fail(e, "CSR work kernel launch");
  }
};

template <class Op>
hp_status launch_op(hp_nest* n, const CsrArgs& a, cudaStream_t st) {
  if (a.hist) {
    CsrRun<Op, true> r{n, a, st};
    return csr_enqueue(r, &n->cs->dirty, HP_OK);
  }
  CsrRun<Op, false> r{n, a, st};
  return csr_enqueue(r, &n->cs->dirty, HP_OK);
}

int smem_bins_for(int64_t n_bins) { return n_bins <= kCsrHistSmemMax ? static_cast<int>(n_bins) : 0; }

}  // namespace

// ---------------------------------------------------------------- host side
hp_status csr_prepare(hp_nest* n, InitStream& init) {
  const CsrPlan& p = n->csr;
  CsrState* cs = new (std::nothrow) CsrState();
  if (!cs) return fail(HP_ENOMEM, "host allocation failed");
  n->cs = cs;
  cudaError_t e;
  e = cudaMalloc(&cs->counters, kCsrCounters * sizeof(int64_t));
  if (e != cudaSuccess) return fail(HP_ENOMEM, "cudaMalloc (CSR counters)");
  e = init.zero(cs->counters, kCsrCounters * sizeof(int64_t));
  if (e != cudaSuccess) return cuda_fail(e, "clear CSR counters");
  if (p.op == HP_RED_HIST_COUNT) return HP_OK;
  const int64_t rows = std::max<int64_t>(p.n_rows, 1);
  // long rows have > kCsrChunk entries, so chunk slots <= 2 * nnz / kCsrChunk + 1
  cs->max_chunks = 2 * (p.nnz / kCsrChunk) + 2;
  if (p.fixed_class == 4) cs->max_chunks = p.nnz / kCsrChunk + p.n_rows + 2;
  if (cudaMalloc(&cs->rows01, rows * sizeof(int32_t)) != cudaSuccess ||
      cudaMalloc(&cs->rows23, rows * sizeof(int32_t)) != cudaSuccess)
    return fail(HP_ENOMEM, "cudaMalloc (CSR row lists)");
  const size_t mc = static_cast<size_t>(cs->max_chunks);
  if (cudaMalloc(&cs->chunk_row, mc * sizeof(int32_t)) != cudaSuccess ||
      cudaMalloc(&cs->chunk_idx, mc * sizeof(int32_t)) != cudaSuccess ||
      cudaMalloc(&cs->chunk_cnt, mc * sizeof(int32_t)) != cudaSuccess ||
      cudaMalloc(&cs->part, mc * sizeof(f2)) != cudaSuccess)
    return fail(HP_ENOMEM, "cudaMalloc (CSR chunk tables)");
  // every slot starts as a valid (row 0, chunk 0) entry and every list place as
  // row 0, so that one the binning did not fill (offsets beyond the declared
  // nnz, flagged) reads in bounds
  for (int32_t* t : {cs->chunk_row, cs->chunk_idx, cs->chunk_cnt}) {
    e = init.zero(t, mc * sizeof(int32_t));
    if (e != cudaSuccess) return cuda_fail(e, "clear chunk tables");
  }
  for (int32_t* t : {cs->rows01, cs->rows23}) {
    e = init.zero(t, rows * sizeof(int32_t));
    if (e != cudaSuccess) return cuda_fail(e, "clear row lists");
  }
  // the attribute first: with close to 12288 bins the kernel's shared memory exceeds
  // 48 KiB, and without it the query answers 0 CTAs (400,000 rows of 40 with 12288
  // bins: 439 us on one CTA per SM, 167 on four)
  const size_t dyn = p.fuse_hist ? smem_bins_for(p.n_bins) * sizeof(int) : 0;
  const hp_status attr = set_smem(csr_work_kernel<OpF32Comp, true>, dyn);
  if (attr != HP_OK) return attr;
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, csr_work_kernel<OpF32Comp, true>, kCsrThreads, dyn);
  // a CTA per 4096 entries and 1024 rows where that is fewer than fit
  const int64_t want = p.nnz / 4096 + p.n_rows / 1024 + 1;
  cs->grid = static_cast<int>(std::min<int64_t>(want, static_cast<int64_t>(std::max(1, per_sm)) * n->sms));
  return HP_OK;
}

hp_status run_csr(hp_nest* n, const void* const* in_dev, void* out_dev, cudaStream_t st) {
  const CsrPlan& p = n->csr;
  CsrState& cs = *n->cs;
  if (!in_dev) return fail(HP_EINVAL, "in_dev is NULL");
  if (!out_dev) return fail(HP_EINVAL, "out_dev is NULL");
  if (p.op == HP_RED_HIST_COUNT) {
    const int32_t* col = static_cast<const int32_t*>(in_dev[1]);
    if (!col && p.nnz > 0) return fail(HP_EINVAL, "missing col");
    if (reinterpret_cast<uintptr_t>(col) & 15u) return fail(HP_EINVAL, "col must be 16-byte aligned");
    long long* hist = static_cast<long long*>(out_dev);
    csr_zero_kernel<<<std::max<int64_t>(1, std::min<int64_t>((p.n_bins + 255) / 256, 4 * n->sms)), 256, 0, st>>>(
        hist, p.n_bins);
    const int sb = smem_bins_for(p.n_bins);
    const size_t dyn = static_cast<size_t>(sb) * sizeof(int);
    hp_status s = set_smem(csr_hist_kernel, dyn);
    if (s != HP_OK) return s;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, csr_hist_kernel, 256, dyn);
    const int64_t want = (p.nnz / 4 + 255) / 256;
    const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(want, std::max(1, per_sm) * n->sms)));
    csr_hist_kernel<<<grid, 256, dyn, st>>>(col, p.nnz, p.hist_shift, p.n_bins, sb, hist);
    const cudaError_t e = cudaPeekAtLastError();
    return e == cudaSuccess ? HP_OK : cuda_fail(e, "CSR histogram launch");
  }
  for (int i = 0; i < 4; ++i)
    if (!in_dev[i]) return fail(HP_EINVAL, "missing CSR input " + std::to_string(i));
  if ((reinterpret_cast<uintptr_t>(in_dev[1]) | reinterpret_cast<uintptr_t>(in_dev[2])) & 15u)
    return fail(HP_EINVAL, "CSR col and val must be 16-byte aligned (128-bit loads)");
  CsrArgs a{};
  a.off = static_cast<const int64_t*>(in_dev[0]);
  a.col = static_cast<const int32_t*>(in_dev[1]);
  a.val = static_cast<const float*>(in_dev[2]);
  a.x = static_cast<const float*>(in_dev[3]);
  a.y = static_cast<float*>(out_dev);
  a.hist = nullptr;
  a.err = n->err;
  a.nnz = p.nnz;
  a.n_cols = p.n_cols;
  if (p.fuse_hist) {
    a.hist = static_cast<long long*>(const_cast<void*>(in_dev[4]));
    if (!a.hist) return fail(HP_EINVAL, "fuse_hist needs the histogram output in in_dev[4]");
    a.shift = p.hist_shift;
    a.n_bins = p.n_bins;
    a.smem_bins = smem_bins_for(p.n_bins);
  }
  if (p.n_rows == 0) return HP_OK;
  switch (p.op) {
    case HP_RED_SUM:
      return p.prec == HP_F32_COMP ? launch_op<OpF32Comp>(n, a, st) : launch_op<OpF32Sum>(n, a, st);
    case HP_RED_MAX:
      return launch_op<OpF32Max>(n, a, st);
    case HP_RED_MIN:
      return launch_op<OpF32Min>(n, a, st);
    default:
      return fail(HP_EINVAL, "bad CSR op");
  }
}

// ---------------------------------------------------------------- gather-rate probe
namespace {

// counter hash (murmur3's 32-bit finalizer over index ^ seed): uniform indices
__device__ __forceinline__ uint32_t probe_hash(uint64_t i, uint32_t seed) {
  uint32_t h = static_cast<uint32_t>(i) ^ static_cast<uint32_t>(i >> 32) * 0x9e3779b9u ^ seed;
  h ^= h >> 16;
  h *= 0x85ebca6bu;
  h ^= h >> 13;
  h *= 0xc2b2ae35u;
  h ^= h >> 16;
  return h;
}

// n random 4-byte reads of x through the CSR executor's x-gather path (__ldcg:
// cached in L2 only), 8 independent reads in flight per thread per round;
// each block adds its sum to *out so that no read is dead code
__global__ void __launch_bounds__(256) gather_probe_kernel(const float* __restrict__ x, uint32_t n_x, int64_t n,
                                                           uint32_t seed, float* out) {
  __shared__ float wsum[8];
  float acc = 0.0f;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  for (; i + 7 * stride < n; i += 8 * stride) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t h = probe_hash(static_cast<uint64_t>(i + u * stride), seed);
      v[u] = __ldcg(x + static_cast<uint32_t>((static_cast<uint64_t>(h) * n_x) >> 32));
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) acc += v[u];
  }
  for (; i < n; i += stride) {
    const uint32_t h = probe_hash(static_cast<uint64_t>(i), seed);
    acc += __ldcg(x + static_cast<uint32_t>((static_cast<uint64_t>(h) * n_x) >> 32));
  }
  for (int m = 16; m >= 1; m >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t += wsum[w];
    atomicAdd(out, t);
  }
}

}  // namespace

size_t csr_out_bytes(const hp_nest* n) {
  return n->csr.op == HP_RED_HIST_COUNT ? static_cast<size_t>(n->csr.n_bins) * 8
                                        : static_cast<size_t>(n->csr.n_rows) * 4;
}

void csr_release(hp_nest* n) {
  CsrState* cs = n->cs;
  if (!cs) return;
  cudaFree(cs->counters);
  cudaFree(cs->rows01);
  cudaFree(cs->rows23);
  cudaFree(cs->chunk_row);
  cudaFree(cs->chunk_idx);
  cudaFree(cs->chunk_cnt);
  cudaFree(cs->part);
  delete cs;
  n->cs = nullptr;
}

}  // namespace hp

extern "C" hp_status hp_probe_gather(const float* x_dev, int64_t n_x, int64_t n_gathers, uint32_t seed, float* sum_dev,
                                     void* stream) {
  using namespace hp;
  if (!x_dev || !sum_dev) return fail(HP_EINVAL, "x_dev and sum_dev must be device pointers");
  if (n_x < 1 || n_x > (int64_t(1) << 32) - 1) return fail(HP_EINVAL, "n_x must be in [1, 2^32)");
  if (n_gathers < 0) return fail(HP_EINVAL, "n_gathers must be >= 0");
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gather_probe_kernel, 256, 0);
  if (e != cudaSuccess) return cuda_fail(e, "gather probe set-up");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  e = cudaMemsetAsync(sum_dev, 0, sizeof(float), st);
  if (e != cudaSuccess) return cuda_fail(e, "gather probe memset");
  if (n_gathers == 0) return HP_OK;
  const int64_t want = (n_gathers + 255) / 256;
  const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(want, static_cast<int64_t>(std::max(1, per_sm)) * sms)));
  gather_probe_kernel<<<grid, 256, 0, st>>>(x_dev, static_cast<uint32_t>(n_x), n_gathers, seed, sum_dev);
  e = cudaPeekAtLastError();
  return e == cudaSuccess ? HP_OK : cuda_fail(e, "gather probe launch");
}
