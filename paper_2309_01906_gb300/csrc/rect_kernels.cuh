// rect_kernels.cuh — the rectangular nest executor (device code).
//
// One output of the nest is combined by a team (plan.cpp decides which):
//   rect_block_kernel  a cluster of C CTAs or a single CTA.  Each thread folds
//                      its share of the reduced levels, then lanes combine by
//                      xor-shuffle (Sec. 3.7), warps through shared memory in
//                      warp order (Sec. 3.7's fallback one level up), CTAs of
//                      a cluster through distributed shared memory in rank
//                      order; items are handled in rounds of M so that one
//                      barrier serves M outputs.
//   rect_lanes_kernel  a group of L lanes of one warp (warp, sub-warp group of
//                      Sec. 3.8, or a single thread): lanes combine by
//                      xor-shuffle with width L.
// When the first reduced level is bound to the grid, every output is cut into
// G parts that write partials; rect_combine_kernel folds them in 32 interleaved
// chains (accum.cuh; compensated partials as a double-float sum).
// The reduction tree depends only on the plan, never on which SM ran what, so
// runs are bit-reproducible.
#pragma once

#include <cooperative_groups.h>
#include <cstdint>

#include "rect_route.h"
#include "accum.cuh"
#include "hp_internal.h"

namespace hp {

namespace cg = cooperative_groups;

#ifndef HP_FOLD_LOADS
#define HP_FOLD_LOADS 4   // loads a thread issues before folding them (plain-load kernels)
#endif

// ---------------------------------------------------------------- loads
__device__ __forceinline__ float4 ld_stream4(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ int4 ld_stream4(const int32_t* p) { return __ldcs(reinterpret_cast<const int4*>(p)); }
__device__ __forceinline__ float4 ld_keep4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ int4 ld_keep4(const int32_t* p) { return __ldg(reinterpret_cast<const int4*>(p)); }
__device__ __forceinline__ float ld_stream(const float* p) { return __ldcs(p); }
__device__ __forceinline__ int32_t ld_stream(const int32_t* p) { return __ldcs(p); }
__device__ __forceinline__ float ld_keep(const float* p) { return __ldg(p); }
__device__ __forceinline__ int32_t ld_keep(const int32_t* p) { return __ldg(p); }

template <class V4>
__device__ __forceinline__ auto v4get(const V4& v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

// ---------------------------------------------------------------- bodies
// fold V consecutive iterations starting at flat (reduced index rflat)
// Memory bodies split a step into load (V consecutive iterations at flat, the
// broadcast operand at rflat) and apply (fold them into the V slots), so that
// fold_item can issue several loads before the first fold.
template <class Op, int V>
struct Vals {
  typename Op::In a[V];
  typename Op::In b[V];
};

template <class Op>
struct BodyLoad {
  static constexpr bool kPipeable = true;
  static constexpr bool kDot = false;
  const typename Op::In* A;
  __host__ __device__ const typename Op::In* wptr() const { return nullptr; }
  template <int V>
  __device__ __forceinline__ Vals<Op, V> load(int64_t flat, int64_t) const {
    Vals<Op, V> v;
    if constexpr (V == 4) {
      const auto q = ld_stream4(A + flat);
      v.a[0] = q.x;
      v.a[1] = q.y;
      v.a[2] = q.z;
      v.a[3] = q.w;
    } else {
#pragma unroll
      for (int i = 0; i < V; ++i) v.a[i] = ld_stream(A + flat + i);
    }
    return v;
  }
  template <int V>
  __device__ __forceinline__ void apply(typename Op::Acc (&acc)[V], const Vals<Op, V>& v) const {
    fold_vals_load<Op, V>(acc, v.a);
  }
  template <int V>
  __device__ __forceinline__ void fold(typename Op::Acc (&acc)[V], int64_t flat, int64_t rflat) const {
    apply<V>(acc, load<V>(flat, rflat));
  }
};

template <class Op>
struct BodyDot {
  static constexpr bool kPipeable = true;
  static constexpr bool kDot = true;
  const typename Op::In* A;
  const typename Op::In* w;
  __host__ __device__ const typename Op::In* wptr() const { return w; }
  template <int V>
  __device__ __forceinline__ Vals<Op, V> load(int64_t flat, int64_t rflat) const {
    Vals<Op, V> v;
    if constexpr (V == 4) {
      const auto q = ld_stream4(A + flat);
      const auto r = ld_keep4(w + rflat);
      v.a[0] = q.x;
      v.a[1] = q.y;
      v.a[2] = q.z;
      v.a[3] = q.w;
      v.b[0] = r.x;
      v.b[1] = r.y;
      v.b[2] = r.z;
      v.b[3] = r.w;
    } else {
#pragma unroll
      for (int i = 0; i < V; ++i) {
        v.a[i] = ld_stream(A + flat + i);
        v.b[i] = ld_keep(w + rflat + i);
      }
    }
    return v;
  }
  template <int V>
  __device__ __forceinline__ void apply(typename Op::Acc (&acc)[V], const Vals<Op, V>& v) const {
    fold_vals_dot<Op, V>(acc, v.a, v.b);
  }
  template <int V>
  __device__ __forceinline__ void fold(typename Op::Acc (&acc)[V], int64_t flat, int64_t rflat) const {
    apply<V>(acc, load<V>(flat, rflat));
  }
};

// a + b * (flat mod m): exact in int64, wrapped for int32, rounded once for FP
template <class Op>
struct BodyAffine {
  static constexpr bool kPipeable = false;
  static constexpr bool kDot = false;
  const typename Op::In* A = nullptr;
  __host__ __device__ const typename Op::In* wptr() const { return nullptr; }
  int64_t a, b, m;
  template <int V>
  __device__ __forceinline__ void fold(typename Op::Acc (&acc)[V], int64_t flat, int64_t) const {
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int64_t v = a + b * ((flat + i) % m);
      if constexpr (Op::kFp) {
        Op::add_val(acc[i], static_cast<float>(v));
      } else if constexpr (sizeof(typename Op::Out) == 4) {
        Op::add_val(acc[i], static_cast<int32_t>(static_cast<uint32_t>(static_cast<uint64_t>(v))));
      } else {
        Op::add_val(acc[i], static_cast<long long>(v));
      }
    }
  }
};

// fl32(q^(flat mod m)) from a table the planner filled
template <class Op>
struct BodyGeo {
  static constexpr bool kPipeable = false;
  static constexpr bool kDot = false;
  const typename Op::In* A = nullptr;
  __host__ __device__ const typename Op::In* wptr() const { return nullptr; }
  const float* table;
  int64_t m;
  template <int V>
  __device__ __forceinline__ void fold(typename Op::Acc (&acc)[V], int64_t flat, int64_t) const {
#pragma unroll
    for (int i = 0; i < V; ++i) Op::add_val(acc[i], __ldg(table + (flat + i) % m));
  }
};

// ---------------------------------------------------------------- per-thread fold of one item
template <class Op, int V, class Body>
__device__ __forceinline__ void fold_item(const RectPlan& p, const Body& body, int64_t o, int64_t g,
                                          const int32_t (&slot)[kMaxV], typename Op::Acc (&acc)[V]) {
  const int nv = p.nv;
  int64_t lo[kMaxV], hi[kMaxV], x[kMaxV];
#pragma unroll
  for (int v = 0; v < kMaxV; ++v) {
    if (v < nv) {
      lo[v] = 0;
      hi[v] = p.vn[v];
    }
  }
  if (p.split) {
    lo[0] = g * p.tile;
    hi[0] = (lo[0] + p.tile < p.vn[0]) ? lo[0] + p.tile : p.vn[0];
  }
  for (int v = 0; v < nv - 1; ++v) {
    x[v] = lo[v] + slot[v];
    if (x[v] >= hi[v]) return;
  }
  const int64_t obase = o * p.R;
  const int last = nv - 1;
  const int64_t in_lo = lo[last] + slot[last], in_hi = hi[last], P = p.vP[last];
  while (true) {
    int64_t roff = 0;
    for (int v = 0; v < last; ++v) roff += x[v] * p.vstride[v];
    const int64_t base = obase + roff;
    if constexpr (Body::kPipeable) {
      // HP_FOLD_LOADS loads in flight before the first of their folds (same fold order)
      constexpr int NL = HP_FOLD_LOADS;
      int64_t xi = in_lo;
      for (; xi + (NL - 1) * P < in_hi; xi += NL * P) {
        decltype(body.template load<V>(base, roff)) v[NL];
#pragma unroll
        for (int q = 0; q < NL; ++q) v[q] = body.template load<V>(base + xi + q * P, roff + xi + q * P);
#pragma unroll
        for (int q = 0; q < NL; ++q) body.template apply<V>(acc, v[q]);
      }
      for (; xi < in_hi; xi += P) body.template fold<V>(acc, base + xi, roff + xi);
    } else {
      for (int64_t xi = in_lo; xi < in_hi; xi += P) body.template fold<V>(acc, base + xi, roff + xi);
    }
    int v = last - 1;
    for (; v >= 0; --v) {
      x[v] += p.vP[v];
      if (x[v] < hi[v]) break;
      x[v] = lo[v] + slot[v];
    }
    if (v < 0) break;
  }
}

template <class Op, int V>
__device__ __forceinline__ typename Op::Acc fold_vec(const typename Op::Acc (&acc)[V]) {
  if constexpr (V == 4) return Op::combine(Op::combine(acc[0], acc[1]), Op::combine(acc[2], acc[3]));
  else if constexpr (V == 2) return Op::combine(acc[0], acc[1]);
  else return acc[0];
}

template <class Op>
__device__ __forceinline__ typename Op::Acc lanes_allreduce(typename Op::Acc a, int width) {
  for (int m = width >> 1; m >= 1; m >>= 1) a = Op::combine(a, Op::shfl_xor(a, m, width));
  return a;
}

template <class Op>
__device__ __forceinline__ void emit(const RectPlan& p, int64_t item, typename Op::Acc a, typename Op::Out* out,
                                     typename Op::Acc* part) {
  if (p.G == 1) {
    out[item] = Op::finish(a);
    if constexpr (std::is_same_v<typename Op::Acc, f2>) {
      if (p.comp) p.comp[item] = Op::residual(a);
    }
  } else {
    part[item] = a;
  }
}

// ---------------------------------------------------------------- team = cluster or CTA
template <class Op, int V, class Body>
__global__ void __launch_bounds__(1024) rect_block_kernel(RectPlan p, Body body, typename Op::Out* out,
                                                          typename Op::Acc* part) {
  using Acc = typename Op::Acc;
  __shared__ Acc wpart[2][kMaxM][kMaxWarps];
  __shared__ Acc cpart[2][kMaxM];
  const int C = p.C;
  int rank = 0;
  int64_t team = blockIdx.x, n_teams = gridDim.x;
  if (C > 1) {
    rank = static_cast<int>(cg::this_cluster().block_rank());
    team = blockIdx.x / C;
    n_teams = gridDim.x / C;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane / p.grp_lanes, lig = lane % p.grp_lanes;
  int32_t slot[kMaxV];
#pragma unroll
  for (int v = 0; v < kMaxV; ++v)
    slot[v] = rank * p.cr[v] + warp * p.cw[v] + grp * p.cg[v] + lig * p.cl[v];
  const int M = p.M, W = p.W;
  const int64_t n_chunks = (p.items + M - 1) / M;
  int buf = 0;
  for (int64_t chunk = team; chunk < n_chunks; chunk += n_teams) {
    const int64_t item0 = chunk * M;
    const int mcount = static_cast<int>((p.items - item0 < M) ? p.items - item0 : M);
    for (int m = 0; m < mcount; ++m) {
      const int64_t item = item0 + m;
      const int64_t o = item / p.G, g = item - o * p.G;
      Acc acc[V];
#pragma unroll
      for (int i = 0; i < V; ++i) acc[i] = Op::ident();
      fold_item<Op, V>(p, body, o, g, slot, acc);
      Acc a = lanes_allreduce<Op>(fold_vec<Op, V>(acc), 32);
      if (lane == 0) wpart[buf][m][warp] = a;
    }
    __syncthreads();
    if (threadIdx.x < mcount) {
      Acc a = wpart[buf][threadIdx.x][0];
      for (int w = 1; w < W; ++w) a = Op::combine(a, wpart[buf][threadIdx.x][w]);
      cpart[buf][threadIdx.x] = a;
    }
    if (C > 1) {
      cg::cluster_group cl = cg::this_cluster();
      cl.sync();  // release own CTA partials, acquire the peers'
      for (int m = rank + C * static_cast<int>(threadIdx.x); m < mcount; m += C * static_cast<int>(blockDim.x)) {
        Acc a = *cl.map_shared_rank(&cpart[buf][m], 0);
        for (int q = 1; q < C; ++q) a = Op::combine(a, *cl.map_shared_rank(&cpart[buf][m], q));
        emit<Op>(p, item0 + m, a, out, part);
      }
    } else if (threadIdx.x < mcount) {
      emit<Op>(p, item0 + threadIdx.x, cpart[buf][threadIdx.x], out, part);
    }
    buf ^= 1;
  }
  if (C > 1) cg::this_cluster().sync();  // peers may still read this CTA's partials
}

// ---------------------------------------------------------------- team = cluster or CTA, pipelined
// Same plan, same fold order and reduction tree as rect_block_kernel (results
// are bit-identical), but every thread streams its own 128-bit element groups
// through a private ring of D item stages in shared memory filled by cp.async,
// so D items' loads per thread stay in flight across item boundaries and
// across the CTA / cluster barriers of the rounds.  A thread only ever reads
// the slots it filled itself, so the ring needs no barrier: cp.async.wait_group
// orders each read after its own copies, and a stage is refilled only after
// the values read from it have been consumed by the folds.
constexpr int kPatMax = 8;    // element groups per thread per item
constexpr int kPipeMaxThreads = 256;
#ifndef HP_PIPE_MIN_BLOCKS
#define HP_PIPE_MIN_BLOCKS 2   // resident CTAs per SM the register budget is sized for
#endif

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ float4 neg4(float4 v) { return make_float4(-v.x, -v.y, -v.z, -v.w); }
__device__ __forceinline__ int4 neg4(int4 v) { return make_int4(-v.x, -v.y, -v.z, -v.w); }

template <class In> struct Vec4Of;
template <> struct Vec4Of<float> { using T = float4; };
template <> struct Vec4Of<int32_t> { using T = int4; };

template <class Op, class V4>
__device__ __forceinline__ void fold4_load(typename Op::Acc (&acc)[4], const V4& a) {
  Op::add_val(acc[0], a.x);
  Op::add_val(acc[1], a.y);
  Op::add_val(acc[2], a.z);
  Op::add_val(acc[3], a.w);
}
template <class Op, class V4>
__device__ __forceinline__ void fold4_dot(typename Op::Acc (&acc)[4], const V4& a, const V4& b) {
  Op::add_prod(acc[0], a.x, b.x);
  Op::add_prod(acc[1], a.y, b.y);
  Op::add_prod(acc[2], a.z, b.z);
  Op::add_prod(acc[3], a.w, b.w);
}

// the element groups (offsets within one output's reduced space) one thread
// folds for any item, in fold_item's order; returns their number
__device__ __forceinline__ int build_pattern(const RectPlan& p, const int32_t (&slot)[kMaxV], int32_t* pat,
                                             int stride) {
  const int nv = p.nv;
  int64_t x[kMaxV];
  int n = 0;
  for (int v = 0; v < nv - 1; ++v) {
    x[v] = slot[v];
    if (x[v] >= p.vn[v]) return 0;
  }
  const int last = nv - 1;
  while (true) {
    int64_t roff = 0;
    for (int v = 0; v < last; ++v) roff += x[v] * p.vstride[v];
    for (int64_t xi = slot[last]; xi < p.vn[last]; xi += p.vP[last]) {
      if (n < kPatMax) pat[n * stride] = static_cast<int32_t>(roff + xi);
      ++n;
    }
    int v = last - 1;
    for (; v >= 0; --v) {
      x[v] += p.vP[v];
      if (x[v] < p.vn[v]) break;
      x[v] = slot[v];
    }
    if (v < 0) break;
  }
  return n < kPatMax ? n : kPatMax;  // the planner only picks this kernel when n <= kPatMax
}

// D items in flight per thread: each stage holds one item's element groups
// (at most kPatMax 16-byte groups per thread), committed as one cp.async group.
template <class Op, bool DOT, int D>
__global__ void __launch_bounds__(kPipeMaxThreads, HP_PIPE_MIN_BLOCKS) rect_block_pipe_kernel(RectPlan p, const typename Op::In* __restrict__ A,
                                                               const typename Op::In* __restrict__ w,
                                                               typename Op::Out* out, typename Op::Acc* part) {
  using Acc = typename Op::Acc;
  using In = typename Op::In;
  using V4 = typename Vec4Of<In>::T;
  extern __shared__ __align__(16) unsigned char pipe_smem[];
  const int nthr = blockDim.x, tid = threadIdx.x;
  const int G = p.groups;                                            // stage width (groups per item)
  V4* ring = reinterpret_cast<V4*>(pipe_smem);                      // [D][G][nthr]
  int32_t* pat = reinterpret_cast<int32_t*>(pipe_smem);             // [kPatMax][nthr], before the ring is used
  __shared__ Acc wpart[2][kMaxM][kPipeMaxThreads / 32];
  __shared__ Acc cpart[2][kMaxM];
  const int C = p.C;
  int rank = 0;
  int64_t team = blockIdx.x, n_teams = gridDim.x;
  if (C > 1) {
    rank = static_cast<int>(cg::this_cluster().block_rank());
    team = blockIdx.x / C;
    n_teams = gridDim.x / C;
  }
  const int warp = tid >> 5, lane = tid & 31;
  const int grp = lane / p.grp_lanes, lig = lane % p.grp_lanes;
  int32_t slot[kMaxV];
#pragma unroll
  for (int v = 0; v < kMaxV; ++v) slot[v] = rank * p.cr[v] + warp * p.cw[v] + grp * p.cg[v] + lig * p.cl[v];
  const int nt = build_pattern(p, slot, pat + tid, nthr);
  int32_t po[kPatMax];
  V4 wv[kPatMax];
#pragma unroll
  for (int k = 0; k < kPatMax; ++k) {
    po[k] = (k < nt) ? pat[k * nthr + tid] : 0;
    if constexpr (DOT) {
      if (k < nt) wv[k] = ld_keep4(w + po[k]);
    }
  }
  __syncthreads();  // every pattern is in registers before the ring (same memory) fills
  const int M = p.M, W = p.W;
  const int64_t R = p.R, items = p.items;
  const int64_t n_chunks = (items + M - 1) / M;
  V4* const ring_t = ring + tid;
  const int stage_stride = G * nthr;

  // producer cursor over this team's items: item pm of chunk pc
  int64_t pc = team;
  int pm = 0;
  int pcount = (pc < n_chunks) ? static_cast<int>((items - pc * M < M) ? items - pc * M : M) : 0;
  bool pvalid = nt > 0 && pc < n_chunks;
  const In* pitem = pvalid ? A + pc * M * R : A;
  auto issue = [&](int stage) {
    if (pvalid) {
      V4* dst = ring_t + stage * stage_stride;
#pragma unroll
      for (int k = 0; k < kPatMax; ++k)
        if (k < nt) cp_async16(dst + k * nthr, pitem + po[k]);
      pitem += R;
      if (++pm == pcount) {
        pm = 0;
        pc += n_teams;
        pvalid = pc < n_chunks;
        pcount = pvalid ? static_cast<int>((items - pc * M < M) ? items - pc * M : M) : 0;
        if (pvalid) pitem = A + pc * M * R;
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < D; ++s) issue(s);

  int rstage = 0;
  int buf = 0;
  for (int64_t chunk = team; chunk < n_chunks; chunk += n_teams) {
    const int64_t item0 = chunk * M;
    const int mcount = static_cast<int>((items - item0 < M) ? items - item0 : M);
    for (int m = 0; m < mcount; ++m) {
      Fold4<Op> f;
      f.init();
      if (nt > 0) {
        cp_async_wait<D - 1>();
        const V4* src = ring_t + rstage * stage_stride;
#pragma unroll
        for (int k = 0; k < kPatMax; ++k) {
          if (k < nt) {
            const V4 a = src[k * nthr];
            if constexpr (DOT) f.dot(a, wv[k], wv[k]);
            else f.load(a);
          }
        }
        issue(rstage);   // the folds above consumed the stage
        rstage = (rstage + 1 == D) ? 0 : rstage + 1;
      }
      Acc acc[4];
      f.get(acc);
      Acc a = lanes_allreduce<Op>(fold_vec<Op, 4>(acc), 32);
      if (lane == 0) wpart[buf][m][warp] = a;
    }
    __syncthreads();
    if (tid < mcount) {
      Acc a = wpart[buf][tid][0];
      for (int q = 1; q < W; ++q) a = Op::combine(a, wpart[buf][tid][q]);
      cpart[buf][tid] = a;
    }
    if (C > 1) {
      cg::cluster_group cl = cg::this_cluster();
      cl.sync();
      for (int m = rank + C * tid; m < mcount; m += C * nthr) {
        Acc a = *cl.map_shared_rank(&cpart[buf][m], 0);
        for (int q = 1; q < C; ++q) a = Op::combine(a, *cl.map_shared_rank(&cpart[buf][m], q));
        emit<Op>(p, item0 + m, a, out, part);
      }
    } else if (tid < mcount) {
      emit<Op>(p, item0 + tid, cpart[buf][tid], out, part);
    }
    buf ^= 1;
  }
  cp_async_wait<0>();
  if (C > 1) cg::this_cluster().sync();
}

// items in flight for a plan with G groups per item
__host__ __device__ constexpr int pipe_depth(int groups) { return groups > 4 ? 2 : 4; }
// largest dynamic shared memory of any pipelined plan: stages of 16-byte groups
// for kPipeMaxThreads threads (D * G <= 16), or the pattern table
constexpr size_t kPipeDynMax = static_cast<size_t>(kPipeMaxThreads) * 16 * 16;

// ---------------------------------------------------------------- team = L lanes of a warp
template <class Op, int V, class Body>
__global__ void __launch_bounds__(1024) rect_lanes_kernel(RectPlan p, Body body, typename Op::Out* out,
                                                          typename Op::Acc* part) {
  using Acc = typename Op::Acc;
  const int L = p.L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lt = lane % L;
  const int grp = lt / p.grp_lanes, lig = lt % p.grp_lanes;
  int32_t slot[kMaxV];
#pragma unroll
  for (int v = 0; v < kMaxV; ++v) slot[v] = grp * p.cg[v] + lig * p.cl[v];
  const int teams_per_warp = 32 / L;
  const int64_t warp_global = static_cast<int64_t>(blockIdx.x) * p.W + warp;
  const int64_t n_teams = static_cast<int64_t>(gridDim.x) * p.W * teams_per_warp;
  for (int64_t base = warp_global * teams_per_warp; base < p.items; base += n_teams) {
    const int64_t item = base + lane / L;
    const bool valid = item < p.items;
    Acc acc[V];
#pragma unroll
    for (int i = 0; i < V; ++i) acc[i] = Op::ident();
    if (valid) {
      const int64_t o = item / p.G, g = item - o * p.G;
      fold_item<Op, V>(p, body, o, g, slot, acc);
    }
    Acc a = lanes_allreduce<Op>(fold_vec<Op, V>(acc), L);
    if (valid && lt == 0) emit<Op>(p, item, a, out, part);
  }
}

// ---------------------------------------------------------------- team = L lanes, whole rows
// The plans that rect_lanes_kernel runs most, without its generality: one
// reduced virtual level of stride 1 and no grid parts, so an output is a row of
// R consecutive elements.  A team folds one row (U = 1) with 4 positions loaded
// ahead; a thread that is a team of its own folds U = 4 rows of at most 4 elements,
// FP32 sums of one slot two rows per packed FP32x2 instruction.  Each row sees the
// fold order and the reduction tree of rect_lanes_kernel, so the bits are the
// same.  Bound by HBM for plain sums (2^26 elements: rows of 64 and 1024, 51 and 47 us
// in the general kernel, 41 here, 6.7 TB/s), by the compensated arithmetic's issue
// rate otherwise (dot products of odd rows of 1021: 136 us, 72 here).
struct RowsArgs {
  int64_t O;
  int32_t R, P, L;             // elements per row, slots (elements per step), lanes per team
  int32_t grp_lanes, cg, cl;   // slot of lane lt: (lt / grp_lanes) * cg + (lt % grp_lanes) * cl
  // One row at a time: teams past the last row fold it once more and store nothing, so
  // that a last warp that is not full keeps its loads in flight (500 rows of 101 f32:
  // 5.9 us a position at a time, 3.2 us in rect_lanes_kernel).  An argument, not a
  // constant: where the compiler knew the single positions' loop to be unreachable,
  // the others' schedule took 3 to 9% longer (300,000 rows of 500 f32: 90 us, 98 so).
  // Compensated dot products have no registers for it (146 us, 164 so).
  int32_t again;
};
constexpr int kRowsThreads = 256;

// the U rows' values at one position, folded into their accumulators
template <class Op, int V, bool DOT, int U>
__device__ __forceinline__ void fold_rows(typename Op::Acc (&acc)[U][V], const Vals<Op, V> (&v)[U],
                                          const typename Op::In (&b)[V]) {
  if constexpr (V == 1 && U % 2 == 0 && std::is_same<Op, OpF32Comp>::value) {
#pragma unroll
    for (int u = 0; u < U; u += 2) {
      float2 sp = make_float2(acc[u][0].s, acc[u + 1][0].s), cp = make_float2(acc[u][0].c, acc[u + 1][0].c);
      const float2 x = make_float2(v[u].a[0], v[u + 1].a[0]);
      if constexpr (DOT) comp_prod_pair(sp, cp, x, make_float2(b[0], b[0]));
      else comp_add_pair(sp, cp, x);
      acc[u][0] = {sp.x, cp.x};
      acc[u + 1][0] = {sp.y, cp.y};
    }
  } else if constexpr (V == 1 && U % 2 == 0 && std::is_same<Op, OpF32Sum>::value) {
#pragma unroll
    for (int u = 0; u < U; u += 2) {
      float2 sp = make_float2(acc[u][0], acc[u + 1][0]);
      const float2 x = make_float2(v[u].a[0], v[u + 1].a[0]);
      if constexpr (DOT) sp = fma2(x, make_float2(b[0], b[0]), sp);
      else sp = add2(sp, x);
      acc[u][0] = sp.x;
      acc[u + 1][0] = sp.y;
    }
  } else {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if constexpr (DOT) fold_vals_dot<Op, V>(acc[u], v[u].a, b);
      else fold_vals_load<Op, V>(acc[u], v[u].a);
    }
  }
}
template <class In, int V>
__device__ __forceinline__ void load_row(const In* p, In (&a)[V]) {
  if constexpr (V == 4) {
    const auto q = ld_stream4(p);
    a[0] = q.x;
    a[1] = q.y;
    a[2] = q.z;
    a[3] = q.w;
  } else {
    a[0] = ld_stream(p);
  }
}
template <class In, int V>
__device__ __forceinline__ void load_bcast(const In* p, In (&b)[V]) {
  if constexpr (V == 4) {
    const auto q = ld_keep4(p);
    b[0] = q.x;
    b[1] = q.y;
    b[2] = q.z;
    b[3] = q.w;
  } else {
    b[0] = ld_keep(p);
  }
}
// A team folds one row at a time with 4 positions loaded ahead: the registers
// that more rows take cost more resident warps than their loads are worth.  A
// thread per row of at most 4 elements has no further positions: 4 rows.
constexpr int kRowsU = 4;

// CTAs per SM the registers are sized for (swept over 5, 6 and 8, and uncapped):
// 2^26 elements in rows of 100 / 511, f32: 6 and 8 CTAs 43 and 48 us, uncapped 45
// and 55; compensated dot: 57 and 70 us, uncapped 77 and 73
template <class Op, int V, bool DOT, int U>
constexpr int rows_blocks() {
  if (U > 1) return 1;
  if (V == 1) return 8;
  return !DOT && sizeof(typename Op::Acc) == 8 ? 5 : 6;
}

template <class Op, int V, bool DOT, int U>
__global__ void __launch_bounds__(kRowsThreads, (rows_blocks<Op, V, DOT, U>()))
    rect_rows_kernel(const RowsArgs g, const typename Op::In* __restrict__ A, const typename Op::In* __restrict__ w,
                     typename Op::Out* out, float* comp) {
  using Acc = typename Op::Acc;
  using In = typename Op::In;
  constexpr int NX = U == 1 ? 4 : 2;            // positions loaded before the first fold
  constexpr bool kAgain = U == 1 && !(DOT && std::is_same_v<Acc, f2>);
  const int L = U > 1 ? 1 : g.L, R = g.R, P = g.P;
  const int lane = threadIdx.x & 31, lt = lane & (L - 1), set = 32 / L;
  const int s0 = (lt / g.grp_lanes) * g.cg + (lt % g.grp_lanes) * g.cl;
  const int64_t per = static_cast<int64_t>(set) * U;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5) * per;
  for (int64_t base = (static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5)) * per; base < g.O;
       base += stride) {
    const int64_t row = base + lane / L;
    const bool full = base + per <= g.O;        // the same in every lane
    int64_t from = row;
    if constexpr (kAgain) {
      if (!full && g.again && row >= g.O) from = g.O - 1;
    }
    const In* a = A + from * R;
    const int dist = set * R;                   // elements between a team's rows
    Acc acc[U][V];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int i = 0; i < V; ++i) acc[u][i] = Op::ident();
    const bool whole = full || (kAgain && g.again);
    int rows = U;                               // this lane's rows
    if (!whole) {
      rows = 0;
#pragma unroll
      for (int u = 0; u < U; ++u) rows += row + static_cast<int64_t>(u) * set < g.O ? 1 : 0;
    }
    int x = s0;
    if (whole) {
      for (; x + (NX - 1) * P < R; x += NX * P) {
        Vals<Op, V> v[NX][U];
        In b[NX][V];
#pragma unroll
        for (int q = 0; q < NX; ++q) {
          if constexpr (DOT) load_bcast<In, V>(w + x + q * P, b[q]);
#pragma unroll
          for (int u = 0; u < U; ++u) load_row<In, V>(a + u * dist + x + q * P, v[q][u].a);
        }
#pragma unroll
        for (int q = 0; q < NX; ++q) fold_rows<Op, V, DOT, U>(acc, v[q], b[q]);
      }
      // the last NX - 1 positions or fewer, again all in flight (2^26 elements in rows of
      // 900, f32 and int64: 45 and 50 us one after the other, 42 and 41 so); the
      // compensated folds and dot products lose more to its registers (compensated
      // 511: 52 us, 72 so; f32 dot of 1200 x 3001: 10 us, 17 so)
      if constexpr (U == 1 && !DOT && !std::is_same_v<Acc, f2>) {
        if (x < R) {
          Vals<Op, V> v[NX - 1][1];
#pragma unroll
          for (int q = 0; q < NX - 1; ++q) load_row<In, V>(a + (x + q * P < R ? x + q * P : x), v[q][0].a);
#pragma unroll
          for (int q = 0; q < NX - 1; ++q)
            if (x + q * P < R) fold_vals_load<Op, V>(acc[0], v[q][0].a);
          x = R;
        }
      }
    }
    for (; x < R; x += P) {
      Vals<Op, V> v[U];
      In b[V];
      if constexpr (DOT) load_bcast<In, V>(w + x, b);
      // rows past the last are folded from the first row's values; their results are not stored
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (rows > 0) load_row<In, V>(a + (u < rows ? u * dist : 0) + x, v[u].a);
      if (rows > 0) fold_rows<Op, V, DOT, U>(acc, v, b);
    }
    Acc part[U];
#pragma unroll
    for (int u = 0; u < U; ++u) part[u] = fold_vec<Op, V>(acc[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const Acc r = lanes_allreduce<Op>(part[u], L);
      const int64_t o = row + static_cast<int64_t>(u) * set;
      if (lt == 0 && o < g.O) {
        out[o] = Op::finish(r);
        if constexpr (std::is_same_v<Acc, f2>) {
          if (comp) comp[o] = Op::residual(r);
        }
      }
    }
  }
}

// ---------------------------------------------------------------- team = a CTA, contiguous items
// The plans of rect_block_kernel with one reduced virtual level of stride 1 and
// a CTA of at most 8 warps: an item (an output, or one grid part of it) is a run
// of consecutive elements.  The per-thread order and the tree are
// rect_block_kernel's; what differs is what limits the rate: 32-bit offsets, no
// general level loop and 256 threads a CTA leave 32 to 48 registers a thread, so
// 4 to 8 CTAs per SM keep 4 or 8 loads per thread in flight.  2^26 elements in
// rows of 16384, 262144 and one row, f32: 45, 61 and 54 us in the general kernel,
// 39, 44 and 47 here (6.9 TB/s; the single row adds its combine's launch); odd
// rows of 8195: 73 and 41; compensated dot of 16384: 69 and 43.
struct FlatArgs {
  int64_t items, R, tile;      // tile: elements per grid part (G > 1)
  int32_t G, P, W;
  int32_t grp_lanes, cw, cg, cl;
};
// CTAs per SM (swept): the dot product's second operand takes the registers of
// one more load per position (600 x 2^18 compensated: 4 CTAs 101 us, 5 107, 6
// 125); scalar loads need the most threads (20011 x 8195 int64: 8 CTAs 98 us, 6
// 100, 5 106), compensated 128-bit loads run at HBM's rate with 5
template <class Op, int V, bool DOT>
constexpr int flat_blocks() { return DOT ? 4 : V == 4 && sizeof(typename Op::Acc) == 8 ? 5 : 8; }

template <class Op, int V, bool DOT>
__global__ void __launch_bounds__(kFlatThreads, (flat_blocks<Op, V, DOT>()))
    rect_flat_kernel(const FlatArgs g, const typename Op::In* __restrict__ A, const typename Op::In* __restrict__ w,
                     typename Op::Out* out, typename Op::Acc* part, float* comp) {
  using Acc = typename Op::Acc;
  using In = typename Op::In;
  constexpr int NL = V == 4 ? 4 : 8;           // loads in flight before the first fold
  __shared__ Acc wpart[2][kFlatThreads / 32];
  if (g.G > 1) grid_launch_dependents();       // the combine kernel: 2^20 elements 10.2 us with it after, 8.9 so
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s0 = warp * g.cw + (lane / g.grp_lanes) * g.cg + (lane % g.grp_lanes) * g.cl;
  const int P = g.P;
  int buf = 0;
  for (int64_t item = blockIdx.x; item < g.items; item += gridDim.x, buf ^= 1) {
    int64_t o = item, lo = 0, n64 = g.R;
    if (g.G > 1) {
      o = item / g.G;
      lo = (item - o * g.G) * g.tile;
      n64 = g.R - lo < g.tile ? g.R - lo : g.tile;
    }
    const int n = static_cast<int>(n64);
    const In* a = A + o * g.R + lo;
    const In* wp = DOT ? w + lo : nullptr;
    Acc acc[1][V];
#pragma unroll
    for (int i = 0; i < V; ++i) acc[0][i] = Op::ident();
    int x = s0;
    for (; x < n - (NL - 1) * P; x += NL * P) {
      Vals<Op, V> v[NL][1];
      In b[NL][V];
#pragma unroll
      for (int q = 0; q < NL; ++q) {
        load_row<In, V>(a + x + q * P, v[q][0].a);
        if constexpr (DOT) load_bcast<In, V>(wp + x + q * P, b[q]);
      }
#pragma unroll
      for (int q = 0; q < NL; ++q) fold_rows<Op, V, DOT, 1>(acc, v[q], b[q]);
    }
    // the last NL - 1 positions or fewer, again all in flight (2^26 elements in rows of
    // 10001: f32 50 us one after the other, 40 so; compensated dot 81 and 64)
    if (x < n) {
      Vals<Op, V> v[NL - 1][1];
      In b[NL - 1][V];
#pragma unroll
      for (int q = 0; q < NL - 1; ++q) {
        const int y = x + q * P < n ? x + q * P : x;
        load_row<In, V>(a + y, v[q][0].a);
        if constexpr (DOT) load_bcast<In, V>(wp + y, b[q]);
      }
#pragma unroll
      for (int q = 0; q < NL - 1; ++q)
        if (x + q * P < n) fold_rows<Op, V, DOT, 1>(acc, v[q], b[q]);
    }
    const Acc r = lanes_allreduce<Op>(fold_vec<Op, V>(acc[0]), 32);
    if (lane == 0) wpart[buf][warp] = r;
    __syncthreads();
    if (threadIdx.x == 0) {
      Acc t = wpart[buf][0];
      for (int q = 1; q < g.W; ++q) t = Op::combine(t, wpart[buf][q]);
      if (g.G > 1) {
        part[item] = t;
      } else {
        out[o] = Op::finish(t);
        if constexpr (std::is_same_v<Acc, f2>) {
          if (comp) comp[o] = Op::residual(t);
        }
      }
    }
  }
}

// Teams of one lane (rows of 5 to 32 elements) or two (odd rows of up to 64): the
// rows of a warp's teams are one contiguous block, so the warp copies it to
// shared memory with 16-byte cp.async (its stage ring keeps the next two blocks
// in flight) and the teams fold their rows from there.  Read straight from global
// memory, such a row takes a sector per team and load: 2^26 elements in rows of
// 31, f32, 135 us so, 46 here.  Short rows come several sets to a block (MANY), so
// that the waits and the ring's bookkeeping are shared: 2^25 elements in rows of 5,
// f32 and compensated dot 50 and 62 us with one set, 37 and 52 with up to 736
// elements, 41 and 54 with 512, 44 and 58 with 1024.  A kernel of its own, since
// the loop over sets costs longer rows a tenth.  Rows of 4 as whole vectors come
// here for dot products on two-word accumulators only, whose four rows a thread
// take too many registers in rect_rows_kernel (compensated 64 us there, 48 here;
// f32 29 and 33).
constexpr int kThreadRowsStages = 3;
constexpr int kThreadRowsElems = 736;
// sets of rows in a block: at least 16 warps' blocks for every SM
inline int thread_rows_sets(int64_t O, int64_t R, int L, int sms) {
  const int64_t set = 32 / L;
  return static_cast<int>(std::max<int64_t>(1, std::min(kThreadRowsElems / (set * R), O / (set * 16 * std::max(sms, 1)))));
}

template <class Op, int V, bool DOT, bool MANY>
__global__ void __launch_bounds__(kRowsThreads) rect_thread_rows_kernel(int64_t O, int R, int L, int K,
                                                                        const typename Op::In* __restrict__ A,
                                                                        const typename Op::In* __restrict__ w,
                                                                        typename Op::Out* out, float* comp) {
  using Acc = typename Op::Acc;
  using In = typename Op::In;
  extern __shared__ __align__(16) unsigned char rows_smem[];
  __shared__ __align__(16) In ws[DOT ? kThreadRowsMax : 4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if constexpr (DOT) {
    if (static_cast<int>(threadIdx.x) < R) ws[threadIdx.x] = w[threadIdx.x];
    __syncthreads();
  }
  const int set = 32 / L;
  const int rows = MANY ? set * K : set;         // rows of a block: K of every team
  const int block = rows * R;                    // its elements; whole 64 R or 128 R bytes, so blocks keep A's alignment
  In* const ring = reinterpret_cast<In*>(rows_smem) + warp * kThreadRowsStages * block;
  const int64_t n_blocks = (O + rows - 1) / rows;
  const int64_t first = static_cast<int64_t>(blockIdx.x) * (kRowsThreads / 32) + warp;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * (kRowsThreads / 32);
  auto issue = [&](int64_t b, int stage) {
    if (b < n_blocks) {
      const int64_t left = (O - b * rows) * R;   // elements of A from the block on
      const In* src = A + b * rows * R;
      for (int i = 4 * lane; i < block; i += 128) {
        const int n = left - i >= 4 ? 4 : left > i ? static_cast<int>(left - i) : 0;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(ring + stage * block + i)),
                     "l"(n > 0 ? src + i : A), "r"(4 * n)
                     : "memory");
      }
    }
    cp_async_commit();
  };
  int64_t next = first;
#pragma unroll
  for (int s = 0; s < kThreadRowsStages - 1; ++s, next += stride) issue(next, s);
  int stage = 0, refill = kThreadRowsStages - 1;
  for (int64_t b = first; b < n_blocks; b += stride, next += stride) {
    cp_async_wait<kThreadRowsStages - 2>();
    __syncwarp();                                // every lane's copies; and every lane has read the stage refilled below
    issue(next, refill);
    const int lt = lane & (L - 1);
    const In* row = ring + stage * block + lane / L * R;
    refill = stage;
    stage = stage + 1 == kThreadRowsStages ? 0 : stage + 1;
    // the same count in every lane
    for (int j = 0; j < (MANY ? K : 1) && (!MANY || b * rows + j * set < O); ++j, row += set * R) {
      Acc acc[1][V];
#pragma unroll
      for (int i = 0; i < V; ++i) acc[0][i] = Op::ident();
#pragma unroll 4
      for (int x = V * lt; x < R; x += V * L) {
        Vals<Op, V> v[1];
        In bb[V];
        if constexpr (V == 4) {
          using V4 = typename Vec4Of<In>::T;
          const V4 q = *reinterpret_cast<const V4*>(row + x);
          v[0].a[0] = q.x;
          v[0].a[1] = q.y;
          v[0].a[2] = q.z;
          v[0].a[3] = q.w;
          if constexpr (DOT) {
            const V4 t = *reinterpret_cast<const V4*>(ws + x);
            bb[0] = t.x;
            bb[1] = t.y;
            bb[2] = t.z;
            bb[3] = t.w;
          }
        } else {
          v[0].a[0] = row[x];
          if constexpr (DOT) bb[0] = ws[x];
        }
        fold_rows<Op, V, DOT, 1>(acc, v, bb);
      }
      const int64_t o = b * rows + j * set + lane / L;
      const Acc t = lanes_allreduce<Op>(fold_vec<Op, V>(acc[0]), L);
      if (lt == 0 && o < O) {
        out[o] = Op::finish(t);
        if constexpr (std::is_same_v<Acc, f2>) {
          if (comp) comp[o] = Op::residual(t);
        }
      }
    }
  }
  cp_async_wait<0>();
}

// ---------------------------------------------------------------- grid parts -> outputs
// A warp per output, a chain of parts per lane (combine_parts_warp).
constexpr int kCombineWarps = 8;
template <class Op>
__global__ void __launch_bounds__(32 * kCombineWarps) rect_combine_kernel(int64_t O, int32_t G,
                                                                        const typename Op::Acc* part,
                                                                        typename Op::Out* out, float* comp) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  grid_wait();   // launched while the parts are still being folded
  for (int64_t o = blockIdx.x * static_cast<int64_t>(kCombineWarps) + warp; o < O;
       o += static_cast<int64_t>(gridDim.x) * kCombineWarps) {
    const typename Op::Out r = combine_parts_warp<Op>(part + o * G, G, lane, comp ? comp + o : nullptr);
    if (lane == 0) out[o] = r;
  }
}

// ---------------------------------------------------------------- no reduction: one output per iteration
template <class Op, class Body>
__global__ void rect_map_kernel(RectPlan p, Body body, typename Op::Out* out) {
  for (int64_t f = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; f < p.O;
       f += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    typename Op::Acc acc[1] = {Op::ident()};
    body.template fold<1>(acc, f, 0);
    out[f] = Op::finish(acc[0]);
    if constexpr (std::is_same_v<typename Op::Acc, f2>) {
      if (p.comp) p.comp[f] = Op::residual(acc[0]);
    }
  }
}

}  // namespace hp
