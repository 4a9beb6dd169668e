// rect_launch.cuh — host-side launch of the rectangular executor for one
// accumulation policy.  Each rect_*.cu translation unit instantiates it for
// its policies so that the kernels compile in parallel.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "hp_internal.h"
#include "rect_kernels.cuh"

namespace hp {

struct RectArgs {
  const void* const* in;   // device inputs
  void* out;               // device outputs
  void* part;              // grid-part partials (G > 1)
  const float* geo;        // GEOMETRIC table (device)
  cudaStream_t stream;
  float* comp = nullptr;   // compensated sums: residual output (hp_nest_run_comp), or null
};

inline hp_status cuda_fail(cudaError_t e, const char* what) {
  return fail(HP_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// launch of a rows kernel; its grid is sized on the nest's first run of that kind
template <class Op, int V, bool DOT>
hp_status launch_rows(const RectPlan& rp, RowsKind kind, LaunchCfg& cfg, const typename Op::In* A,
                      const typename Op::In* w, const RectArgs& a) {
  using Out = typename Op::Out;
  auto k1 = rect_rows_kernel<Op, V, DOT, 1>;
  auto k4 = rect_rows_kernel<Op, V, DOT, kRowsU>;
  const int set = 32 / rp.L, K = kind == ROWS_THREAD ? thread_rows_sets(rp.O, rp.R, rp.L, cfg.sms) : 1;
  auto kt = K > 1 ? rect_thread_rows_kernel<Op, V, DOT, true> : rect_thread_rows_kernel<Op, V, DOT, false>;
  const size_t dyn = kind == ROWS_THREAD ? sizeof(int32_t) * (kRowsThreads / 32) * kThreadRowsStages * set * K * rp.R : 0;
  const int U = rp.L == 1 ? kRowsU : 1;
  int& grid = cfg.rows_grid[kind - 1];
  if (grid == 0) {
    const void* f = kind == ROWS_THREAD ? reinterpret_cast<const void*>(kt)
                    : U == 1            ? reinterpret_cast<const void*>(k1)
                                        : reinterpret_cast<const void*>(k4);
    cudaError_t e = cudaSuccess;
    if (kind == ROWS_THREAD)   // the kernel's largest, whatever this nest needs
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               kRowsThreads / 32 * kThreadRowsStages * 4 * 32 * 32);
    if (e != cudaSuccess) return cuda_fail(e, "dynamic shared memory size");
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, kRowsThreads, dyn);
    if (e != cudaSuccess) return cuda_fail(e, "occupancy query");
    if (per_sm < 1) return fail(HP_EUNSUPPORTED, "kernel does not fit on an SM with this CTA size");
    const int64_t cta_rows = static_cast<int64_t>(kRowsThreads / 32) * set * (kind == ROWS_THREAD ? K : U);
    const int64_t blocks = std::min<int64_t>((rp.O + cta_rows - 1) / cta_rows, static_cast<int64_t>(per_sm) * cfg.sms);
    grid = static_cast<int>(std::max<int64_t>(blocks, 1));
    cfg.ready = true;
  }
  if (rp.O == 0) return HP_OK;
  Out* out = static_cast<Out*>(a.out);
  if (kind == ROWS_THREAD) {
    kt<<<grid, kRowsThreads, dyn, a.stream>>>(rp.O, static_cast<int>(rp.R), rp.L, K, A, w, out, a.comp);
  } else {
    const RowsArgs g{rp.O, static_cast<int32_t>(rp.R), rp.vP[0], rp.L, rp.grp_lanes, rp.cg[0], rp.cl[0], U == 1 ? 1 : 0};
    if (U == 1) k1<<<grid, kRowsThreads, 0, a.stream>>>(g, A, w, out, a.comp);
    else k4<<<grid, kRowsThreads, 0, a.stream>>>(g, A, w, out, a.comp);
  }
  const cudaError_t e = cudaPeekAtLastError();
  return e == cudaSuccess ? HP_OK : cuda_fail(e, "rect_rows_kernel launch");
}

// the second pass over grid parts
template <class Op>
hp_status launch_combine(const RectPlan& rp, int sms, const RectArgs& a) {
  const int64_t cb = (rp.O + kCombineWarps - 1) / kCombineWarps;   // a warp per output
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(cb, 4LL * sms));
  const cudaError_t e = launch_dependent(rect_combine_kernel<Op>, static_cast<int>(grid), 32 * kCombineWarps, 0, a.stream,
                                         rp.O, rp.G, static_cast<const typename Op::Acc*>(a.part),
                                         static_cast<typename Op::Out*>(a.out), a.comp);
  return e == cudaSuccess ? HP_OK : cuda_fail(e, "rect_combine_kernel launch");
}

template <class Op, int V, bool DOT>
hp_status launch_flat(const RectPlan& rp, LaunchCfg& cfg, const typename Op::In* A, const typename Op::In* w,
                      const RectArgs& a) {
  auto k = rect_flat_kernel<Op, V, DOT>;
  if (cfg.grid == 0) {
    cfg.threads = 32 * rp.W;
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, cfg.threads, 0);
    if (e != cudaSuccess) return cuda_fail(e, "occupancy query");
    if (per_sm < 1) return fail(HP_EUNSUPPORTED, "kernel does not fit on an SM with this CTA size");
    // as many CTAs as run in whole rounds of the items
    const int64_t resident = static_cast<int64_t>(per_sm) * cfg.sms;
    const int64_t rounds = std::max<int64_t>(1, (rp.items + resident - 1) / resident);
    cfg.grid = static_cast<int>(std::max<int64_t>(1, rounds > 4 ? resident : (rp.items + rounds - 1) / rounds));
    cfg.ready = true;
  }
  if (rp.items == 0) return HP_OK;
  const FlatArgs g{rp.items, rp.R, rp.tile, rp.G, rp.vP[0], rp.W, rp.grp_lanes, rp.cw[0], rp.cg[0], rp.cl[0]};
  k<<<cfg.grid, cfg.threads, 0, a.stream>>>(g, A, w, static_cast<typename Op::Out*>(a.out),
                                            static_cast<typename Op::Acc*>(a.part), a.comp);
  const cudaError_t e = cudaPeekAtLastError();
  if (e != cudaSuccess) return cuda_fail(e, "rect_flat_kernel launch");
  return rp.G > 1 ? launch_combine<Op>(rp, cfg.sms, a) : HP_OK;
}

template <class Op, int V, class Body>
hp_status launch_team(const NestPlan& np, RectPlan rp, LaunchCfg& cfg, const Body& body, const RectArgs& a) {
  using Out = typename Op::Out;
  using Acc = typename Op::Acc;
  cudaError_t e;
  rp.comp = a.comp;
  if (rp.team == TEAM_MAP) {
    auto k = rect_map_kernel<Op, Body>;
    if (cfg.grid == 0) {
      cfg.threads = 256;
      const int64_t blocks = (rp.O + 255) / 256;
      cfg.grid = static_cast<int>(blocks < 8LL * cfg.sms ? (blocks > 0 ? blocks : 1) : 8LL * cfg.sms);
      cfg.ready = true;
    }
    if (rp.O == 0) return HP_OK;
    k<<<cfg.grid, cfg.threads, 0, a.stream>>>(rp, body, static_cast<Out*>(a.out));
    e = cudaPeekAtLastError();
    return e == cudaSuccess ? HP_OK : cuda_fail(e, "rect_map_kernel launch");
  }
  if constexpr (Body::kPipeable) {
    const RowsKind kind = rows_kind(np, (reinterpret_cast<uintptr_t>(body.A) & 15u) == 0);
    if (kind != ROWS_NONE) return launch_rows<Op, V, Body::kDot>(rp, kind, cfg, body.A, body.wptr(), a);
    if (flat_plan(np)) return launch_flat<Op, V, Body::kDot>(rp, cfg, body.A, body.wptr(), a);
  }
  const bool block = rp.team == TEAM_BLOCK;
  constexpr bool kPipeable = Body::kPipeable && V == 4;
  const bool pipe = kPipeable && block && rp.pipe;
  auto kb = rect_block_kernel<Op, V, Body>;
  auto kl = rect_lanes_kernel<Op, V, Body>;
  const bool deep = rp.groups <= 4;
  auto kp = deep ? rect_block_pipe_kernel<Op, Body::kDot, pipe_depth(4)> : rect_block_pipe_kernel<Op, Body::kDot, pipe_depth(8)>;
  const void* kfn = pipe ? reinterpret_cast<const void*>(kp)
                         : block ? reinterpret_cast<const void*>(kb) : reinterpret_cast<const void*>(kl);
  const size_t dyn =
      pipe ? static_cast<size_t>(32 * rp.W) *
                 std::max<size_t>(pipe_depth(rp.groups) * rp.groups * 16, kPatMax * sizeof(int32_t))
           : 0;
  if (cfg.grid == 0) {
    cfg.threads = 32 * rp.W;
    cfg.cluster = block ? rp.C : 1;
    if (pipe) {
      // the attribute belongs to the kernel, not to this nest: always the
      // largest size any plan of this kernel uses (static + dynamic may
      // exceed the 48 KiB default)
      e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kPipeDynMax));
      if (e != cudaSuccess) return cuda_fail(e, "dynamic shared memory size");
    }
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, cfg.threads, dyn);
    if (e != cudaSuccess) return cuda_fail(e, "occupancy query");
    if (per_sm < 1) return fail(HP_EUNSUPPORTED, "kernel does not fit on an SM with this CTA size");
    int64_t max_teams;
    if (block && rp.C > 1) {
      if (rp.C > 8) {
        e = cudaFuncSetAttribute(kfn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return cuda_fail(e, "non-portable cluster size");
      }
      cudaLaunchConfig_t lc = {};
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = rp.C;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      lc.gridDim = dim3(rp.C * cfg.sms);
      lc.blockDim = dim3(cfg.threads);
      lc.dynamicSmemBytes = dyn;
      lc.attrs = at;
      lc.numAttrs = 1;
      int n_clusters = 0;
      e = cudaOccupancyMaxActiveClusters(&n_clusters, kfn, &lc);
      if (e != cudaSuccess) return cuda_fail(e, "cluster occupancy query");
      if (n_clusters < 1) return fail(HP_EUNSUPPORTED, "a cluster of this size does not fit on the GPU");
      max_teams = n_clusters;
    } else if (block) {
      max_teams = static_cast<int64_t>(per_sm) * cfg.sms;
    } else {
      max_teams = static_cast<int64_t>(per_sm) * cfg.sms * rp.W * (32 / rp.L);
    }
    if (block) {
      int64_t teams = rp.items < max_teams ? rp.items : max_teams;
      if (teams < 1) teams = 1;
      int64_t M = (rp.items + teams - 1) / teams;
      cfg.M = static_cast<int>(M < 1 ? 1 : (M > kMaxM ? kMaxM : M));
      cfg.grid = static_cast<int>(teams * cfg.cluster);
    } else {
      const int64_t teams_per_cta = static_cast<int64_t>(rp.W) * (32 / rp.L);
      int64_t blocks = (rp.items + teams_per_cta - 1) / teams_per_cta;
      const int64_t max_blocks = static_cast<int64_t>(per_sm) * cfg.sms;
      if (blocks > max_blocks) blocks = max_blocks;
      cfg.grid = static_cast<int>(blocks < 1 ? 1 : blocks);
    }
    cfg.ready = true;
  }
  if (rp.items == 0) return HP_OK;
  rp.M = cfg.M;
  Out* out = static_cast<Out*>(a.out);
  Acc* part = static_cast<Acc*>(a.part);
  if (block) {
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    lc.gridDim = dim3(cfg.grid);
    lc.blockDim = dim3(cfg.threads);
    lc.stream = a.stream;
    if (cfg.cluster > 1) {
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cfg.cluster;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      lc.attrs = at;
      lc.numAttrs = 1;
    }
    if constexpr (kPipeable) {
      if (pipe) {
        lc.dynamicSmemBytes = dyn;
        e = cudaLaunchKernelEx(&lc, kp, rp, body.A, body.wptr(), out, part);
        if (e != cudaSuccess) return cuda_fail(e, "rect_block_pipe_kernel launch");
      } else {
        e = cudaLaunchKernelEx(&lc, kb, rp, body, out, part);
        if (e != cudaSuccess) return cuda_fail(e, "rect_block_kernel launch");
      }
    } else {
      e = cudaLaunchKernelEx(&lc, kb, rp, body, out, part);
      if (e != cudaSuccess) return cuda_fail(e, "rect_block_kernel launch");
    }
  } else {
    kl<<<cfg.grid, cfg.threads, 0, a.stream>>>(rp, body, out, part);
    e = cudaPeekAtLastError();
    if (e != cudaSuccess) return cuda_fail(e, "rect_lanes_kernel launch");
  }
  return rp.G > 1 ? launch_combine<Op>(rp, cfg.sms, a) : HP_OK;
}

template <class Op, class Body>
hp_status launch_v(const NestPlan& np, const RectPlan& rp, LaunchCfg& cfg, const Body& body, const RectArgs& a) {
  if (rp.V == 4) return launch_team<Op, 4>(np, rp, cfg, body, a);
  return launch_team<Op, 1>(np, rp, cfg, body, a);
}

// Entry for one accumulation policy: pick the body.
template <class Op>
hp_status launch_rect(const NestPlan& np, LaunchCfg& cfg, const RectArgs& a) {
  const RectPlan& rp = np.rp;
  using In = typename Op::In;
  switch (np.body) {
    case HP_BODY_LOAD: {
      BodyLoad<Op> b{static_cast<const In*>(a.in[0])};
      return launch_v<Op>(np, rp, cfg, b, a);
    }
    case HP_BODY_DOT_BCAST: {
      BodyDot<Op> b{static_cast<const In*>(a.in[0]), static_cast<const In*>(a.in[1])};
      return launch_v<Op>(np, rp, cfg, b, a);
    }
    case HP_BODY_AFFINE: {
      BodyAffine<Op> b;
      b.a = rp.aff_a;
      b.b = rp.aff_b;
      b.m = rp.aff_m;
      return launch_v<Op>(np, rp, cfg, b, a);
    }
    case HP_BODY_GEOMETRIC: {
      if constexpr (Op::kFp && sizeof(typename Op::Out) == 4) {
        BodyGeo<Op> b;
        b.table = a.geo;
        b.m = rp.geo_m;
        return launch_v<Op>(np, rp, cfg, b, a);
      }
      return fail(HP_EUNSUPPORTED, "GEOMETRIC body needs an FP precision");
    }
    default:
      return fail(HP_EUNSUPPORTED, "body not supported by the rectangular executor");
  }
}

// explicit instantiations live in rect_f32.cu, rect_f32mm.cu, rect_i32.cu, rect_i64.cu
hp_status launch_rect_f32_sum(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_f32_comp(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_f32_max(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_f32_min(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_i32_sum(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_i32_max(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_i32_min(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_i64_sum(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_i64_max(const NestPlan&, LaunchCfg&, const RectArgs&);
hp_status launch_rect_i64_min(const NestPlan&, LaunchCfg&, const RectArgs&);

// size in bytes of one grid-part partial for a precision / op
inline size_t partial_bytes(hp_prec prec, hp_red_op op) {
  if (prec == HP_F32_COMP && op == HP_RED_SUM) return 8;
  if (prec == HP_I64) return 8;
  return 4;
}

}  // namespace hp
