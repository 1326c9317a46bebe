// bbw_stage_inst.cuh -- instantiate the stage and WADG kernels for one degree.
// Included by bbw_stage_n<N>.cu with BBW_N defined.
#pragma once

#include <new>

#include <cstddef>

#include "bbw_ops.h"
#include "bbw_stage.cuh"
#include "bbw_tile.cuh"

#ifndef BBW_N
#error "define BBW_N before including bbw_stage_inst.cuh"
#endif

namespace bbw {
namespace {

constexpr int kN = BBW_N;

template <typename real>
using Shape = TileShape<kN, real>;

template <int M, typename real>
constexpr int kGC = fat_cta_groups<kN, M, real, Shape<real>::T, Shape<real>::V>();

template <int M, typename real>
using Cfg = StageCfg<kN, M, real, Shape<real>::T, Shape<real>::V, kGC<M, real>>;

template <int M, typename real>
constexpr auto stage_fn() {
  return stage_kernel<kN, M, real, Shape<real>::T, Shape<real>::V, kGC<M, real>>;
}
template <int M, typename real>
constexpr auto spatial_fn() {
  return stage_kernel<kN, M, real, Shape<real>::T, Shape<real>::V, kGC<M, real>, true>;
}
template <int M, typename real>
constexpr auto wadg_fn() {
  return wadg_kernel<kN, M, real, Shape<real>::T, Shape<real>::V, kGC<M, real>>;
}
template <int M, typename real>
constexpr auto adj_pre_fn() {
  return adj_pre_kernel<kN, M, real, Shape<real>::T, Shape<real>::V, kGC<M, real>>;
}

// The tile kernels (bbw_tile.cuh) run solvers of at least kLaneMin elements,
// N <= 6 in FP32 and N <= 5 in FP64; the team kernels (bbw_stage.cuh) the rest
// (the same bits either way). A tile has 32 elements, so small meshes leave
// SMs idle, and a warp's chain of work is longer than a team's. Both times rise
// in steps, at the sizes where an SM gets one more CTA (tile: multiples of 32 x
// 152 = 4,864 elements; team: of its CTA's elements x 152), so their ratio
// jumps there, and the constants lie at the steps from which on the tile kernel
// is nowhere slower (every 3 to 5 % of size measured, M = 0..3; tile / team):
//   FP32, N = 1  M = 0, 1: 1.00 below 4,900, 1.26 up to 9,728 (both sizes one
//                step higher: 7.9 us against 6.2 a stage), 0.95 to 1.00 above, and
//                at M = 0 again 1.03 to 1.14 between 34,800 and 57,000;
//                M = 2, 3: below 1 everywhere (4,374 elements: 0.78)
//         N = 2  1.00 to 1.25 below, 0.91 to 0.97 at 9,867
//         N = 3  1.0 to 1.2 below 4,864, 0.86 to 0.97 above, 0.70 to 0.85 from 9,757
//         N = 4  0.79 to 0.98 below 9,728, 0.55 to 0.85 above
//         N = 5  0.60 to 0.75 below, 0.38 to 0.78 above
//         N = 6  1.6 to 1.95 below 4,864, 1.05 to 1.2 below 14,600, then by steps
//                0.82 to 1.05, and 0.80 to 0.99 from 65,000
//   FP64, N = 1  0.50 to 0.94       N = 2  0.98 to 1.10 below 4,864, 0.76 to 0.89 above
//         N = 3  up to 1.7 below 2,432, 0.91 to 1.01 up to 4,864, 0.91 to 0.96 above
//         N = 4  0.55 to 0.98       N = 5  1.01 to 2.1 below, 0.93 to 0.97 above
// Us a stage, M = 2, 82,944 elements, FP32, tile / team: N = 1 21/27, 2 33/46,
// 3 50/82, 4 110/146, 5 142/219, 6 270/302; N = 7 456/412, and N >= 8 does not
// fit the registers.
template <typename real>
constexpr bool kLane = kN <= (sizeof(real) == 4 ? 6 : 5);
template <int M, typename real>
constexpr int64_t kLaneMin = sizeof(real) == 4
                                 ? (kN == 1 ? (M == 0 ? 59000 : M == 1 ? 9800 : 0)
                                    : kN == 2 ? 10000
                                    : kN == 3 ? 9000
                                    : kN == 6 ? 80000
                                              : 0)
                                 : (kN == 2 || kN == 3 ? 5000 : kN == 5 ? 6000 : 0);
// The team kernels of the stage exist for solvers below that size only.
template <int M, typename real>
constexpr bool kTeam = !kLane<real> || kLaneMin<M, real> > 0;
// The projection of p runs in the tile kernel where its levels fit the
// registers (N <= 5, FP64 4); at N = 6 one warp of four would work on it for
// longer than the rest of the tile takes (291 us fused, 270 apart).
template <typename real>
constexpr bool kFuseProjection = kN <= (sizeof(real) == 4 ? 5 : 4);
template <typename real>
constexpr int kStageMode = kFuseProjection<real> ? kFused : kBracket;
template <int M, typename real, int MODE>
constexpr auto tile_fn() {
  return acoustic_tile_kernel<kN, MODE == kFused ? M : 0, real, MODE>;  // only the fused kernel depends on M
}

template <typename F>
auto dispatch(int M, bool dbl, F&& f) {
  switch (M) {
    case 0: return dbl ? f.template operator()<0, double>() : f.template operator()<0, float>();
    case 1: return dbl ? f.template operator()<1, double>() : f.template operator()<1, float>();
    case 2: return dbl ? f.template operator()<2, double>() : f.template operator()<2, float>();
    default: return dbl ? f.template operator()<3, double>() : f.template operator()<3, float>();
  }
}

void launch_shape(int M, bool dbl, int* team, int* width, int* groups) {
  dispatch(M, dbl, [&]<int MM, typename real>() {
    *team = Shape<real>::T;
    *width = Shape<real>::V;
    *groups = kGC<MM, real>;
    return 0;
  });
}

size_t tables_size(int M, bool dbl) {
  return dispatch(M, dbl, []<int MM, typename real>() { return size_t(Cfg<MM, real>::TAB); });
}

void build(int M, bool dbl, const double* cj, void* buf) {
  dispatch(M, dbl, [&]<int MM, typename real>() {
    auto* t = new (buf) Tables<kN, MM, real>();
    build_tables<kN, MM, real>(*t, cj);
    return 0;
  });
}

const char* check_tables(int M, bool dbl, const double* cj) {
  return dispatch(M, dbl, [&]<int MM, typename real>() -> const char* {
    auto* t = new Tables<kN, MM, real>();
    build_tables<kN, MM, real>(*t, cj);
    const char* msg = validate_tables<kN, MM, real>(*t);
    delete t;
    return msg;
  });
}

void face_maps(int* fidx, int* nidx) {
  auto* t = new Tables<kN, 0, double>();
  const double cj[kN + 1] = {};
  build_tables<kN, 0, double>(*t, cj);
  for (int i = 0; i < 4 * np2(kN); ++i) fidx[i] = t->fidx[i];
  for (int i = 0; i < 24 * np2(kN); ++i) nidx[i] = t->nidx[i];
  delete t;
}

template <typename K>
cudaError_t allow_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t prepare(int M, bool dbl, int* per_sm_stage, int* per_sm_wadg) {
  return dispatch(M, dbl, [&]<int MM, typename real>() {
    using C = Cfg<MM, real>;
    *per_sm_stage = 1;
    cudaError_t err = cudaSuccess;
    // (the stage kernel before the WADG kernel: instantiated the other way round,
    // the latter is compiled to other registers, up to 5 % slower)
    if constexpr (kTeam<MM, real>) {
      auto ks = stage_fn<MM, real>();
      err = allow_smem(ks, C::SMEM);
      if (err == cudaSuccess)
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm_stage, ks, C::THREADS, C::SMEM);
    }
    auto kw = wadg_fn<MM, real>();
    if (err == cudaSuccess) err = allow_smem(kw, C::SMEM);
    if constexpr (kTeam<MM, real>) {
      if (err == cudaSuccess) err = allow_smem(spatial_fn<MM, real>(), C::SMEM);
      if (err == cudaSuccess) err = allow_smem(adj_pre_fn<MM, real>(), C::SMEM);
    }
    if constexpr (kLane<real>) {
      using PC = ProjectShape<kN, MM, real>;
      if (err == cudaSuccess) err = allow_smem(tile_fn<MM, real, kStageMode<real>>(), TileCfg<kN, real>::SMEM);
      if (err == cudaSuccess) err = allow_smem(tile_fn<MM, real, kSpatial>(), TileCfg<kN, real>::SMEM);
      if (err == cudaSuccess) err = allow_smem(lane_adj_pre_kernel<kN, MM, real>, PC::SMEM);
      if constexpr (!kFuseProjection<real>)
        if (err == cudaSuccess) err = allow_smem(acoustic_project_kernel<kN, MM, real>, PC::SMEM);
    }
    if (err != cudaSuccess) return err;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm_wadg, kw, C::THREADS, C::SMEM);
  });
}

// Warps per CTA of a kernel with one warp per 32 elements: one where the warps
// would not fill two CTAs on each of the 152 SMs.
template <typename C>
int lane_warps(int64_t G) {
  return (G + 31) / 32 < int64_t(2 * 152) * C::WARPS ? 1 : C::WARPS;
}

template <int M, typename real, int MODE>
void launch_tiles(const LaneStageParams<real>& P, cudaStream_t s) {
  using Tab = Tables<kN, M, real>;
  constexpr size_t at = offsetof(Tab, fidx);  // fidx and nidx, one after the other
  static_assert(at % 4 == 0 && offsetof(Tab, nidx) == at + sizeof(uint16_t) * 4 * np2(kN), "face tables");
  tile_fn<M, real, MODE>()<<<unsigned((P.G + 31) / 32), 128, TileCfg<kN, real>::SMEM, s>>>(
      P, reinterpret_cast<const uint32_t*>(static_cast<const char*>(P.tables) + at));
}

cudaError_t launch_stage(int M, bool dbl, const void* params, int grid, cudaStream_t s) {
  return dispatch(M, dbl, [&]<int MM, typename real>() {
    using C = Cfg<MM, real>;
    const auto& P = *static_cast<const LaneStageParams<real>*>(params);
    if constexpr (kLane<real>) {
      if (P.lane || !kTeam<MM, real>) {
        launch_tiles<MM, real, kStageMode<real>>(P, s);
        if constexpr (!kFuseProjection<real>) {
          using PC = ProjectShape<kN, MM, real>;
          const int w = lane_warps<PC>(P.G);
          acoustic_project_kernel<kN, MM, real>
              <<<unsigned((P.G + 32 * w - 1) / (32 * w)), 32 * w, w * PC::WARP_BYTES, s>>>(P);
        }
        return cudaGetLastError();
      }
    }
    if constexpr (kTeam<MM, real>) stage_fn<MM, real>()<<<grid, C::THREADS, C::SMEM, s>>>(P);
    return cudaGetLastError();
  });
}

cudaError_t launch_spatial(int M, bool dbl, const void* params, int grid, cudaStream_t s) {
  return dispatch(M, dbl, [&]<int MM, typename real>() {
    using C = Cfg<MM, real>;
    const auto& P = *static_cast<const LaneStageParams<real>*>(params);
    if constexpr (kLane<real>) {
      if (P.lane || !kTeam<MM, real>) {
        launch_tiles<MM, real, kSpatial>(P, s);
        return cudaGetLastError();
      }
    }
    if constexpr (kTeam<MM, real>) spatial_fn<MM, real>()<<<grid, C::THREADS, C::SMEM, s>>>(P);
    return cudaGetLastError();
  });
}

cudaError_t launch_wadg(int M, bool dbl, const void* params, int grid, cudaStream_t s) {
  return dispatch(M, dbl, [&]<int MM, typename real>() {
    using C = Cfg<MM, real>;
    wadg_fn<MM, real>()<<<grid, C::THREADS, C::SMEM, s>>>(
        *static_cast<const WadgParams<real>*>(params));
    return cudaGetLastError();
  });
}

cudaError_t launch_adj_pre(int M, bool dbl, const void* params, int grid, cudaStream_t s) {
  return dispatch(M, dbl, [&]<int MM, typename real>() {
    using C = Cfg<MM, real>;
    const auto& P = *static_cast<const LaneAdjPreParams<real>*>(params);
    if constexpr (kLane<real>) {
      if (P.lane || !kTeam<MM, real>) {
        using PC = ProjectShape<kN, MM, real>;
        const int w = lane_warps<PC>(P.G);
        lane_adj_pre_kernel<kN, MM, real>
            <<<4 * unsigned((P.G + 32 * w - 1) / (32 * w)), 32 * w, w * PC::WARP_BYTES, s>>>(P);
        return cudaGetLastError();
      }
    }
    if constexpr (kTeam<MM, real>) adj_pre_fn<MM, real>()<<<grid, C::THREADS, C::SMEM, s>>>(P);
    return cudaGetLastError();
  });
}

int64_t lane_min(int M, bool dbl) {
  return dispatch(M, dbl, [&]<int MM, typename real>() { return kLane<real> ? kLaneMin<MM, real> : INT64_MAX; });
}

}  // namespace

#define BBW_CAT2(a, b) a##b
#define BBW_CAT(a, b) BBW_CAT2(a, b)
const KernelOps& BBW_CAT(ops_n, BBW_N)() {
  static const KernelOps ops = {&tables_size,  &build,          &face_maps,    &prepare,
                                &launch_stage, &launch_wadg,    &launch_shape, &launch_spatial,
                                &check_tables, &launch_adj_pre, &lane_min};
  return ops;
}

}  // namespace bbw
