// bbw_elastic_lane.cuh -- the elastic stage with one element per lane (see
// bbw_lane.cuh): the flux kernel, and one warp per 32 elements and field for
// the spatial operator, the weight-adjusted projections and the RK update.
//
// Each of the nine fields is a task of its own: derivative terms, one lift per
// face of the field's flux (F_v,c, or A_n h combined from the three h before
// the lift, since A_n is constant on an affine face), projection, RK update.
// The trace of the stress bracket is a tenth task (div v and n . h), projected
// with lambda in an earlier launch than the normal stresses, which add it to
// their own projection with 2 mu. Ten tasks per 32 elements give every degree
// enough warps. Up to N = 5 a task projects its bracket in registers; above,
// the brackets of the nine fields wait for the projection kernels in their
// fields' places of q_out, which nothing reads before the RK update writes
// them. So only the fluxes and the trace take memory of their own,
// 24 N_fp + N_p values an element, beside a state of 45 N_p (three copies in
// FP32 and the FP64 staging).
#pragma once

#include "bbw_elastic.cuh"
#include "bbw_lane.cuh"

namespace bbw {

struct Elastic {
  static constexpr int NF = 9;  // v_x, v_y, v_z, s_xx, s_yy, s_zz, s_yz, s_xz, s_xy
  static constexpr int NQ = 6;  // F_v (3), h (3)
  static constexpr int MAXL = 3;
  static constexpr int SIGN = 1;
  static __device__ __forceinline__ TaskDesc task(int t) {
    switch (t) {
      case 0: return {3, 1, {{3, 0}, {8, 1}, {7, 2}}, {{0, -1}, {0, -1}, {0, -1}}};
      case 1: return {3, 1, {{8, 0}, {4, 1}, {6, 2}}, {{1, -1}, {1, -1}, {1, -1}}};
      case 2: return {3, 1, {{7, 0}, {6, 1}, {5, 2}}, {{2, -1}, {2, -1}, {2, -1}}};
      case 3: return {1, 1, {{0, 0}, {0, 0}, {0, 0}}, {{3, 0}, {3, 0}, {3, 0}}};
      case 4: return {1, 1, {{1, 1}, {1, 1}, {1, 1}}, {{4, 1}, {4, 1}, {4, 1}}};
      case 5: return {1, 1, {{2, 2}, {2, 2}, {2, 2}}, {{5, 2}, {5, 2}, {5, 2}}};
      case 6: return {2, 2, {{1, 2}, {2, 1}, {2, 1}}, {{4, 2}, {5, 1}, {5, 1}}};
      case 7: return {2, 2, {{0, 2}, {2, 0}, {2, 0}}, {{3, 2}, {5, 0}, {5, 0}}};
      case 8: return {2, 2, {{0, 1}, {1, 0}, {1, 0}}, {{3, 1}, {4, 0}, {4, 0}}};
      default: return {3, 3, {{0, 0}, {1, 1}, {2, 2}}, {{3, 0}, {4, 1}, {5, 2}}};  // the stress trace
    }
  }
};

template <int N, typename real>
__global__ void __launch_bounds__(kFluxThreads) elastic_flux_kernel(const LaneElasticParams<real> P,
                                                                    const uint16_t* __restrict__ fidx,
                                                                    const uint16_t* __restrict__ nidx) {
  flux_tile<Elastic, N, real>(
      P, fidx, nidx,
      [](const real (&own)[9], real (&nb)[9]) {  // traction-free mirror
#pragma unroll
        for (int k = 0; k < 9; ++k) nb[k] = k < 3 ? own[k] : -own[k];
      },
      [&](const real* n, const real (&own)[9], const real (&nb)[9], real (&out)[6]) {
        vec<real, 1> nv[3], jv[3], js[6], ts[3], anv[6], tan[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          nv[c].x[0] = n[c];
          jv[c].x[0] = nb[c] - own[c];
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) js[c].x[0] = nb[3 + c] - own[3 + c];
        traction(nv[0], nv[1], nv[2], js, ts);
        sym_normal(nv[0], nv[1], nv[2], jv, anv);
        traction(nv[0], nv[1], nv[2], anv, tan);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          out[c] = n[3] * fma(P.tau_v, tan[c].x[0], ts[c].x[0]);
          out[3 + c] = n[3] * fma(P.tau_s, ts[c].x[0], jv[c].x[0]);
        }
      });
}

// The projected right-hand side of a field in the columns -> its RK update;
// the trace task stores its projection instead. task as in Elastic::task.
template <int N, typename real, int S>
__device__ __forceinline__ void elastic_finish(const LaneElasticParams<real>& P, real* cols, int64_t e0, int ne, int lane,
                                               int task) {
  using Tile = WarpTile<np3(N), real>;
  constexpr int Np = np3(N);
  real* tr = P.trace + size_t(e0) * Np;
  if (task == 9) {
    Tile::template unstage<Np, S>(cols, tr, lane, ne);
    return;
  }
  if (task >= 3 && task < 6) {  // the lane adds to the column entries that it reads again below
    const real* p = tr + Tile::template first<Np>(lane);
    real* c = cols + Tile::template first<S>(lane);
    constexpr int U = Tile::IT < 16 ? Tile::IT : 16;
#pragma unroll
    for (int i0 = 0; i0 < Tile::IT; i0 += U) {
      typename Tile::Chunk t[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (Tile::has(lane, i0 + u, ne)) t[u] = Tile::load(p + Tile::template offset<Np>(i0 + u));
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (Tile::has(lane, i0 + u, ne))
#pragma unroll
          for (int w = 0; w < Tile::W; ++w) c[Tile::template offset<S>(i0 + u) + w] += t[u].x[w];
    }
  }
  lane_rk<N, 9, real, S>(P, cols, e0, ne, lane, task, [&](int) { return P.dt; }, [](int) { return false; });
}

// weight of a task and its factor
__device__ __forceinline__ int elastic_weight(int task) { return task < 3 ? 0 : task == 9 ? 1 : 2; }

// One warp per 32 elements and task. FUSED: the tasks of one
// launch are TRACE ? {trace, v_x, v_y, v_z} : the six stresses. Otherwise the
// brackets go to q_out and P.trace for elastic_project_kernel.
template <int N, int M, typename real, bool FUSED, bool TRACE>
__global__ void __launch_bounds__(FieldShape<N, real>::THREADS, N == 5 ? 2 : kFieldCtas<N>)
    elastic_field_kernel(const LaneElasticParams<real> P) {
  using C = FieldShape<N, real>;
  using Tile = WarpTile<np3(N), real>;
  constexpr int Np = np3(N), Mp = np3(M), S = C::S;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  real* cols = reinterpret_cast<real*>(smem + warp * C::WARP_BYTES);
  // the tasks of the same elements run in neighbouring CTAs (shared inputs in L2)
  constexpr int NT = !FUSED ? 10 : TRACE ? 4 : 6;
  const int64_t e0 = (int64_t(blockIdx.x / NT) * C::WARPS + warp) * 32;
  const int ne = P.G - e0 < 32 ? int(P.G - e0) : 32;
  if (ne <= 0) return;  // warps are independent
  const int y = blockIdx.x % NT;
  const int task = !FUSED ? y : TRACE ? (y == 0 ? 9 : y - 1) : 3 + y;
  LaneGeom<real> gm;
  gm.load(P.geom, e0, lane);
  typename WeightTile<M, real>::Held wt;
  if constexpr (FUSED)
    WeightTile<M, real>::template hold<3 * Mp>(wt, P.media + (size_t(e0) * 3 + elastic_weight(task)) * Mp, lane, ne);
  if (FUSED && task < 9) {
    Tile::template prefetch<9 * Np>(P.qin + (size_t(e0) * 9 + task) * Np, lane, ne);
    if (P.a != real(0)) Tile::template prefetch<9 * Np>(P.res + (size_t(e0) * 9 + task) * Np, lane, ne);
  }
  real r[Np];
  field_rhs<Elastic, N, real, S>(Elastic::task(task), P.qin, P.flux, e0, ne, lane, cols, gm, r);
  to_power<N, real>(r);
  if constexpr (FUSED) {
    real wc[Mp];
    const bool normal = !TRACE && task < 6;
    lane_weight<M, S>(wt, cols, lane, ne, normal ? real(2) : real(1), wc);
    Projector<N, M, real>::run(r, r, static_cast<real*>(nullptr), wc, P.cs);
    put_column(cols + lane * S, r);
    __syncwarp();
    elastic_finish<N, real, S>(P, cols, e0, ne, lane, task);
  } else {
    put_column(cols + lane * S, r);
    __syncwarp();
    if (task == 9)
      Tile::template unstage<Np, S>(cols, P.trace + size_t(e0) * Np, lane, ne);
    else
      Tile::template unstage<9 * Np, S>(cols, P.qout + (size_t(e0) * 9 + task) * Np, lane, ne);
  }
}

// Projections and RK updates from the brackets in q_out and P.trace, tasks per
// launch as in the fused elastic_field_kernel. A warp reads its whole bracket
// before it writes the field there.
template <int N, int M, typename real, bool TRACE>
__global__ void __launch_bounds__(ProjectShape<N, M, real>::THREADS)
    elastic_project_kernel(const LaneElasticParams<real> P) {
  using C = ProjectShape<N, M, real>;
  using Tile = WarpTile<np3(N), real>;
  constexpr int Np = np3(N), Mp = np3(M), S = C::S;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  real* cols = reinterpret_cast<real*>(smem + warp * C::WARP_BYTES);
  constexpr int NT = TRACE ? 4 : 6;
  const int64_t e0 = (int64_t(blockIdx.x / NT) * C::WARPS + warp) * 32;
  const int ne = P.G - e0 < 32 ? int(P.G - e0) : 32;
  if (ne <= 0) return;
  const int y = blockIdx.x % NT;
  const int task = TRACE ? (y == 0 ? 9 : y - 1) : 3 + y;
  typename WeightTile<M, real>::Held wt;
  WeightTile<M, real>::template hold<3 * Mp>(wt, P.media + (size_t(e0) * 3 + elastic_weight(task)) * Mp, lane, ne);
  if (task < 9) {
    Tile::template prefetch<9 * Np>(P.qin + (size_t(e0) * 9 + task) * Np, lane, ne);
    if (P.a != real(0)) Tile::template prefetch<9 * Np>(P.res + (size_t(e0) * 9 + task) * Np, lane, ne);
  }
  real wc[Mp];
  const bool normal = !TRACE && task < 6;
  lane_weight<M, S>(wt, cols, lane, ne, normal ? real(2) : real(1), wc);
  constexpr int U = Tile::IT < 28 ? Tile::IT : 28;
  if (task == 9)
    Tile::template stage<Np, S, U>(cols, P.trace + size_t(e0) * Np, lane, ne);
  else
    Tile::template stage<9 * Np, S, U>(cols, P.qout + (size_t(e0) * 9 + task) * Np, lane, ne);
  __syncwarp();
  Projector<N, M, real>::run(cols + lane * S, cols + lane * S, cols + lane * S, wc, P.cs);
  __syncwarp();
  elastic_finish<N, real, S>(P, cols, e0, ne, lane, task);
}

}  // namespace bbw
