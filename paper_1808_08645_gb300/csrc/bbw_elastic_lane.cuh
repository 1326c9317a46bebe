// bbw_elastic_lane.cuh -- the elastic stage with one element per lane (see
// bbw_lane.cuh), two kinds of kernels:
//   flux kernel   the penalty fluxes at the face nodes of every element, one
//                 face node per lane (neighbour traces are short runs of the
//                 neighbour's field, so a warp's gather covers few sectors),
//                 transposed through shared memory to lines of 32 elements;
//   field tasks   one warp per 32 elements and field, one element per lane:
//                 spatial operator, weight-adjusted projection, RK update.
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
//
// The field tasks of the same elements run in neighbouring CTAs, so that their
// common inputs come from L2 (task-major order took 1.8 times the DRAM bytes).
// Registers bound the warps per SM (8 to 24); the code of a task (30 to 100 KB)
// exceeds the instruction cache from N = 5 on, which is why warps of a CTA, in
// step with each other, do better than as many smaller CTAs.
#pragma once

#include "bbw_elastic.cuh"
#include "bbw_lane.cuh"

namespace bbw {

constexpr int kElasticFields = 9;  // v_x, v_y, v_z, s_xx, s_yy, s_zz, s_yz, s_xz, s_xy
constexpr int kElasticFluxes = 6;  // F_v (3), h (3)

// A field task: derivative term t adds d f / d x_d of field `what`, lift term t
// the flux `what` times n_d (d < 0: times 1).
struct Term {
  int8_t what, dir;
};
struct TaskDesc {
  int nd, nl;
  Term d[3];
  Term l[3];
};

__device__ __forceinline__ TaskDesc elastic_task(int t) {
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

// Flux kernel: 4 warps per CTA and a tile of 16 elements, 8 where 16 elements'
// fluxes would take the shared memory that the gathers need as L1.
constexpr int kFluxThreads = 128;
template <int N>
constexpr int kFluxTile = kElasticFluxes * 4 * np2(N) <= 224 ? 16 : 8;

template <int N, typename real>
constexpr int flux_smem() {
  // fluxes [6][4 Nfp][tile + 1] | normals [tile][4][4] | connectivity [tile][4]
  constexpr int T = kFluxTile<N>;
  return int(sizeof(real)) * (kElasticFluxes * 4 * np2(N) * (T + 1) + T * 16) + T * 16;
}
// values of the flux buffer of K elements (whole tiles of 32)
constexpr size_t flux_values(int64_t K, int Nfp) {
  return size_t((K + 31) / 32) * 32 * kElasticFluxes * 4 * size_t(Nfp);
}

// The fluxes of a tile: flux(nrm, own[NF], nb[NF], out[NQ]) per face node.
// Walls: mirror(own, nb). Layout of P.flux: [K / 32][6][4][Nfp][32].
template <int N, typename real, typename Mirror, typename Flux>
__device__ __forceinline__ void flux_tile(const LaneElasticParams<real>& P, const uint16_t* __restrict__ fidx,
                                          const uint16_t* __restrict__ nidx, Mirror&& mirror, Flux&& flux) {
  constexpr int Np = np3(N), Nfp = np2(N), NF = kElasticFields, NQ = kElasticFluxes, ITEMS = 4 * Nfp;
  constexpr int T = kFluxTile<N>, ST = T + 1;
  extern __shared__ __align__(16) unsigned char smem[];
  real* FL = reinterpret_cast<real*>(smem);           // [NQ][4 Nfp][ST]
  real* NRM = FL + NQ * ITEMS * ST;                   // [tile][4][nx, ny, nz, |f| / (2 |D|)]
  int* CS = reinterpret_cast<int*>(NRM + T * 16);  // [tile][4]
  const int64_t e0 = int64_t(blockIdx.x) * T;
  const int ne = P.G - e0 < T ? int(P.G - e0) : T;
  const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
  bool oob = false;
  (void)oob;
  if (tid < 4 * T) {
    const int e = tid / 4, f = tid % 4;
    if (e < ne) {
      CS[tid] = P.conn[size_t(e0 + e) * 4 + f];
      const real* g = P.geom + size_t((e0 + e) / 32) * 32 * kLaneGeom + (e0 + e) % 32;
      const real inv = g[(9 + f) * 32];
      real* nr = NRM + tid * 4;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const real a = g[d * 32], b = g[(3 + d) * 32], c = g[(6 + d) * 32];
        nr[d] = (f == 0 ? a + b + c : f == 1 ? -a : f == 2 ? -b : -c) * inv;
      }
      nr[3] = real(1.5) / inv;
    }
  }
  __syncthreads();
  constexpr int EW = T / (kFluxThreads / 32);  // elements per warp
  constexpr int UE = 1;                        // of which in flight together (nine fields each)
#pragma unroll 1
  for (int it = lane; it < ITEMS; it += 32) {
    const int f = it / Nfp, a = it - f * Nfp;
    int io = fidx[it];
    if constexpr (kChecked) {
      if (io >= Np) {
        oob = true;
        io = 0;
      }
    }
#pragma unroll 1
    for (int j0 = 0; j0 < EW; j0 += UE) {
      real own[UE][NF], nbv[UE][NF];
      bool wall[UE];
#pragma unroll
      for (int u = 0; u < UE; ++u) {
        const int e = warp * EW + j0 + u;
        const int c = e < ne ? CS[e * 4 + f] : -1;
        wall[u] = c < 0;
        const real* src = P.qin + size_t(e0 + (e < ne ? e : 0)) * NF * Np + io;
#pragma unroll
        for (int k = 0; k < NF; ++k) own[u][k] = src[k * Np];
        if (c >= 0) {
          const int64_t nb = int64_t(c >> 5);
          if constexpr (kChecked) {
            if (nb >= P.G || (c & 7) >= 6) {
              oob = true;
              wall[u] = true;
              continue;
            }
          }
          const int ni = nidx[(((c >> 3) & 3) * 6 + (c & 7)) * Nfp + a];
          if constexpr (kChecked) {
            if (ni >= Np) {
              oob = true;
              wall[u] = true;
              continue;
            }
          }
          const real* nsrc = P.qin + size_t(nb) * NF * Np + ni;
#pragma unroll
          for (int k = 0; k < NF; ++k) nbv[u][k] = nsrc[k * Np];
        }
      }
#pragma unroll
      for (int u = 0; u < UE; ++u) {
        const int e = warp * EW + j0 + u;
        if (e >= ne) continue;
        if (wall[u]) mirror(own[u], nbv[u]);
        real out[NQ];
        flux(NRM + (e * 4 + f) * 4, own[u], nbv[u], out);
#pragma unroll
        for (int q = 0; q < NQ; ++q) FL[(q * ITEMS + it) * ST + e] = out[q];
      }
    }
  }
  __syncthreads();
  real* dst = P.flux + size_t(e0 / 32) * 32 * NQ * ITEMS + e0 % 32;
  for (int x = tid; x < NQ * ITEMS * T; x += kFluxThreads) {
    const int r = x / T, e = x % T;
    if (e < ne) dst[size_t(r) * 32 + e] = FL[r * ST + e];
  }
  if constexpr (kChecked) {
    if (oob) atomicOr(P.status, 2u);
  }
}

template <int N, typename real>
__global__ void __launch_bounds__(kFluxThreads) elastic_flux_kernel(const LaneElasticParams<real> P,
                                                                    const uint16_t* __restrict__ fidx,
                                                                    const uint16_t* __restrict__ nidx) {
  flux_tile<N, real>(
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

// grad lambda_0..3 and 1 / |grad lambda_f| of the lane's element
// (LaneGeom::load: rows of the warp's block of kLaneGeom x 32 values)
template <typename real>
struct LaneGeom {
  real g[4][3], inv[4];
  __device__ __forceinline__ void load(const real* __restrict__ geom, int64_t e0, int lane) {
    const real* p = geom + size_t(e0 / 32) * 32 * kLaneGeom + lane;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
      for (int m = 1; m < 4; ++m) g[m][d] = p[(3 * (m - 1) + d) * 32];
      g[0][d] = -g[1][d] - g[2][d] - g[3][d];
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) inv[f] = p[(9 + f) * 32];
  }
};

// The lane's flux q on face f (fl: the warp's [NQ][4][Nfp][32] block at the lane).
template <int N, int f, typename real>
__device__ __forceinline__ void load_flux(const real* __restrict__ fl, int q, real (&F)[np2(N)]) {
  const real* src = fl + (q * 4 + f) * np2(N) * 32;
#pragma unroll
  for (int i = 0; i < np2(N); ++i) F[i] = src[i * 32];
}

// The task's flux on face f, sum over its lift terms of n_d F_q (F holds the
// first term's flux), lifted into the lane's right-hand side.
template <int N, int f, typename real>
__device__ __forceinline__ void lift_face(const TaskDesc& td, const real* __restrict__ fl, const LaneGeom<real>& gm,
                                          real (&F)[np2(N)], real (&r)[np3(N)]) {
  constexpr int Nfp = np2(N);
  real w = td.l[0].dir >= 0 ? -pick(gm.g[f], td.l[0].dir) * gm.inv[f] : real(1);
  if (td.nl > 1) {
#pragma unroll
    for (int i = 0; i < Nfp; ++i) F[i] *= w;
    w = real(1);
#pragma unroll 1
    for (int t = 1; t < td.nl; ++t) {
      const Term tm = t == 1 ? td.l[1] : td.l[2];
      const real wt = tm.dir >= 0 ? -pick(gm.g[f], tm.dir) * gm.inv[f] : real(1);
      const real* src = fl + (tm.what * 4 + f) * Nfp * 32;
#pragma unroll
      for (int i = 0; i < Nfp; ++i) F[i] = fma(wt, src[i * 32], F[i]);
    }
  }
  FieldRhs<N, real>::template lift<f>(r, F, w);
}

// Right-hand side r of field task td, lane = element; gm: the lane's
// geometry, cols: the warp's columns (stride S) for the staged fields.
// Loads are issued one step ahead: the first flux before the staging, each
// term's field (where the registers allow) and each face's flux during the
// work on the one before.
template <int N, typename real, int S>
__device__ __forceinline__ void field_rhs(const TaskDesc& td, const real* __restrict__ qin,
                                          const real* __restrict__ fluxes, int64_t e0, int ne, int lane, real* cols,
                                          const LaneGeom<real>& gm, real (&r)[np3(N)]) {
  using R = FieldRhs<N, real>;
  using Tile = WarpTile<np3(N), real>;
  constexpr int Np = R::Np, Nfp = R::Nfp, NF = kElasticFields, ES = NF * Np;
  constexpr bool AHEAD = Tile::IT * Tile::W * int(sizeof(real)) <= 4 * 100;
  constexpr int U = Tile::IT < 16 ? Tile::IT : 16;
  const real* col = cols + lane * S;
  const real* q0 = qin + size_t(e0) * ES;
  const real* fl = fluxes + size_t(e0 / 32) * 32 * kElasticFluxes * 4 * Nfp + lane;
  typename Tile::Held held;
  if constexpr (AHEAD) Tile::template hold<ES>(held, q0 + td.d[0].what * Np, lane, ne);
  real F3[Nfp], F2[Nfp], F1[Nfp], F0[Nfp];
  load_flux<N, 3>(fl, td.l[0].what, F3);
  real v1[R::Nm1p];
#pragma unroll
  for (int i = 0; i < R::Nm1p; ++i) v1[i] = real(0);
#pragma unroll 1
  for (int t = 0; t < td.nd; ++t) {
    const Term tm = t == 0 ? td.d[0] : t == 1 ? td.d[1] : td.d[2];
    if (t > 0) __syncwarp();
    if constexpr (AHEAD) {
      Tile::template put<S>(held, cols, lane, ne);
      if (t + 1 < td.nd) Tile::template hold<ES>(held, q0 + (t == 0 ? td.d[1].what : td.d[2].what) * Np, lane, ne);
    } else {
      Tile::template stage<ES, S, U>(cols, q0 + tm.what * Np, lane, ne);
    }
    __syncwarp();
    real w[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) w[m] = pick(gm.g[m], tm.dir);
    R::add_term(v1, col, w);
  }
  __syncwarp();  // the columns are free
  R::elevate_all(v1, r);
  load_flux<N, 2>(fl, td.l[0].what, F2);
  lift_face<N, 3>(td, fl, gm, F3, r);
  load_flux<N, 1>(fl, td.l[0].what, F1);
  lift_face<N, 2>(td, fl, gm, F2, r);
  load_flux<N, 0>(fl, td.l[0].what, F0);
  lift_face<N, 1>(td, fl, gm, F1, r);
  lift_face<N, 0>(td, fl, gm, F0, r);
}

template <int N, typename real>
using FieldShape = LaneShape<(np3(N) > np3(kMaxM) ? np3(N) : np3(kMaxM)), real, (N >= 6 ? 8 : 4)>;
// CTAs per SM that the field kernels' registers have to allow. Stack at
// M <= 2: 8 to 72 bytes at N = 2, 32 to 112 at N = 3, none to 16 above
template <int N>
constexpr int kFieldCtas = N == 2 ? 8 : N == 3 ? 6 : N == 4 ? 4 : N == 5 ? 2 : 1;

// The projected right-hand side of a field in the columns -> its RK update;
// the trace task stores its projection instead. task as in elastic_task.
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
__global__ void __launch_bounds__(FieldShape<N, real>::THREADS, kFieldCtas<N>)
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
  field_rhs<N, real, S>(elastic_task(task), P.qin, P.flux, e0, ne, lane, cols, gm, r);
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
// before it writes the field there. At N = 7 the levels do not fit the 255
// registers: 136 to 280 bytes of stack.
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
