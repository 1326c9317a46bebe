// bbw_lane.cuh -- the spatial operator and the RK update with one element per
// lane: the parts shared by the acoustic tile kernel (bbw_tile.cuh) and the
// elastic field tasks (bbw_elastic_lane.cuh), and the elastic form, two kinds
// of kernels per stage:
//   flux kernel   the penalty fluxes at the face nodes of every element, with
//                 one face node per lane (neighbour traces are short runs of
//                 the neighbour's field, so a warp's gather covers few
//                 sectors), transposed through shared memory to [32 elements]
//                 lines;
//   field tasks   one warp per 32 elements and field, one element per lane:
//                 derivative terms, lift of the four faces, the projection
//                 (bbw_project.cuh) and the RK update.
// A field's right-hand side is  E sum_t D_{d_t} f_t + sum_face L^f F: with the
// element in a lane every stencil index and weight is an immediate, the degree
// N-1 combination (V1), the lift pyramid and the right-hand side are registers
// (N_p <= 120: up to N = 7), and shared memory only transposes between the
// lanes' elements and contiguous global accesses. Nothing is shared between
// warps, so they never wait for each other.
//
// The field tasks of the same elements run in neighbouring CTAs, so that their
// common inputs come from L2 (task-major order took 1.8 times the DRAM bytes).
// Registers bound the warps per SM (8 to 24); the code of a task (30 to 100 KB)
// exceeds the instruction cache from N = 5 on, which is why warps of a CTA, in
// step with each other, do better than as many smaller CTAs.
#pragma once

#include "bbw_project.cuh"
#include "bbw_stage.cuh"
#include "bbw_warp_tile.cuh"

namespace bbw {

// Physics descriptions: fields, flux quantities and the terms of each field
// task. Derivative term t adds sgn * d f / d x_d; lift term t the flux
// quantity q times n_d (d < 0: times 1).
struct Term {
  int8_t what, dir;
};
struct TaskDesc {
  int nd, nl;
  Term d[3];
  Term l[3];
};

// Flux kernel: 4 warps per CTA and a tile of 16 elements, 8 where 16 elements'
// fluxes would take the shared memory that the gathers need as L1.
constexpr int kFluxThreads = 128;
template <int N, int NQ>
constexpr int kFluxTile = NQ * 4 * np2(N) <= 224 ? 16 : 8;

template <int N, int NQ, typename real>
constexpr int flux_smem() {
  // fluxes [NQ][4 Nfp][tile + 1] | normals [tile][4][4] | connectivity [tile][4]
  constexpr int T = kFluxTile<N, NQ>;
  return int(sizeof(real)) * (NQ * 4 * np2(N) * (T + 1) + T * 16) + T * 16;
}
// values of the flux buffer of K elements (whole tiles of 32)
template <int NQ>
constexpr size_t flux_values(int64_t K, int Nfp) {
  return size_t((K + 31) / 32) * 32 * NQ * 4 * size_t(Nfp);
}

// The fluxes of a tile: flux(nrm, own[NF], nb[NF], out[NQ]) per face node.
// Walls: mirror(own, nb). Layout of P.flux: [K / 32][NQ][4][Nfp][32].
template <typename Phys, int N, typename real, typename Params, typename Mirror, typename Flux>
__device__ __forceinline__ void flux_tile(const Params& P, const uint16_t* __restrict__ fidx,
                                          const uint16_t* __restrict__ nidx, Mirror&& mirror, Flux&& flux) {
  constexpr int Np = np3(N), Nfp = np2(N), NF = Phys::NF, NQ = Phys::NQ, ITEMS = 4 * Nfp;
  constexpr int T = kFluxTile<N, NQ>, ST = T + 1;
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
  constexpr int UE = NF <= 4 ? EW : 1;                 // of which in flight together
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

// ---------------------------------------------------------------------------
// field tasks

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

// component d of the gradient of lambda_m
template <typename real>
__device__ __forceinline__ real pick(const real (&g)[3], int d) {
  return d == 0 ? g[0] : d == 1 ? g[1] : g[2];
}

// volume index of node (b1, b2) of level i (degree N - i) of face f's pyramid
template <int N>
BBW_HD constexpr int lift_node(int f, int i, int b1, int b2) {
  // (b0, b1, b2) on the vertices other than f in increasing order, alpha_f = i
  const int b0 = N - i - b1 - b2;
  return f == 0 ? idx3(N, b0, b1, b2) : f == 1 ? idx3(N, i, b1, b2) : f == 2 ? idx3(N, b1, i, b2) : idx3(N, b1, b2, i);
}
// ell_i / (ell_{i-1} (N - i + 1)), ell_i = (-1)^i C(N, i) / (i + 1): from the
// integer-weight reduction of stored level i - 1 to stored level i (computed as
// for the tables, so that the factor is the same number)
BBW_HD constexpr double lift_ell(int N, int i) { return ((i & 1) ? -1.0 : 1.0) * cbinom(N, i) / (i + 1); }
BBW_HD constexpr double lift_scale(int N, int i) { return lift_ell(N, i) / (lift_ell(N, i - 1) * (N - i + 1)); }

template <int N, typename real>
struct FieldRhs {
  static constexpr int Np = np3(N), Nm1p = np3(N - 1), Nfp = np2(N);

  // V1 += sum_m w_m f_{b + e_m} of the field in the column
  static __device__ __forceinline__ void add_term(real (&v1)[Nm1p], const real* col, const real (&w)[4]) {
    static_for<0, N + 1>([&](auto l_) BBW_ALWAYS_INLINE {
      constexpr int l = decltype(l_)::value;
      static_for<0, N - l + 1>([&](auto k_) BBW_ALWAYS_INLINE {
        constexpr int k = decltype(k_)::value;
#pragma unroll
        for (int j = 0; j <= N - l - k; ++j) {
          const real x = col[row3(N, k, l) + j];
          if (j + k + l < N) {
            real& o = v1[idx3(N - 1, j, k, l)];
            o = fma(w[0], x, o);
          }
          if (j > 0) {
            real& o = v1[idx3(N - 1, j - 1, k, l)];
            o = fma(w[1], x, o);
          }
          if (k > 0) {
            real& o = v1[idx3(N - 1, j, k - 1, l)];
            o = fma(w[2], x, o);
          }
          if (l > 0) {
            real& o = v1[idx3(N - 1, j, k, l - 1)];
            o = fma(w[3], x, o);
          }
        }
      });
    });
  }

  // V1 -= sum_m (g_m . (u, v, w)_{b + e_m}), m by m in the order of stage_kernel
  static __device__ __forceinline__ void add_div(real (&v1)[Nm1p], const real* u, const real* v, const real* w,
                                                 const real (&g)[4][3]) {
    static_for<0, N + 1>([&](auto l_) BBW_ALWAYS_INLINE {
      constexpr int l = decltype(l_)::value;
      static_for<0, N - l + 1>([&](auto k_) BBW_ALWAYS_INLINE {
        constexpr int k = decltype(k_)::value;
#pragma unroll
        for (int j = 0; j <= N - l - k; ++j) {
          const int i = row3(N, k, l) + j;
          const real x = u[i], y = v[i], z = w[i];
          auto add = [&](int m, int at) BBW_ALWAYS_INLINE {
            v1[at] = fma(-g[m][0], x, v1[at]);
            v1[at] = fma(-g[m][1], y, v1[at]);
            v1[at] = fma(-g[m][2], z, v1[at]);
          };
          if (j + k + l < N) add(0, idx3(N - 1, j, k, l));
          if (j > 0) add(1, idx3(N - 1, j - 1, k, l));
          if (k > 0) add(2, idx3(N - 1, j, k - 1, l));
          if (l > 0) add(3, idx3(N - 1, j, k, l - 1));
        }
      });
    });
  }

  static __device__ __forceinline__ void elevate_all(const real (&v1)[Nm1p], real (&r)[Np]) {
    static_for<0, N + 1>([&](auto l_) BBW_ALWAYS_INLINE {
      constexpr int l = decltype(l_)::value;
      static_for<0, N - l + 1>([&](auto k_) BBW_ALWAYS_INLINE {
        constexpr int k = decltype(k_)::value;
#pragma unroll
        for (int j = 0; j <= N - l - k; ++j) r[row3(N, k, l) + j] = elevate(v1, j, k, l);
      });
    });
  }

  // node (j, k, l) of the elevation N E^N_{N-1} V1 (integer weights)
  static __device__ __forceinline__ real elevate(const real (&v1)[Nm1p], int j, int k, int l) {
    const int a = N - j - k - l;
    real x = real(0);
    if (a > 0) x = wmul(real(a), v1[idx3(N - 1, j, k, l)]);
    if (j > 0) x = a > 0 ? wfma(real(j), v1[idx3(N - 1, j - 1, k, l)], x) : wmul(real(j), v1[idx3(N - 1, j - 1, k, l)]);
    if (k > 0) x = wfma(real(k), v1[idx3(N - 1, j, k - 1, l)], x);
    if (l > 0) x = wfma(real(l), v1[idx3(N - 1, j, k, l - 1)], x);
    return x;
  }

  // r += w L^f F of face f: L0 F, then the levels by 2D reductions, each added
  // to its nodes alpha_f = i.
  template <int f>
  static __device__ __forceinline__ void lift(real (&r)[Np], real (&F)[Nfp], real w) {
    real t[Nfp];
    // t = E'^T F at degree N - 1 (integer weights)
#pragma unroll
    for (int b2 = 0; b2 < N; ++b2)
#pragma unroll
      for (int b1 = 0; b1 < N; ++b1)
        if (b1 + b2 < N) {
          real x = wmul(real(N - b1 - b2), F[idx2(N, b1, b2)]);
          x = wfma(real(b1 + 1), F[idx2(N, b1 + 1, b2)], x);
          x = wfma(real(b2 + 1), F[idx2(N, b1, b2 + 1)], x);
          t[idx2(N - 1, b1, b2)] = x;
        }
    // level 0: ((2N+3) F + E' t) / 3
    const real third = real(1) / real(3);
#pragma unroll
    for (int b2 = 0; b2 <= N; ++b2)
#pragma unroll
      for (int b1 = 0; b1 <= N; ++b1)
        if (b1 + b2 <= N) {
          real x = wmul(real(2 * N + 3), F[idx2(N, b1, b2)]);
          const int a = N - b1 - b2;
          if (a > 0) x = wfma(real(a), t[idx2(N - 1, b1, b2)], x);
          if (b1 > 0) x = wfma(real(b1), t[idx2(N - 1, b1 - 1, b2)], x);
          if (b2 > 0) x = wfma(real(b2), t[idx2(N - 1, b1, b2 - 1)], x);
          F[idx2(N, b1, b2)] = wmul(third, x);
        }
    static_for<0, N + 1>([&](auto i_) BBW_ALWAYS_INLINE {
      constexpr int i = decltype(i_)::value, n = N - i;  // level i: degree n
      if constexpr (i > 0) {
        constexpr real s = real(lift_scale(N, i));
#pragma unroll
        for (int b2 = 0; b2 <= n; ++b2)
#pragma unroll
          for (int b1 = 0; b1 <= n; ++b1)
            if (b1 + b2 <= n) {
              real x = wmul(real(n + 1 - b1 - b2) * s, F[idx2(n + 1, b1, b2)]);
              x = wfma(real(b1 + 1) * s, F[idx2(n + 1, b1 + 1, b2)], x);
              x = wfma(real(b2 + 1) * s, F[idx2(n + 1, b1, b2 + 1)], x);
              t[idx2(n, b1, b2)] = x;
            }
#pragma unroll
        for (int x = 0; x < np2(n); ++x) F[x] = t[x];
      }
#pragma unroll
      for (int b2 = 0; b2 <= n; ++b2)
#pragma unroll
        for (int b1 = 0; b1 <= n; ++b1)
          if (b1 + b2 <= n) {
            real& o = r[lift_node<N>(f, i, b1, b2)];
            o = fma(w, F[idx2(n, b1, b2)], o);
          }
    });
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
template <typename Phys, int N, int f, typename real>
__device__ __forceinline__ void lift_face(const TaskDesc& td, const real* __restrict__ fl, const LaneGeom<real>& gm,
                                          real (&F)[np2(N)], real (&r)[np3(N)]) {
  constexpr int Nfp = np2(N);
  real w = td.l[0].dir >= 0 ? -pick(gm.g[f], td.l[0].dir) * gm.inv[f] : real(1);
  if constexpr (Phys::MAXL > 1) {
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
  }
  FieldRhs<N, real>::template lift<f>(r, F, w);
}

// Right-hand side r of field task td, lane = element; gm: the lane's
// geometry, cols: the warp's columns (stride S) for the staged fields.
// Loads are issued one step ahead: the first flux before the staging, each
// term's field (where the registers allow) and each face's flux during the
// work on the one before.
template <typename Phys, int N, typename real, int S>
__device__ __forceinline__ void field_rhs(const TaskDesc& td, const real* __restrict__ qin,
                                          const real* __restrict__ fluxes, int64_t e0, int ne, int lane, real* cols,
                                          const LaneGeom<real>& gm, real (&r)[np3(N)]) {
  using R = FieldRhs<N, real>;
  using Tile = WarpTile<np3(N), real>;
  constexpr int Np = R::Np, Nfp = R::Nfp, NF = Phys::NF, ES = NF * Np;
  constexpr bool AHEAD = Tile::IT * Tile::W * int(sizeof(real)) <= 4 * 100;
  constexpr int U = Tile::IT < 16 ? Tile::IT : 16;
  const real* col = cols + lane * S;
  const real* q0 = qin + size_t(e0) * ES;
  const real* fl = fluxes + size_t(e0 / 32) * 32 * Phys::NQ * 4 * Nfp + lane;
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
    for (int m = 0; m < 4; ++m) w[m] = real(Phys::SIGN) * pick(gm.g[m], tm.dir);
    R::add_term(v1, col, w);
  }
  __syncwarp();  // the columns are free
  R::elevate_all(v1, r);
  load_flux<N, 2>(fl, td.l[0].what, F2);
  lift_face<Phys, N, 3>(td, fl, gm, F3, r);
  load_flux<N, 1>(fl, td.l[0].what, F1);
  lift_face<Phys, N, 2>(td, fl, gm, F2, r);
  load_flux<N, 0>(fl, td.l[0].what, F0);
  lift_face<Phys, N, 1>(td, fl, gm, F1, r);
  lift_face<Phys, N, 0>(td, fl, gm, F0, r);
}

// Power coefficients c_beta / beta! of the lane's degree-M weight, times s.
// The weights of the warp's elements (ES values apart) are loaded ahead
// (WeightTile::hold) and transposed through the free columns.
template <int M, typename real>
using WeightTile = WarpTile<np3(M), real>;
template <int M, int S, typename real>
__device__ __forceinline__ void lane_weight(const typename WeightTile<M, real>::Held& h, real* cols, int lane, int ne,
                                            real s, real (&wc)[np3(M)]) {
  WeightTile<M, real>::template put<S>(h, cols, lane, ne);
  __syncwarp();
  static_for<0, M + 1>([&](auto l_) BBW_ALWAYS_INLINE {
    constexpr int l = decltype(l_)::value;
#pragma unroll
    for (int k = 0; k <= M - l; ++k)
#pragma unroll
      for (int j = 0; j <= M - l; ++j)
        if (j + k <= M - l) {
          const int b = idx3(M, j, k, l);
          wc[b] = wmul(real(1.0 / (cfact(j) * cfact(k) * cfact(l) * cfact(M - j - k - l))) * s, cols[lane * S + b]);
        }
  });
  __syncwarp();
}

// Bernstein -> power coefficients in place
template <int N, typename real, typename Vec>
__device__ __forceinline__ void to_power(Vec&& v) {
  static_for<0, N + 1>([&](auto l_) BBW_ALWAYS_INLINE {
    constexpr int l = decltype(l_)::value;
    static_for<0, N - l + 1>([&](auto k_) BBW_ALWAYS_INLINE {
      constexpr int k = decltype(k_)::value;
#pragma unroll
      for (int j = 0; j <= N - l - k; ++j)
        v[row3(N, k, l) + j] = wmul(real(1.0 / (cfact(j) * cfact(k) * cfact(l) * cfact(N - j - k - l))), v[row3(N, k, l) + j]);
    });
  });
}

// Warps per CTA for columns of COL entries: as asked for where two such CTAs
// fit an SM. Warps are independent, but those of a CTA start together and
// share the instruction fetch of code that exceeds the instruction cache.
template <int COL, typename real, int WANT = 4>
struct LaneShape {
  static constexpr int S = COL | 1;
  static constexpr int WARP_BYTES = int(sizeof(real)) * 32 * S;
  static constexpr int WARPS = WANT * WARP_BYTES <= kSmemPerCta ? WANT : 4 * WARP_BYTES <= kSmemPerCta ? 2 : 1;
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int SMEM = WARPS * WARP_BYTES;
};

// columns of the projection kernels (at least the N_p values and the weights)
template <int N, int M, typename real>
using ProjectShape = LaneShape<(Projector<N, M, real>::COL > np3(kMaxM) ? Projector<N, M, real>::COL : np3(kMaxM)), real>;

template <int Np, typename real>
__device__ __forceinline__ void put_column(real* col, const real (&r)[Np]) {
#pragma unroll
  for (int i = 0; i < Np; ++i) col[i] = r[i];
}

template <int N, typename real>
using FieldShape = LaneShape<(np3(N) > np3(kMaxM) ? np3(N) : np3(kMaxM)), real, (N >= 6 ? 8 : 4)>;
// CTAs per SM that the field kernels' registers have to allow: as many as fit
// without spills at M <= 2
template <int N>
constexpr int kFieldCtas = N == 1 ? 10 : N == 2 ? 8 : N == 3 ? 6 : N == 4 ? 4 : N == 5 ? 3 : 1;

// RK update of field fld (of NF) of the warp's elements from the columns:
// res = a res + dt rhs, q_out = q_in + b res.
// dt(gl): the time step of the warp's element gl; done(gl): it is left as it is.
template <int N, int NF, typename real, int S, typename Params, typename Dt, typename Done>
__device__ __forceinline__ void lane_rk(const Params& P, const real* cols, int64_t e0, int ne, int lane, int fld,
                                        Dt&& dt, Done&& done) {
  using Tile = WarpTile<np3(N), real>;
  constexpr int Np = np3(N), ES = NF * Np, U = Tile::IT < 8 ? Tile::IT : 8;
  const bool read_res = P.a != real(0);
  const size_t base = (size_t(e0) * NF + fld) * Np + Tile::template first<ES>(lane);
  const real* qi = P.qin + base;
  real* qo = P.qout + base;
  real* re = P.res + base;
  const real* c = cols + Tile::template first<S>(lane);
  bool bad = false;
#pragma unroll
  for (int i0 = 0; i0 < Tile::IT; i0 += U) {
    typename Tile::Chunk q[U], r[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (Tile::has(lane, i0 + u, ne)) {
        q[u] = Tile::load(qi + Tile::template offset<ES>(i0 + u));
        if (read_res) r[u] = Tile::load(re + Tile::template offset<ES>(i0 + u));
      }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (Tile::has(lane, i0 + u, ne)) {
        const int gl = Tile::element(lane, i0 + u);
        if (!done(gl)) {
          const real h = dt(gl);
#pragma unroll
          for (int w = 0; w < Tile::W; ++w) {
            real x = h * c[Tile::template offset<S>(i0 + u) + w];
            if (read_res) x = fma(P.a, r[u].x[w], x);
            r[u].x[w] = x;
            q[u].x[w] = fma(P.b, x, q[u].x[w]);
            bad |= !isfinite(q[u].x[w]);
          }
          Tile::store(re + Tile::template offset<ES>(i0 + u), r[u]);
        }
        Tile::store(qo + Tile::template offset<ES>(i0 + u), q[u]);
      }
  }
  if (bad) atomicOr(P.status, 1u);
}

}  // namespace bbw
