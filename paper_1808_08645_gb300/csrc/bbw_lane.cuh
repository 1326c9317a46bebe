// bbw_lane.cuh -- the spatial operator and the RK update with one element per
// lane: the parts shared by the acoustic tile kernel (bbw_tile.cuh) and the
// elastic field tasks (bbw_elastic_lane.cuh).
// A field's right-hand side is  E sum_t D_{d_t} f_t + sum_face L^f F: with the
// element in a lane every stencil index and weight is an immediate, the degree
// N-1 combination (V1), the lift pyramid and the right-hand side are registers
// (N_p <= 120: up to N = 7), and shared memory only transposes between the
// lanes' elements and contiguous global accesses.
#pragma once

#include "bbw_project.cuh"
#include "bbw_stage.cuh"
#include "bbw_warp_tile.cuh"

namespace bbw {

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
