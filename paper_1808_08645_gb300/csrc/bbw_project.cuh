// bbw_project.cuh -- the weight-adjusted update of Sec. 5 for one element per
// thread: u = P^{N+M}_N (c r) with every stencil index a compile-time
// constant.
//
// A thread owns one element. The sparse Bernstein operators then need no
// index words and no exchange between lanes: a level of the telescoped
// projection is a register array, or (degrees above kRegDegree) a column of
// shared memory that only this thread touches. Columns are [element][stride]
// with an odd stride, so the 32 lanes of a warp, which all access the same
// entry of their columns, hit 32 different banks.
//
// EXACT = false runs on power coefficients a_alpha / alpha!, in which
//   the product of Eq. (11) is a plain convolution,
//   a one-degree reduction is  (D h)_b = sum_m (b_m + 1)^2 h_{b + e_m},
//   a one-degree elevation is  (s w)_g = sum_m w_{g - e_m}  (no weights),
// so a reduction costs 4 FMAs with immediate weights per output and an
// elevation 4 additions. The factors 1/n of the Bernstein operators are
// folded into the constants c_j (projection_scale below). Each D is scaled by
// the power of two nearest below 1/n^2 (exact), which keeps every level at
// the magnitude of its input.
//
// EXACT = true performs the operations of the team kernels' wadg_group one by
// one, in its order (product of factorial-scaled coefficients, Bernstein
// reductions and elevations), so that its results are the same bits; it costs
// one more multiplication per reduction and two more operations per elevation.
// (Of degree 1 the team kernels' w = c v + (1/n) E w is one FMA; so it is here.)
#pragma once

#include <type_traits>
#include <utility>

#include "bbw_common.h"

#define BBW_ALWAYS_INLINE __attribute__((always_inline))

namespace bbw {

template <int B, int E, typename F>
BBW_HD void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}
// B, B - 1, ..., E
template <int B, int E, typename F>
BBW_HD void static_for_down(F&& f) {
  if constexpr (B >= E) {
    f(std::integral_constant<int, B>{});
    static_for_down<B - 1, E>(f);
  }
}

// w v + x for a weight that is a constant after inlining. fma(+-1, v, x) would be
// folded to an addition, which may then be contracted with the product that x
// is: an FMA fewer, but other bits than the table-driven kernels'.
template <typename real>
BBW_HD real wfma(real w, real v, real x) {
#ifdef __CUDA_ARCH__
  if (w == real(1)) {
    if constexpr (sizeof(real) == 4)
      return __fadd_rn(v, x);
    else
      return __dadd_rn(v, x);
  }
  if (w == real(-1)) {
    if constexpr (sizeof(real) == 4)
      return __fsub_rn(x, v);
    else
      return __dsub_rn(x, v);
  }
#endif
  return fma(w, v, x);
}

// w v, rounded on its own (2 v would become v + v, which may be contracted with
// the product that v is)
template <typename real>
BBW_HD real wmul(real w, real v) {
#ifdef __CUDA_ARCH__
  if constexpr (sizeof(real) == 4)
    return __fmul_rn(w, v);
  else
    return __dmul_rn(w, v);
#else
  return w * v;
#endif
}

BBW_HD constexpr double cfact(int n) {
  double f = 1.0;
  for (int i = 2; i <= n; ++i) f *= i;
  return f;
}
// power-of-two scale of the reduction from degree n: 2^-ceil(2 log2 n)
BBW_HD constexpr double reduce_scale(int n) {
  double s = 1.0;
  while (s * n * n > 1.0) s *= 0.5;
  return s;
}

// c_j of Theorem 5.3 -> the constants of the power-basis sweeps, for
// W_j = c'_j V_j + s W_{j+1}: the 1/n of the elevations give (N-j)!/N!, those
// of the reductions (N-j)!/(N+M)!, the product 1/C(N+M,N), and the scales of
// the reductions are divided out.
template <int N, int M>
inline void projection_scale(const double* cj, double* out) {
  double scale = 1.0;  // product of the reductions' scales so far
  for (int n = N + M; n > N; --n) scale *= reduce_scale(n);
  const double binom = cfact(N + M) / (cfact(N) * cfact(M));
  for (int j = 0; j <= N; ++j) {
    out[j] = cj[j] * cfact(N - j) / cfact(N) * cfact(N - j) / cfact(N + M) / binom / scale;
    scale *= reduce_scale(N - j);
  }
}

// offset of row (k, l) in the degree-n lattice
BBW_HD constexpr int row3(int n, int k, int l) { return idx3(n, 0, k, l); }

BBW_HD constexpr double cbinom(int n, int k) { return cfact(n) / (cfact(k) * cfact(n - k)); }

template <int N, int M, typename real, bool EXACT = false>
struct Projector {
  static constexpr int Np = np3(N), Mp = np3(M);
  // levels of degree <= kRegDegree are registers (sum np3(0..5) = 126), the
  // ones above entries of the column
  static constexpr int kRegDegree = sizeof(real) == 4 ? 5 : 4;
  static constexpr int RD = N < kRegDegree ? N : kRegDegree;
  static constexpr int REGS = off3(RD + 1);
  // column entries: levels of degree N, N-1, ..., RD+1 (at least the N_p of the input and output)
  static constexpr int COL = N > RD ? off3(N + 1) - off3(RD + 1) : Np;
  BBW_HD static constexpr int col_base(int d) { return off3(N + 1) - off3(d + 1); }  // of degree d > RD

  // one plane (degree P lattice in j, k) of a reduction from degree n: cur the
  // input plane l (degree P + 1), nxt the input plane l + 1 (degree P)
  template <int n, int l, typename Cur, typename Nxt, typename Out>
  BBW_HD static void reduce_plane(const Cur& cur, const Nxt& nxt, Out& out) {
    constexpr int P = n - 1 - l;
    static_for<0, P + 1>([&](auto kk) BBW_ALWAYS_INLINE {
      constexpr int k = decltype(kk)::value;
#pragma unroll
      for (int j = 0; j <= P - k; ++j) {
        real x = wmul(reduce_weight(n, P - j - k + 1), cur[idx2(P + 1, j, k)]);
        x = wfma(reduce_weight(n, j + 1), cur[idx2(P + 1, j + 1, k)], x);
        x = wfma(reduce_weight(n, k + 1), cur[idx2(P + 1, j, k + 1)], x);
        x = wfma(reduce_weight(n, l + 1), nxt[idx2(P, j, k)], x);
        if constexpr (EXACT) x = wmul(real(1) / real(n), x);
        out[idx2(P, j, k)] = x;
      }
    });
  }

  // row (k, l) of the degree N+M product: h_g = sum_b c_b r_{g-b}, r = src
  template <int k, int l, typename Src>
  BBW_HD static void product_row(const Src& src, const real (&c)[Mp], real (&h)[N + M + 1]) {
    constexpr int L = N + M - l - k + 1;
#pragma unroll
    for (int j = 0; j < L; ++j) h[j] = real(0);
    static_for<0, M + 1>([&](auto bl_) BBW_ALWAYS_INLINE {
      static_for<0, M + 1>([&](auto bk_) BBW_ALWAYS_INLINE {
        constexpr int bl = decltype(bl_)::value, bk = decltype(bk_)::value;
        constexpr int rl = l - bl, rk = k - bk;  // row of r
        if constexpr (bl + bk <= M && rl >= 0 && rk >= 0 && rl + rk <= N) {
          real r[N + 1];
#pragma unroll
          for (int j = 0; j <= N - rl - rk; ++j) r[j] = src[row3(N, rk, rl) + j];
#pragma unroll
          for (int bj = 0; bj <= M - bl - bk; ++bj)
#pragma unroll
            for (int j = 0; j <= N - rl - rk; ++j) h[j + bj] = fma(c[idx3(M, bj, bk, bl)], r[j], h[j + bj]);
        }
      });
    });
    if constexpr (EXACT)
#pragma unroll
      for (int j = 0; j < L; ++j)
        h[j] = wmul(real(cfact(L - 1 - j) * cfact(j) * cfact(k) * cfact(l) / cbinom(N + M, N)), h[j]);
  }
  // weight of an input of a reduction from degree n with b_m + 1 = b
  BBW_HD static constexpr real reduce_weight(int n, int b) {
    return EXACT ? real(b) : real(reduce_scale(n) * b * b);
  }

  // product, the M reductions and so the first level v_0, from the top plane
  // and within a plane from the top row down: row (k, l) of a reduction needs
  // rows (k, l), (k + 1, l) and (k, l + 1) of its input. plane[m] holds plane
  // l + 1 of level m (degree N + M - m).
  // put(k, l, row) receives the rows of v_0; row (k, l) of r is not read after
  // that, so v_0 may overwrite r.
  template <typename Src, typename Put>
  BBW_HD static void product_reduce(const Src& src, const real (&c)[Mp], Put&& put) {
    real plane[M > 0 ? M : 1][np2(N + M)];
    static_for_down<N + M, 0>([&](auto l_) BBW_ALWAYS_INLINE {
      constexpr int l = decltype(l_)::value;
      real next[M > 0 ? M : 1][np2(N + M)];
      real above[M > 0 ? M : 1][N + M + 1];  // row k + 1 of level m
      static_for_down<N + M - l, 0>([&](auto k_) BBW_ALWAYS_INLINE {
        constexpr int k = decltype(k_)::value;
        real row[M + 1][N + M + 1];
        product_row<k, l>(src, c, row[0]);
        static_for<0, M>([&](auto m_) BBW_ALWAYS_INLINE {
          constexpr int m = decltype(m_)::value, n = N + M - m, P = n - l;  // input degree, its plane's degree
          if constexpr (k <= P) {
#pragma unroll
            for (int j = 0; j < P - k; ++j) {
              real x = wmul(reduce_weight(n, P - j - k), row[m][j]);
              x = wfma(reduce_weight(n, j + 1), row[m][j + 1], x);
              x = wfma(reduce_weight(n, k + 1), above[m][j], x);
              x = wfma(reduce_weight(n, l + 1), plane[m][idx2(P - 1, j, k)], x);
              if constexpr (EXACT) x = wmul(real(1) / real(n), x);
              row[m + 1][j] = x;
            }
          }
        });
        // (row k of plane l + 1 is dead from here on, so the two planes share registers)
        static_for<0, M>([&](auto m_) BBW_ALWAYS_INLINE {
          constexpr int m = decltype(m_)::value, P = N + M - m - l;
          if constexpr (k <= P) {
#pragma unroll
            for (int j = 0; j <= P - k; ++j) {
              above[m][j] = row[m][j];
              next[m][idx2(P, j, k)] = row[m][j];
            }
          }
        });
        if constexpr (k <= N - l) put(k_, l_, row[M]);
      });
      static_for<0, M>([&](auto m_) BBW_ALWAYS_INLINE {
        constexpr int m = decltype(m_)::value, P = N + M - m - l;
        if constexpr (P >= 0)
#pragma unroll
          for (int i = 0; i < np2(P); ++i) plane[m][i] = next[m][i];
      });
    });
  }

  // dst = P^{N+M}_N (c src): src the coefficients r_alpha / alpha!, dst
  // the Bernstein coefficients of the result (arrays in registers or the
  // column; they may be the same); c the power coefficients of the weight, cs
  // the constants of projection_scale. col: the thread's column of COL entries,
  // used (and then src itself) only where N > RD. EXACT: cs are the c_j.
  template <typename Src, typename Dst>
  BBW_HD static void run(const Src& src, Dst&& dst, real* col, const real (&c)[Mp], const real* cs) {
    real v[REGS];  // degree d <= RD at off3(d)
    // v_0
    product_reduce(src, c, [&](auto k_, auto l_, const auto& row) BBW_ALWAYS_INLINE {
      constexpr int k = decltype(k_)::value, l = decltype(l_)::value;
#pragma unroll
      for (int j = 0; j <= N - l - k; ++j) {
        if constexpr (N > RD)
          col[row3(N, k, l) + j] = row[j];
        else
          v[off3(N) + row3(N, k, l) + j] = row[j];
      }
    });
    // downward sweep
    static_for_down<N, 1>([&](auto n_) BBW_ALWAYS_INLINE {
      constexpr int n = decltype(n_)::value;  // degree n -> n - 1
      real nxt[np2(n)];
      static_for_down<n, 0>([&](auto l_) BBW_ALWAYS_INLINE {
        constexpr int l = decltype(l_)::value;
        constexpr int o = np3(n) - np3(n - l);
        real cur[np2(n)];
#pragma unroll
        for (int i = 0; i < np2(n - l); ++i) {
          if constexpr (n > RD)
            cur[i] = col[col_base(n) + o + i];
          else
            cur[i] = v[off3(n) + o + i];
        }
        if constexpr (l <= n - 1) {
          real out[np2(n)];
          reduce_plane<n, l>(cur, nxt, out);
          constexpr int oo = np3(n - 1) - np3(n - 1 - l);
#pragma unroll
          for (int i = 0; i < np2(n - 1 - l); ++i) {
            if constexpr (n - 1 > RD)
              col[col_base(n - 1) + oo + i] = out[i];
            else
              v[off3(n - 1) + oo + i] = out[i];
          }
        }
#pragma unroll
        for (int i = 0; i < np2(n - l); ++i) nxt[i] = cur[i];
      });
    });
    // upward sweep, in place: degree d becomes c_{N-d} v + s w
    v[0] = wmul(cs[N], v[0]);
    static_for<1, N + 1>([&](auto d_) BBW_ALWAYS_INLINE {
      constexpr int d = decltype(d_)::value;
      const real cd = cs[N - d];
      real below[np2(d)];  // plane l - 1 of the level below (degree d - 1)
      static_for<0, d + 1>([&](auto l_) BBW_ALWAYS_INLINE {
        constexpr int l = decltype(l_)::value;
        constexpr int P = d - l;
        constexpr int o = np3(d) - np3(d - l);
        real same[np2(d)];  // plane l of the level below
        if constexpr (l <= d - 1) {
          constexpr int ob = np3(d - 1) - np3(d - 1 - l);
#pragma unroll
          for (int i = 0; i < np2(d - 1 - l); ++i) {
            if constexpr (d - 1 > RD)
              same[i] = col[col_base(d - 1) + ob + i];
            else
              same[i] = v[off3(d - 1) + ob + i];
          }
        }
        static_for<0, P + 1>([&](auto k_) BBW_ALWAYS_INLINE {
          constexpr int k = decltype(k_)::value;
#pragma unroll
          for (int j = 0; j <= P - k; ++j) {
            const int i = o + idx2(P, j, k);
            real vd;
            if constexpr (d > RD)
              vd = col[col_base(d) + i];
            else
              vd = v[off3(d) + i];
            real x;
            if constexpr (EXACT) {
              real a = real(0);
              if (j + k < P) a = wmul(real(P - j - k), same[idx2(P - 1, j, k)]);
              if (j > 0) a = j + k < P ? wfma(real(j), same[idx2(P - 1, j - 1, k)], a) : wmul(real(j), same[idx2(P - 1, j - 1, k)]);
              if (k > 0) a = j > 0 || j + k < P ? wfma(real(k), same[idx2(P - 1, j, k - 1)], a) : wmul(real(k), same[idx2(P - 1, j, k - 1)]);
              if (l > 0) a = P > 0 ? wfma(real(l), below[idx2(P, j, k)], a) : wmul(real(l), below[idx2(P, j, k)]);
              if constexpr (d == 1)
                x = fma(cd, vd, a);
              else
                x = wfma(real(1) / real(d), a, wmul(cd, vd));
            } else {
              x = cd * vd;
              if (j + k < P) x += same[idx2(P - 1, j, k)];
              if (j > 0) x += same[idx2(P - 1, j - 1, k)];
              if (k > 0) x += same[idx2(P - 1, j, k - 1)];
              if (l > 0) x += below[idx2(P, j, k)];
              if constexpr (d == N) x *= real(cfact(j) * cfact(k) * cfact(l) * cfact(P - j - k));
            }
            if constexpr (d == N)
              dst[i] = x;
            else if constexpr (d > RD)
              col[col_base(d) + i] = x;
            else
              v[off3(d) + i] = x;
          }
        });
        if constexpr (l <= d - 1)
#pragma unroll
          for (int i = 0; i < np2(d - 1 - l); ++i) below[i] = same[i];
      });
    });
  }
};

}  // namespace bbw
