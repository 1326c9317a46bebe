// bbw_tile.cuh -- the acoustic stage with one element per lane: a CTA of four
// warps takes 32 consecutive elements, one warp per field.
//
// Per tile and stage:
//   0  each warp stages its field into columns of shared memory
//      ([element][S], S odd: lanes on the same entry of their columns hit 32
//      banks); connectivity, geometry and the face tables once per CTA;
//   1  penalty fluxes, one face node per thread: own traces from the columns,
//      neighbour traces gathered from q_in (short runs of one element's field,
//      so a warp's gather covers few sectors);
//   2  one element per lane, one field per warp: every stencil index and weight
//      is an immediate, the degree N-1 combination (V1), the lift pyramids and
//      the right-hand side are registers (N_p <= 84: up to N = 6);
//   3  the p right-hand side is projected (bbw_project.cuh) in registers for
//      N <= 5, elsewhere by acoustic_project_kernel; RK update through the
//      columns.
//
// What bounded the team kernel was the shared-memory pipe and instruction
// issue (each stencil operand a shared load, each output a decoded table
// word), and in FP64 the double-precision pipe, on which the conversions of
// the integer weights cost as much as the products; here a stage needs about
// half the warp instructions per element and no conversions. What bounds it
// now (N = 5, 82,944 elements: 142 us against 219) is latency: 9.7 of 12 warps
// per SM at 0.33 instructions per scheduler and cycle, waiting for the staged
// field, the neighbour gather and the RK operands in turn and for instructions;
// L1 wavefronts 38 % of their peak, DRAM 21 %. Separate kernels for the fluxes and the fields (more warps in
// flight, the fluxes through L2) took 150 us.
// The operations and their order are those of stage_kernel (bbw_stage.cuh):
// the results are the same bits, so the two can be chosen by size.
#pragma once

#include "bbw_lane.cuh"

namespace bbw {

// kBracket: the p bracket goes to p's place in q_out, which nothing reads before
// the RK update writes it, for acoustic_project_kernel;
// kSpatial: the spatial operator alone (as the SP form of stage_kernel).
enum TileMode { kFused = 0, kBracket = 1, kSpatial = 2 };

// hide a value from the compiler, which would fold fma(1, x, y) and contract the
// addition with the product that x is
__device__ __forceinline__ void keep(float& x) { asm volatile("" : "+f"(x)); }
__device__ __forceinline__ void keep(double& x) { asm volatile("" : "+d"(x)); }
template <int N, typename real>
struct TileCfg {
  static constexpr int Np = np3(N), Nfp = np2(N), ITEMS = 4 * Nfp;
  static constexpr int S = (Np > np3(kMaxM) ? Np : np3(kMaxM)) | 1;  // columns also stage the c2 coefficients
  static constexpr int FS = 33;  // stride of the flux rows
  // columns [4][32 S] | fluxes [2][ITEMS][FS] | normals [4][nx, ny, nz, |f|/(2|D|)][32] | geometry [32][9] |
  // per-warp element scalars [4][32] | connectivity [32][4] | face tables (fidx [4 Nfp], nidx [24 Nfp], uint16)
  static constexpr int REALS = 4 * 32 * S + 2 * ITEMS * FS + 512 + 288 + 128;
  static constexpr int SMEM = (REALS * int(sizeof(real)) + 512 + 56 * Nfp + 15) / 16 * 16;
  static constexpr int THREADS = 128;
  // CTAs per SM that the registers have to allow. Stack of the fused kernel:
  // FP32 none but 40 bytes at N = M = 3; FP64 at N = 4 72 to 88 bytes at
  // M <= 1, 528 at M = 2, 1,240 at M = 3, and 360 at N = M = 3
  static constexpr int CTAS = sizeof(real) == 8 ? (N <= 4 ? 4 : 2) : N <= 2 ? 8 : N == 3 ? 6 : N == 4 ? 4 : N == 5 ? 3 : 2;
};

// whether all ne elements from e0 on have used up their step budgets (the whole warp)
template <typename real>
__device__ __forceinline__ bool all_finished(const StageParams<real>& P, int64_t e0, int ne, int lane) {
  if (!P.steps_group) return false;
  const int64_t step = P.step_dev ? *P.step_dev : P.step_host;
  return __all_sync(0xffffffffu, step >= P.steps_group[e0 + min(lane, ne - 1)]);
}

// q_out = q_in of a tile's ne elements, by the CTA. Out of line: inline, it cost
// the tiles that are not finished up to 1 % (and N = 3 eight bytes of stack).
template <int N, typename real>
__device__ __noinline__ void carry_tile(const real* qin, real* qout, int64_t e0, int ne) {
  constexpr int ES = 4 * np3(N);
  const uint4* src = reinterpret_cast<const uint4*>(qin + size_t(e0) * ES);
  uint4* dst = reinterpret_cast<uint4*>(qout + size_t(e0) * ES);
  constexpr int ALL = 32 * ES * int(sizeof(real)) / 16, U = ALL < 12 * 128 ? (ALL + 127) / 128 : 12;
  const int n = ALL / 32 * ne;
  for (int i0 = threadIdx.x; i0 < n; i0 += 128 * U) {  // few CTAs fit an SM: many loads in flight in each
    uint4 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + 128 * u < n) x[u] = src[i0 + 128 * u];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + 128 * u < n) dst[i0 + 128 * u] = x[u];
  }
}

template <int N, int M, typename real, int MODE>
__global__ void __launch_bounds__(128, TileCfg<N, real>::CTAS)
    acoustic_tile_kernel(const LaneStageParams<real> P, const uint32_t* __restrict__ face_tables) {
  using C = TileCfg<N, real>;
  using R = FieldRhs<N, real>;
  using Tile = WarpTile<np3(N), real>;
  constexpr int Np = C::Np, Nm1p = R::Nm1p, Nfp = C::Nfp, ITEMS = C::ITEMS, Mp = np3(M), S = C::S, ES = 4 * Np;
  extern __shared__ __align__(16) unsigned char smem[];
  real* COLS = reinterpret_cast<real*>(smem);
  real* FL = COLS + 4 * 32 * S;
  real* NRM = FL + 2 * ITEMS * C::FS;
  real* GEO = NRM + 512;
  real* SCAL = GEO + 288;
  int* CS = reinterpret_cast<int*>(SCAL + 128);
  uint32_t* TAB = reinterpret_cast<uint32_t*>(CS + 128);
  const uint16_t* fidx = reinterpret_cast<const uint16_t*>(TAB);
  const uint16_t* nidx = fidx + 4 * Nfp;
  const int tid = threadIdx.x, lane = tid % 32, fld = tid / 32;
  const int64_t e0 = int64_t(blockIdx.x) * 32;
  const int ne = P.G - e0 < 32 ? int(P.G - e0) : 32;
  bool oob = false;
  (void)oob;
  if constexpr (MODE != kSpatial) {
    // A tile of elements whose instances have all taken their steps carries
    // its state over (every warp tests the same elements): N = 5, 63,888 finished
    // elements beside 48 live ones take 36 us a stage, and 124 when they are live.
    if (all_finished(P, e0, ne, lane)) {
      carry_tile<N, real>(P.qin, P.qout, e0, ne);
      return;
    }
  }

  // ---- 0: columns, connectivity, geometry, tables ----
  CS[tid] = tid / 4 < ne ? P.conn[size_t(e0) * 4 + tid] : -1;
  for (int i = tid; i < 9 * ne; i += 128) GEO[i] = P.geom[size_t(e0) * 9 + i];
  for (int i = tid; i < 14 * Nfp; i += 128) TAB[i] = face_tables[i];
  real* cols = COLS + fld * 32 * S;  // this warp's columns
  const size_t base = size_t(e0) * ES + fld * Np;
  Tile::template stage<ES, S, (Tile::IT < 16 ? Tile::IT : 16)>(cols, P.qin + base, lane, ne);
  if constexpr (MODE != kSpatial)  // the RK update's operand
    if (P.a != real(0)) Tile::template prefetch<ES>(P.res + base, lane, ne);
  __syncthreads();

  // ---- 1: normals, then fluxes ----
  {
    const int e = tid / 4, f = tid % 4;
    real g[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const real g1 = GEO[e * 9 + d], g2 = GEO[e * 9 + 3 + d], g3 = GEO[e * 9 + 6 + d];
      g[d] = f == 0 ? -g1 - g2 - g3 : f == 1 ? g1 : f == 2 ? g2 : g3;
    }
    const real gx = g[0], gy = g[1], gz = g[2];
    const real gn = sqrt(norm2<TileShape<N, real>::V>(gx, gy, gz));
    const real inv = real(1) / gn;
    real* nr = NRM + f * 128 + e;
    nr[0] = -gx * inv;
    nr[32] = -gy * inv;
    nr[64] = -gz * inv;
    nr[96] = wmul(real(1.5), gn);
  }
  __syncthreads();
  {
    constexpr int U = N <= 2 ? 3 : N <= 4 ? 5 : 7;  // items in flight per thread (Nfp rounds of 128 items)
#pragma unroll 1
    for (int r0 = 0; r0 < Nfp; r0 += U) {
      real nb[U][4];
      int io[U], at[U], ee[U], ff[U], cc[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int idx = (r0 + u) * 128 + tid;
        const int e = idx / ITEMS, it = idx - e * ITEMS, f = it / Nfp, a = it - f * Nfp;
        ee[u] = r0 + u < Nfp ? e : 32;
        at[u] = it;
        ff[u] = f;
        if (ee[u] >= ne) continue;
        io[u] = fidx[it];
        const int c = CS[e * 4 + f];
        cc[u] = c;
        if constexpr (kChecked) {
          if (io[u] >= Np) {
            oob = true;
            io[u] = 0;
          }
        }
        if (c >= 0) {
          const int64_t k = int64_t(c >> 5);
          if constexpr (kChecked) {
            if (k >= P.G || (c & 7) >= 6) {
              oob = true;
              cc[u] = -1;
              continue;
            }
          }
          const int ni = nidx[(((c >> 3) & 3) * 6 + (c & 7)) * Nfp + a];
          if constexpr (kChecked) {
            if (ni >= Np) {
              oob = true;
              cc[u] = -1;
              continue;
            }
          }
          const real* src = P.qin + size_t(k) * ES + ni;
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4) nb[u][k4] = src[k4 * Np];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = ee[u], f = ff[u];
        if (e >= ne) continue;
        real own[4];
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) own[k4] = COLS[(k4 * 32 + e) * S + io[u]];
        if (cc[u] < 0) {  // p = 0 wall: mirror state
          nb[u][0] = -own[0];
          nb[u][1] = own[1];
          nb[u][2] = own[2];
          nb[u][3] = own[3];
        }
        const real* n = NRM + f * 128 + e;
        const real jp = nb[u][0] - own[0];
        real ndu = mul_rn(n[0], nb[u][1] - own[1]);
        ndu = fma(n[32], nb[u][2] - own[2], ndu);
        ndu = fma(n[64], nb[u][3] - own[3], ndu);
        FL[at[u] * C::FS + e] = mul_rn(n[96], penalty(P.tau_p, jp, ndu));
        FL[(ITEMS + at[u]) * C::FS + e] = mul_rn(n[96], penalty(P.tau_u, ndu, jp));
      }
    }
  }
  __syncthreads();

  // ---- 2: right-hand side of this warp's field, one element per lane ----
  real r[Np];
  real gm[4][3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int m = 1; m < 4; ++m) gm[m][d] = GEO[lane * 9 + 3 * (m - 1) + d];
    gm[0][d] = -gm[1][d] - gm[2][d] - gm[3][d];
  }
  {
    real v1[Nm1p];
#pragma unroll
    for (int i = 0; i < Nm1p; ++i) v1[i] = real(0);
    if (fld == 0) {
      const real* u = COLS + (32 + lane) * S;  // u, v, w: -div
      R::add_div(v1, u, u + 32 * S, u + 64 * S, gm);
    } else {
      real w[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) w[m] = -pick(gm[m], fld - 1);
      R::add_term(v1, COLS + lane * S, w);  // p: -grad
    }
    __syncthreads();  // the columns are free
    R::elevate_all(v1, r);
  }
  {
    const real* fl = FL + (fld == 0 ? 0 : ITEMS * C::FS) + lane;
    static_for<0, 4>([&](auto f_) BBW_ALWAYS_INLINE {
      constexpr int f = decltype(f_)::value;
      real F[Nfp];
#pragma unroll
      for (int i = 0; i < Nfp; ++i) F[i] = fl[(f * Nfp + i) * C::FS];
      real w = fld == 0 ? real(1) : NRM[f * 128 + (fld - 1) * 32 + lane];
      keep(w);
      R::template lift<f>(r, F, w);
    });
  }

  // ---- 3: sources, projection, RK ----
  real* col = cols + lane * S;
  if (fld == 0 && (P.n_src_groups > 0 || (MODE != kSpatial && P.vout))) {
    // this lane's entry in the ascending list of source elements, if any; the
    // warp adds each found source vector together, in the columns
    const int64_t el = e0 + min(lane, ne - 1);
    int64_t lo = 0, hi = P.n_src_groups;
    while (lo < hi) {
      const int64_t mid = (lo + hi) / 2;
      if (P.src_groups[mid] < el)
        lo = mid + 1;
      else
        hi = mid;
    }
    const int sd = lane < ne && lo < P.n_src_groups && P.src_groups[lo] == el ? P.src_slots[lo] : -1;
    const real amp = sd >= 0 ? real(stage_amplitude(P, sd)) : real(0);
    unsigned has = __ballot_sync(0xffffffffu, sd >= 0);
    if (has || (MODE != kSpatial && P.vout)) {
      put_column(col, r);
      __syncwarp();
      while (has) {
        const int src = __ffs(int(has)) - 1;
        has &= has - 1;
        const int s = __shfl_sync(0xffffffffu, sd, src);
        const real a = __shfl_sync(0xffffffffu, amp, src);
        for (int i = lane; i < Np; i += 32) cols[src * S + i] = fma(a, P.src_vec[size_t(s) * Np + i], cols[src * S + i]);
      }
      __syncwarp();
      if (MODE != kSpatial && P.vout) Tile::template unstage<Np, S>(cols, P.vout + size_t(e0) * Np, lane, ne);
#pragma unroll
      for (int i = 0; i < Np; ++i) r[i] = col[i];
      __syncwarp();
    }
  }
  const int64_t step_now = P.step_dev ? *P.step_dev : P.step_host;
  auto dt = [&](int gl) { return P.dt_group ? P.dt_group[e0 + gl] : P.dt; };
  auto done = [&](int gl) { return P.steps_group && step_now >= P.steps_group[e0 + gl]; };
  if constexpr (MODE == kSpatial) {
    put_column(col, r);
    if (P.accumulate) {
      // q_out -= dt |D| rhs, |D| = 1 / (6 det[grad lambda_1; grad lambda_2; grad lambda_3])
      const real a1 = gm[1][0], a2 = gm[1][1], a3 = gm[1][2], b1 = gm[2][0], b2 = gm[2][1], b3 = gm[2][2],
                 c1 = gm[3][0], c2v = gm[3][1], c3 = gm[3][2];
      const real det = a1 * (b2 * c3 - b3 * c2v) - a2 * (b1 * c3 - b3 * c1) + a3 * (b1 * c2v - b2 * c1);
      SCAL[tid] = -(dt(min(lane, ne - 1)) / (real(6) * det));
      __syncwarp();
      constexpr int U = Tile::IT < 8 ? Tile::IT : 8;
      real* qo = P.qout + base + Tile::template first<ES>(lane);
      const real* c = cols + Tile::template first<S>(lane);
#pragma unroll
      for (int i0 = 0; i0 < Tile::IT; i0 += U) {
        typename Tile::Chunk q[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (Tile::has(lane, i0 + u, ne)) q[u] = Tile::load(qo + Tile::template offset<ES>(i0 + u));
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (Tile::has(lane, i0 + u, ne)) {
            const real h = SCAL[fld * 32 + Tile::element(lane, i0 + u)];
#pragma unroll
            for (int w = 0; w < Tile::W; ++w) q[u].x[w] = fma(h, c[Tile::template offset<S>(i0 + u) + w], q[u].x[w]);
            Tile::store(qo + Tile::template offset<ES>(i0 + u), q[u]);
          }
      }
    } else {
      __syncwarp();
      Tile::template unstage<ES, S>(cols, P.qout + base, lane, ne);
    }
  } else {
    if (fld == 0) {
      if constexpr (MODE == kFused) {
        typename WeightTile<M, real>::Held wt;
        WeightTile<M, real>::template hold<Mp>(wt, P.c2 + size_t(e0) * Mp, lane, ne);
        real wc[Mp];
        lane_weight<M, S>(wt, cols, lane, ne, real(1), wc);
        to_power<N, real>(r);
        Projector<N, M, real, true>::run(r, r, static_cast<real*>(nullptr), wc, P.cs);
      } else {
        put_column(col, r);
        __syncwarp();
        Tile::template unstage<ES, S>(cols, P.qout + base, lane, ne);
      }
    }
    if (MODE == kFused || fld != 0) {
      put_column(col, r);
      __syncwarp();
      lane_rk<N, 4, real, S>(P, cols, e0, ne, lane, fld, dt, done);
    }
  }
  if constexpr (kChecked) {
    if (oob) atomicOr(P.status, 2u);
  }
}

// Projection and RK update of p from the bracket in q_out (kBracket), which the
// warp reads whole before it writes p there: one warp per 32 elements,
// blockDim.x / 32 warps per CTA.
template <int N, int M, typename real>
__global__ void __launch_bounds__(ProjectShape<N, M, real>::THREADS) acoustic_project_kernel(const LaneStageParams<real> P) {
  using C = ProjectShape<N, M, real>;
  using Tile = WarpTile<np3(N), real>;
  using Pr = Projector<N, M, real, true>;
  constexpr int Np = np3(N), Mp = np3(M), S = C::S;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  real* cols = reinterpret_cast<real*>(smem + warp * C::WARP_BYTES);
  const int64_t e0 = (int64_t(blockIdx.x) * (blockDim.x / 32) + warp) * 32;
  const int ne = P.G - e0 < 32 ? int(P.G - e0) : 32;
  if (ne <= 0) return;  // warps are independent
  const int64_t step_now = P.step_dev ? *P.step_dev : P.step_host;
  if (all_finished(P, e0, ne, lane)) return;  // the tile kernel has copied p
  typename WeightTile<M, real>::Held wt;
  WeightTile<M, real>::template hold<Mp>(wt, P.c2 + size_t(e0) * Mp, lane, ne);
  Tile::template prefetch<4 * Np>(P.qin + size_t(e0) * 4 * Np, lane, ne);
  if (P.a != real(0)) Tile::template prefetch<4 * Np>(P.res + size_t(e0) * 4 * Np, lane, ne);
  real wc[Mp];
  lane_weight<M, S>(wt, cols, lane, ne, real(1), wc);
  Tile::template stage<4 * Np, S, (Tile::IT < 28 ? Tile::IT : 28)>(cols, P.qout + size_t(e0) * 4 * Np, lane, ne);
  __syncwarp();
  real* col = cols + lane * S;
  if constexpr (N > Pr::RD) {
    to_power<N, real>(col);
    Pr::run(col, col, col, wc, P.cs);
  } else {
    real r[Np];
#pragma unroll
    for (int i = 0; i < Np; ++i) r[i] = col[i];
    to_power<N, real>(r);
    Pr::run(r, col, col, wc, P.cs);
  }
  __syncwarp();
  lane_rk<N, 4, real, S>(
      P, cols, e0, ne, lane, 0, [&](int gl) { return P.dt_group ? P.dt_group[e0 + gl] : P.dt; },
      [&](int gl) { return P.steps_group && step_now >= P.steps_group[e0 + gl]; });
}

// The adjoint stage's update before its spatial operator (LaneAdjPreParams), one
// warp per 32 elements and field (blockIdx.x % 4).
template <int N, int M, typename real>
__global__ void __launch_bounds__(ProjectShape<N, M, real>::THREADS) lane_adj_pre_kernel(const LaneAdjPreParams<real> P) {
  using C = ProjectShape<N, M, real>;
  using Tile = WarpTile<np3(N), real>;
  using Pr = Projector<N, M, real, true>;
  constexpr int Np = np3(N), Mp = np3(M), S = C::S, ES = 4 * Np;
  constexpr int U = Tile::IT < 8 ? Tile::IT : 8;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  real* cols = reinterpret_cast<real*>(smem + warp * C::WARP_BYTES);
  const int64_t e0 = (int64_t(blockIdx.x / 4) * (blockDim.x / 32) + warp) * 32;
  const int ne = P.G - e0 < 32 ? int(P.G - e0) : 32;
  if (ne <= 0) return;
  const int fld = blockIdx.x % 4;
  const size_t base = size_t(e0) * ES + fld * Np;
  real iv;  // 1 / |D| = 6 det[grad lambda_1; grad lambda_2; grad lambda_3]
  {
    const real* g = P.geom + size_t(e0 + min(lane, ne - 1)) * 9;
    const real a1 = g[0], a2 = g[1], a3 = g[2], b1 = g[3], b2 = g[4], b3 = g[5], c1 = g[6], c2v = g[7], c3 = g[8];
    iv = real(6) * (a1 * (b2 * c3 - b3 * c2v) - a2 * (b1 * c3 - b3 * c1) + a3 * (b1 * c2v - b2 * c1));
  }
  real wc[Mp];
  if (fld == 0) {
    typename WeightTile<M, real>::Held wt;
    WeightTile<M, real>::template hold<Mp>(wt, P.c2 + size_t(e0) * Mp, lane, ne);
    lane_weight<M, S>(wt, cols, lane, ne, real(1), wc);
  }
  // rho_t = a rho + b kap, into the columns
  {
    real* rho = P.rho + base + Tile::template first<ES>(lane);
    const real* kap = P.kap + base + Tile::template first<ES>(lane);
    real* c = cols + Tile::template first<S>(lane);
#pragma unroll
    for (int i0 = 0; i0 < Tile::IT; i0 += U) {
      typename Tile::Chunk r[U], k[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (Tile::has(lane, i0 + u, ne)) {
          r[u] = Tile::load(rho + Tile::template offset<ES>(i0 + u));
          k[u] = Tile::load(kap + Tile::template offset<ES>(i0 + u));
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (Tile::has(lane, i0 + u, ne)) {
#pragma unroll
          for (int w = 0; w < Tile::W; ++w) {
            const real bk = mul_rn(P.b, k[u].x[w]);
            r[u].x[w] = fma(P.a, r[u].x[w], bk);
            c[Tile::template offset<S>(i0 + u) + w] = r[u].x[w];
          }
          Tile::store(rho + Tile::template offset<ES>(i0 + u), r[u]);
        }
    }
  }
  __syncwarp();
  real* col = cols + lane * S;
  if (fld == 0) {
    if constexpr (N > Pr::RD) {
      to_power<N, real>(col);
      Pr::run(col, col, col, wc, P.cs);
    } else {
      real r[Np];
#pragma unroll
      for (int i = 0; i < Np; ++i) r[i] = col[i];
      to_power<N, real>(r);
      Pr::run(r, col, col, wc, P.cs);
    }
  }
#pragma unroll 8
  for (int i = 0; i < Np; ++i) col[i] *= iv;
  __syncwarp();
  Tile::template unstage<ES, S>(cols, P.y + base, lane, ne);
}

}  // namespace bbw
