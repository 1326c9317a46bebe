// bbw_elastic_inst.cuh -- instantiate the elastic stage kernel for one
// degree. Included by bbw_elastic_n<N>.cu with BBW_N defined.
#pragma once

#include <cstddef>

#include "bbw_elastic.cuh"
#include "bbw_elastic_lane.cuh"
#include "bbw_elastic_ops.h"

#ifndef BBW_N
#error "define BBW_N before including bbw_elastic_inst.cuh"
#endif

namespace bbw {
namespace {

constexpr int kN = BBW_N;

template <typename real>
using EShape = ElasticShape<kN, real>;

template <int M, typename real>
constexpr int kEGC = elastic_cta_groups<kN, M, real, EShape<real>::T, EShape<real>::V>();

template <int M, typename real>
using ECfg = ElasticCfg<kN, M, real, EShape<real>::T, EShape<real>::V, kEGC<M, real>>;

template <int M, typename real>
constexpr auto elastic_fn() {
  return elastic_stage_kernel<kN, M, real, EShape<real>::T, EShape<real>::V, kEGC<M, real>>;
}

template <typename F>
auto edispatch(int M, bool dbl, F&& f) {
  switch (M) {
    case 0: return dbl ? f.template operator()<0, double>() : f.template operator()<0, float>();
    case 1: return dbl ? f.template operator()<1, double>() : f.template operator()<1, float>();
    case 2: return dbl ? f.template operator()<2, double>() : f.template operator()<2, float>();
    default: return dbl ? f.template operator()<3, double>() : f.template operator()<3, float>();
  }
}

// FP32, N = 2..7: the kernels with one element per lane for solvers of at
// least kELaneMin elements, otherwise the team kernel: below that the lane
// kernels' two or three more launches and their few, long warps cost more than
// they save. The team kernel's time jumps where an SM gets one more CTA (its
// elements x 152 SMs: N = 2, 3 every 2,432 elements a CTA, up to four CTAs;
// N = 4 3,648, N = 5 and 6 2,432, N = 7 1,672) and the lane kernels' rises
// evenly, so the constants lie behind the step from which on they are nowhere
// slower (every 3.5 % of size measured, M = 0..3; lane / team before and behind):
//   N = 2  M = 0: 1.54 below 9,728, 1.05 to 1.09 up to 19,456, 0.88 above; M = 1: 1.40, 0.96;
//          M = 2: 1.22, 0.76; M = 3: 1.03 below 4,864, 0.95 up to 9,728, 0.54 above
//   N = 3  M = 0: 1.32 below 7,296, 0.92; M = 1: 1.20, 0.84; M = 2, 3: 1.4 and 1.03 below 4,864, 0.82 and 0.58
//   N = 4  1.06 to 1.7 below 3,648, 0.58 to 0.92; M = 0: 1.00 to 1.11 up to 7,296, 0.79 above
//   N = 5  0.91 to 1.29 below 2,432, 0.50 to 0.80       N = 6  0.98 to 1.5 below 2,432, 0.55 to 0.87;
//          M = 0 1.02 between 4,086 and 4,864           N = 7  1.4 to 1.66 below 1,672, 0.75 to 0.90
// The projections are fused up to N = 5, where their levels fit the register file.
template <typename real>
constexpr bool kELane = sizeof(real) == 4 && kN >= 2 && kN <= 7;
template <int M>
constexpr int64_t kELaneMin = kN == 2   ? (M == 0 ? 19500 : M == 3 ? 7000 : 9800)
                              : kN == 3 ? (M <= 1 ? 7300 : 7000)
                              : kN == 4 ? (M == 0 ? 7300 : 4000)
                              : kN == 5 ? 3000
                              : kN == 6 ? (M == 0 ? 4900 : 4000)
                                        : 1700;
constexpr bool kEFused = kN <= 5;
template <int M, typename real>
using EFCfg = FieldShape<kN, real>;
template <int M, typename real, bool TRACE>
constexpr auto efield_fn() {
  return elastic_field_kernel<kN, kEFused ? M : 0, real, kEFused, TRACE>;
}
template <int M, typename real>
using EPCfg = ProjectShape<kN, M, real>;

cudaError_t eprepare(int M, bool dbl, int* per_sm) {
  return edispatch(M, dbl, [&]<int MM, typename real>() {
    using C = ECfg<MM, real>;
    auto allow = [](auto k, int bytes) {
      return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    auto k = elastic_fn<MM, real>();
    cudaError_t err = allow(k, C::SMEM);
    if constexpr (kELane<real>) {
      if (err == cudaSuccess) err = allow(elastic_flux_kernel<kN, real>, flux_smem<kN, real>());
      if (err == cudaSuccess) err = allow(efield_fn<MM, real, true>(), EFCfg<MM, real>::SMEM);
      if constexpr (kEFused) {
        if (err == cudaSuccess) err = allow(efield_fn<MM, real, false>(), EFCfg<MM, real>::SMEM);
      } else {
        if (err == cudaSuccess) err = allow(elastic_project_kernel<kN, MM, real, true>, EPCfg<MM, real>::SMEM);
        if (err == cudaSuccess) err = allow(elastic_project_kernel<kN, MM, real, false>, EPCfg<MM, real>::SMEM);
      }
    }
    if (err != cudaSuccess) return err;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k, C::THREADS, C::SMEM);
  });
}

cudaError_t elaunch(int M, bool dbl, const void* params, int grid, cudaStream_t s) {
  return edispatch(M, dbl, [&]<int MM, typename real>() {
    using C = ECfg<MM, real>;
    const auto& P = *static_cast<const LaneElasticParams<real>*>(params);
    if constexpr (kELane<real>) {
      if (P.flux) {
        using Tab = Tables<kN, MM, real>;
        const char* t = static_cast<const char*>(P.tables);
        elastic_flux_kernel<kN, real>
            <<<unsigned((P.G + kFluxTile<kN> - 1) / kFluxTile<kN>), kFluxThreads, flux_smem<kN, real>(), s>>>(
                P, reinterpret_cast<const uint16_t*>(t + offsetof(Tab, fidx)),
                reinterpret_cast<const uint16_t*>(t + offsetof(Tab, nidx)));
        auto blocks = [&](int warps) { return unsigned((P.G + 32 * warps - 1) / (32 * warps)); };
        using FC = EFCfg<MM, real>;
        const unsigned nb = blocks(FC::WARPS);
        efield_fn<MM, real, true>()<<<nb * (kEFused ? 4 : 10), FC::THREADS, FC::SMEM, s>>>(P);
        if constexpr (kEFused) {
          efield_fn<MM, real, false>()<<<nb * 6, FC::THREADS, FC::SMEM, s>>>(P);
        } else {
          using PC = EPCfg<MM, real>;
          const unsigned np = blocks(PC::WARPS);
          elastic_project_kernel<kN, MM, real, true><<<np * 4, PC::THREADS, PC::SMEM, s>>>(P);
          elastic_project_kernel<kN, MM, real, false><<<np * 6, PC::THREADS, PC::SMEM, s>>>(P);
        }
        return cudaGetLastError();
      }
    }
    elastic_fn<MM, real>()<<<grid, C::THREADS, C::SMEM, s>>>(P);
    return cudaGetLastError();
  });
}

int64_t elane_min(int M, bool dbl) {
  return edispatch(M, dbl, [&]<int MM, typename real>() { return kELane<real> ? kELaneMin<MM> : INT64_MAX; });
}

// Elements per group and scratch of a solver of K elements; see ElasticOps.
int elayout(int M, bool dbl, int64_t K, size_t* flux, size_t* trace) {
  return edispatch(M, dbl, [&]<int MM, typename real>() {
    *flux = *trace = 0;
    if constexpr (kELane<real>) {
      if (K >= kELaneMin<MM>) {
        *flux = flux_values(K, np2(kN));
        *trace = size_t(K) * np3(kN);
        return 1;
      }
    }
    return EShape<real>::V;
  });
}

void escale(int M, const double* cj, double* cs) {
  edispatch(M, true, [&]<int MM, typename real>() {
    projection_scale<kN, MM>(cj, cs);
    return 0;
  });
}

void eshape(int M, bool dbl, int* team, int* width, int* groups) {
  edispatch(M, dbl, [&]<int MM, typename real>() {
    *team = EShape<real>::T;
    *width = EShape<real>::V;
    *groups = kEGC<MM, real>;
    return 0;
  });
}

}  // namespace

#define BBW_ECAT2(a, b) a##b
#define BBW_ECAT(a, b) BBW_ECAT2(a, b)
const ElasticOps& BBW_ECAT(elastic_ops_n, BBW_N)() {
  static const ElasticOps ops = {&eprepare, &elaunch, &eshape, &elayout, &elane_min, &escale};
  return ops;
}

}  // namespace bbw
