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
// kernels' two more launches and their few, long warps cost more than they save.
// Stage times in us, lane / team, M = 2, at 2,058 / 4,374 / 24,576 elements:
// N = 2 29/21, 29/21, 44/72; N = 3 31/21, 36/27, 71/133; N = 4 42/31, 45/58,
// 122/191; N = 5 36/35, 41/66, 156/348; N = 6 56/49, 71/90, 274/468; N = 7
// 76/99, 124/146, 458/744. The projections are fused up to N = 5, where their
// levels fit the register file.
template <typename real>
constexpr bool kELane = sizeof(real) == 4 && kN >= 2 && kN <= 7;
constexpr int64_t kELaneMin = kN <= 3 ? 7000 : kN == 4 ? 4000 : kN == 5 ? 3000 : kN == 6 ? 4000 : 1500;
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

// Elements per group and scratch of a solver of K elements; see ElasticOps.
int elayout(int M, bool dbl, int64_t K, size_t* flux, size_t* trace) {
  return edispatch(M, dbl, [&]<int MM, typename real>() {
    *flux = *trace = 0;
    if constexpr (kELane<real>) {
      if (K >= kELaneMin) {
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
  static const ElasticOps ops = {&eprepare, &elaunch, &eshape, &elayout, &escale};
  return ops;
}

}  // namespace bbw
