// bbw_warp_tile.cuh -- how a warp moves one field of its 32 elements between
// global memory ([element][field][Np]) and one column per element in shared
// memory (kernels with one element per lane).
#pragma once

#include <cstdint>
#include <cstring>

namespace bbw {

// A field of an element is Np consecutive values. A lane takes chunks of W
// consecutive values (16 bytes where Np allows it); GL lanes take GL elements
// and CL = 32 / GL lanes consecutive chunks of each, GL chosen for the fewest
// line accesses. Consecutive lanes take consecutive chunks: a 16-byte access
// is served eight lanes at a time, which then lie in one 128-byte line (with
// consecutive lanes on different elements it took four times the wavefronts).
// Chunk `it` of a lane lies at a compile-time offset from the lane's first
// one, in global memory and in the columns, so a round costs its memory
// instructions and no address arithmetic.
template <int Np, typename real>
struct WarpTile {
  static constexpr int WMAX = 16 / int(sizeof(real));
  static constexpr int W = Np % WMAX == 0 ? WMAX : (Np % 2 == 0 && WMAX >= 2 ? 2 : 1);
  static constexpr int NC = Np / W;  // chunks per element
  // an access of a warp costs its 128-byte lines, at least one per element, and
  // about as much as ten more in instructions
  static constexpr int pick_gl() {
    constexpr int lines = W * int(sizeof(real)) * 32 / 128;
    int best = 32, cost = 1 << 30;
    for (int gl = 32; gl >= 2; gl /= 2) {
      const int cl = 32 / gl, it = (32 / gl) * ((NC + cl - 1) / cl), c = it * ((gl > lines ? gl : lines) + 10);
      if (c < cost) {
        cost = c;
        best = gl;
      }
    }
    return best;
  }
  static constexpr int GL = pick_gl();
  static constexpr int CL = 32 / GL;  // chunk lanes
  static constexpr int CB = (NC + CL - 1) / CL;
  static constexpr int IT = (32 / GL) * CB;  // chunks per lane
  struct Chunk {
    real x[W];
  };
  // first chunk of a lane; offset of its chunk it (ES: values between elements)
  template <int ES>
  static __device__ __forceinline__ int first(int lane) {
    return (lane / CL) * ES + (lane % CL) * W;
  }
  template <int ES>
  static constexpr __device__ int offset(int it) {
    return (it / CB) * GL * ES + (it % CB) * CL * W;
  }
  static __device__ __forceinline__ int element(int lane, int it) { return (it / CB) * GL + lane / CL; }
  // whether the lane's chunk it exists, of ne elements
  static __device__ __forceinline__ bool has(int lane, int it, int ne) {
    return it < IT && element(lane, it) < ne && ((it % CB + 1) * CL <= NC || (it % CB) * CL + lane % CL < NC);
  }
  static __device__ __forceinline__ Chunk load(const real* p) {
    Chunk c;
    if constexpr (W * sizeof(real) == 16) {
      const uint4 t = *reinterpret_cast<const uint4*>(p);
      memcpy(c.x, &t, 16);
    } else if constexpr (W * sizeof(real) == 8) {
      const uint2 t = *reinterpret_cast<const uint2*>(p);
      memcpy(c.x, &t, 8);
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w) c.x[w] = p[w];
    }
    return c;
  }
  static __device__ __forceinline__ void store(real* p, const Chunk& c) {
    if constexpr (W * sizeof(real) == 16) {
      uint4 t;
      memcpy(&t, c.x, 16);
      *reinterpret_cast<uint4*>(p) = t;
    } else if constexpr (W * sizeof(real) == 8) {
      uint2 t;
      memcpy(&t, c.x, 8);
      *reinterpret_cast<uint2*>(p) = t;
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w) p[w] = c.x[w];
    }
  }
  // The lane's chunks held in registers between their loads and their use.
  struct Held {
    Chunk c[IT];
  };
  template <int ES>
  static __device__ __forceinline__ void hold(Held& h, const real* __restrict__ src, int lane, int ne) {
    const real* p = src + first<ES>(lane);
#pragma unroll
    for (int it = 0; it < IT; ++it)
      if (has(lane, it, ne)) h.c[it] = load(p + offset<ES>(it));
  }
  template <int S>
  static __device__ __forceinline__ void put(const Held& h, real* cols, int lane, int ne) {
    real* c = cols + first<S>(lane);
#pragma unroll
    for (int it = 0; it < IT; ++it)
      if (has(lane, it, ne))
#pragma unroll
        for (int w = 0; w < W; ++w) c[offset<S>(it) + w] = h.c[it].x[w];
  }
  // global field -> columns of stride S, U chunks in flight
  template <int ES, int S, int U>
  static __device__ __forceinline__ void stage(real* cols, const real* __restrict__ src, int lane, int ne) {
    const real* p = src + first<ES>(lane);
    real* c = cols + first<S>(lane);
#pragma unroll
    for (int i0 = 0; i0 < IT; i0 += U) {
      Chunk h[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (has(lane, i0 + u, ne)) h[u] = load(p + offset<ES>(i0 + u));
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (has(lane, i0 + u, ne))
#pragma unroll
          for (int w = 0; w < W; ++w) c[offset<S>(i0 + u) + w] = h[u].x[w];
    }
  }
  static __device__ __forceinline__ Chunk take(const real* c) {
    Chunk h;
#pragma unroll
    for (int w = 0; w < W; ++w) h.x[w] = c[w];
    return h;
  }
  // columns -> global field
  template <int ES, int S>
  static __device__ __forceinline__ void unstage(const real* cols, real* __restrict__ dst, int lane, int ne) {
    real* p = dst + first<ES>(lane);
    const real* c = cols + first<S>(lane);
#pragma unroll
    for (int it = 0; it < IT; ++it)
      if (has(lane, it, ne)) store(p + offset<ES>(it), take(c + offset<S>(it)));
  }
  // Prefetch the field of the lane's element (ES values apart) into L2, whole
  // 16-byte pieces only.
  template <int ES>
  static __device__ __forceinline__ void prefetch(const real* src, int lane, int ne) {
    if (lane < ne) {
      const uintptr_t b = reinterpret_cast<uintptr_t>(src + size_t(lane) * ES);
      const uintptr_t lo = (b + 15) & ~uintptr_t(15), hi = (b + Np * sizeof(real)) & ~uintptr_t(15);
      if (hi > lo)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"(uint32_t(hi - lo)) : "memory");
    }
  }
};

}  // namespace bbw
