// Team primitives shared by the per-source kernels: a team is one warp or one
// CTA that works on one source.  Barriers, scans and minima over a team, and
// the loads and atomics on a team's own arrays.  Anonymous namespace: each
// translation unit owns its copies.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace bcgpu {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t NONE = 0xffffffffu;

template <typename D>
__device__ __forceinline__ D dinf() {
  return ~D(0);
}

__device__ __forceinline__ uint32_t ldcg(const uint32_t* p) { return __ldcg(p); }
__device__ __forceinline__ uint64_t ldcg(const uint64_t* p) {
  return (uint64_t)__ldcg(reinterpret_cast<const unsigned long long*>(p));
}
__device__ __forceinline__ double ldcg(const double* p) { return __ldcg(p); }

__device__ __forceinline__ uint32_t atomic_min_d(uint32_t* p, uint32_t v) { return atomicMin(p, v); }
__device__ __forceinline__ uint64_t atomic_min_d(uint64_t* p, uint64_t v) {
  return (uint64_t)atomicMin(reinterpret_cast<unsigned long long*>(p), (unsigned long long)v);
}

template <typename D>
__device__ __forceinline__ D sat_add(D a, uint64_t b) {
  uint64_t lim = (uint64_t)dinf<D>() - 1;
  uint64_t aa = (uint64_t)a;
  if (aa >= lim || b >= lim - aa) return (D)lim;
  return (D)(aa + b);
}

template <typename D>
__device__ __forceinline__ D shfl_xor_d(D x, int o) {
  return __shfl_xor_sync(FULL, x, o);
}

template <typename D>
__device__ __forceinline__ D dmin(D a, D b) {
  return a < b ? a : b;
}
template <typename D>
__device__ __forceinline__ D dmax(D a, D b) {
  return a < b ? b : a;
}

template <int TEAM>
__device__ __forceinline__ void team_sync() {
  // __syncthreads alone does not bring the lanes of a diverged warp back
  // together; left apart they issue every later instruction twice over
  __syncwarp();
  if constexpr (TEAM > 32) __syncthreads();
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Exclusive prefix sum over the team; *total receives the team-wide sum.
// Every thread of the team must call it.
template <int TEAM>
__device__ __forceinline__ uint32_t team_excl_scan(uint32_t x, uint32_t* total, uint32_t* scratch) {
  uint32_t inc = warp_incl_scan(x);
  if constexpr (TEAM == 32) {
    *total = __shfl_sync(FULL, inc, 31);
    return inc - x;
  } else {
    constexpr int NW = TEAM / 32;
    const int w = (threadIdx.x % TEAM) >> 5, lane = threadIdx.x & 31;
    if (lane == 31) scratch[w] = inc;
    __syncthreads();
    if (w == 0) {
      uint32_t v = lane < NW ? scratch[lane] : 0u;
      uint32_t vi = warp_incl_scan(v);
      if (lane < NW) scratch[lane] = vi - v;
      if (lane == NW - 1) scratch[NW] = vi;
    }
    __syncthreads();
    *total = scratch[NW];
    uint32_t r = scratch[w] + inc - x;
    __syncthreads();
    return r;
  }
}

// Two exclusive prefix sums at once (shares the barriers).
template <int TEAM>
__device__ __forceinline__ void team_excl_scan2(uint32_t x, uint32_t y, uint32_t* ex, uint32_t* ey, uint32_t* tx,
                                                uint32_t* ty, uint32_t* scratch) {
  const uint32_t ix = warp_incl_scan(x), iy = warp_incl_scan(y);
  if constexpr (TEAM == 32) {
    *tx = __shfl_sync(FULL, ix, 31);
    *ty = __shfl_sync(FULL, iy, 31);
    *ex = ix - x;
    *ey = iy - y;
  } else {
    constexpr int NW = TEAM / 32;
    const int w = (threadIdx.x % TEAM) >> 5, lane = threadIdx.x & 31;
    if (lane == 31) {
      scratch[w] = ix;
      scratch[NW + 1 + w] = iy;
    }
    __syncthreads();
    if (w == 0) {
      const uint32_t vx = lane < NW ? scratch[lane] : 0u, vy = lane < NW ? scratch[NW + 1 + lane] : 0u;
      const uint32_t sx = warp_incl_scan(vx), sy = warp_incl_scan(vy);
      if (lane < NW) {
        scratch[lane] = sx - vx;
        scratch[NW + 1 + lane] = sy - vy;
      }
      if (lane == NW - 1) {
        scratch[NW] = sx;
        scratch[2 * NW + 1] = sy;
      }
    }
    __syncthreads();
    *tx = scratch[NW];
    *ty = scratch[2 * NW + 1];
    *ex = scratch[w] + ix - x;
    *ey = scratch[NW + 1 + w] + iy - y;
    __syncthreads();
  }
}

// Team-wide minimum of two values at once.
template <typename D, int TEAM>
__device__ __forceinline__ void team_min2(D& a, D& b, D* scratch) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a = dmin(a, shfl_xor_d(a, o));
    b = dmin(b, shfl_xor_d(b, o));
  }
  if constexpr (TEAM > 32) {
    constexpr int NW = TEAM / 32;
    const int w = (threadIdx.x % TEAM) >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
      scratch[w] = a;
      scratch[NW + w] = b;
    }
    __syncthreads();
    if (w == 0) {
      D x = lane < NW ? scratch[lane] : dinf<D>();
      D y = lane < NW ? scratch[NW + lane] : dinf<D>();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        x = dmin(x, shfl_xor_d(x, o));
        y = dmin(y, shfl_xor_d(y, o));
      }
      if (lane == 0) {
        scratch[2 * NW] = x;
        scratch[2 * NW + 1] = y;
      }
    }
    __syncthreads();
    a = scratch[2 * NW];
    b = scratch[2 * NW + 1];
    __syncthreads();
  }
}

}  // namespace
}  // namespace bcgpu
