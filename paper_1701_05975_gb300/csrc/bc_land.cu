// Landmark preparation for the sweep schedule (once per graph): distances
// from the landmarks come from the sweep kernel's distance rounds; the
// kernels here judge them on a few probe sources, pack the bound table and
// put every row in the order of w - D(h, u) (the prefix test of bc_sweep.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "bc_common.h"

namespace bcgpu {
namespace {

// 64-bit finaliser of SplitMix64 (Steele, Lea and Flood, OOPSLA 2014).
__device__ __forceinline__ unsigned long long land_mix(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// out[0] - out[1] = sum over entries of hash(v, u, w) - hash(u, v, w), mod
// 2^64: zero for a symmetric CSR, and for another only with probability about
// 2^-64.  One warp per row.
__global__ void land_symmetry_kernel(uint32_t n, const uint64_t* __restrict__ row_ptr, const uint2* __restrict__ adj,
                                     unsigned long long* out) {
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  unsigned long long fwd = 0, rev = 0;
  for (uint64_t v = warp; v < n; v += nwarps)
    for (uint64_t e = row_ptr[v] + lane; e < row_ptr[v + 1]; e += 32) {
      const uint2 x = adj[e];
      const unsigned long long hw = land_mix((unsigned long long)x.y + 0x9e3779b97f4a7c15ull);
      fwd += land_mix(((v << 32) | x.x) ^ hw);
      rev += land_mix((((unsigned long long)x.x << 32) | v) ^ hw);
    }
  for (int o = 16; o > 0; o >>= 1) {
    fwd += __shfl_xor_sync(0xffffffffu, fwd, o);
    rev += __shfl_xor_sync(0xffffffffu, rev, o);
  }
  if (lane == 0) {
    atomicAdd(&out[0], fwd);
    atomicAdd(&out[1], rev);
  }
}

// Judge the main landmark h on probe sources (distances probe[p * n + v],
// so D(probe p, h) = probe[p * n + h]): out[0] entries of reached rows, out[1] those the
// prefix test keeps, out[2] reached vertices.  out[3]: 1 + the largest
// vertex the main landmark reaches.  One warp per row.
__global__ void land_judge_kernel(uint32_t n, const uint64_t* __restrict__ row_ptr, const uint2* __restrict__ adj,
                                  const uint32_t* __restrict__ from_h, const uint32_t* __restrict__ probe,
                                  uint32_t h, uint32_t nprobe, unsigned long long* out) {
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  unsigned long long all = 0, kept = 0, reached = 0, last = 0;
  for (uint64_t v = warp; v < n; v += nwarps) {
    const uint64_t r0 = row_ptr[v], r1 = row_ptr[v + 1];
    if (lane == 0 && from_h[v] != 0xffffffffu) last = v + 1;
    for (uint32_t p = 0; p < nprobe; ++p) {
      const uint32_t c = probe[(uint64_t)p * n + h], d = probe[(uint64_t)p * n + v];
      if (c == 0xffffffffu || d == 0xffffffffu) continue;
      if (lane == 0) {
        all += r1 - r0;
        ++reached;
      }
      for (uint64_t e = r0 + lane; e < r1; e += 32) {
        const uint2 x = adj[e];
        const uint32_t hu = from_h[x.x];
        kept += hu == 0xffffffffu || (long long)x.y - (long long)hu <= (long long)c - (long long)d;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, o);
  if (lane == 0) {
    atomicAdd(&out[0], all);
    atomicAdd(&out[1], kept);
    atomicAdd(&out[2], reached);
    atomicMax(&out[3], last);
  }
}

// Largest finite word of a distance table.
__global__ void land_max_kernel(uint64_t count, const uint32_t* __restrict__ tab, uint32_t* out) {
  uint32_t m = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x)
    if (tab[i] != 0xffffffffu) m = max(m, tab[i]);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// Rows of n words to rows of `stride` words, 16-bit (0x7fff: unreachable) or
// 32-bit; the padding is unreachable.
template <typename W>
__global__ void land_pack_kernel(uint32_t n, uint64_t stride, uint32_t rows, const uint32_t* __restrict__ tab,
                                 W* __restrict__ out) {
  const W none = sizeof(W) == 2 ? (W)0x7fff : (W)0xffffffffu;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < stride * rows;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t l = i / stride, v = i % stride;
    const uint32_t x = v < n ? tab[l * n + v] : 0xffffffffu;
    out[i] = x == 0xffffffffu ? none : (W)x;
  }
}

// Sort key of every entry: w - D(h, u) (an unreachable u sorts first: its
// entries always pass), then the entry's place in the row.
__global__ void land_key_kernel(uint32_t n, const uint64_t* __restrict__ row_ptr, const uint2* __restrict__ adj,
                                const uint32_t* __restrict__ from_h, unsigned long long* __restrict__ key) {
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t v = warp; v < n; v += nwarps) {
    const uint64_t r0 = row_ptr[v], r1 = row_ptr[v + 1];
    for (uint64_t e = r0 + lane; e < r1; e += 32) {
      const uint2 x = adj[e];
      const uint32_t h = from_h[x.x];
      // both words are below 2^31, so the difference fits 32 bits signed
      const uint32_t k = h == 0xffffffffu ? 0u : (x.y - h) ^ 0x80000000u;
      key[e] = ((unsigned long long)k << 32) | (uint32_t)(e - r0);
    }
  }
}

// Rows of up to 32 entries: one warp per row, a bitonic network in registers.
__global__ void land_sort_warp(uint32_t n, const uint64_t* __restrict__ row_ptr, unsigned long long* __restrict__ key) {
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t v = warp; v < n; v += nwarps) {
    const uint64_t r0 = row_ptr[v], deg = row_ptr[v + 1] - r0;
    if (deg < 2 || deg > 32) continue;
    unsigned long long x = lane < deg ? key[r0 + lane] : ~0ull;
#pragma unroll
    for (uint32_t k = 2; k <= 32; k <<= 1) {
#pragma unroll
      for (uint32_t j = k >> 1; j > 0; j >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, j);
        const bool up = ((lane & k) == 0) == ((lane & j) == 0);
        x = up ? (x < y ? x : y) : (x < y ? y : x);
      }
    }
    if (lane < deg) key[r0 + lane] = x;
  }
}

// In-place bitonic sort of a[0, len) by one CTA: every comparison is
// ascending (the first step of a merge compares with the mirrored index), so
// elements past the end behave as +infinity without being stored.
__device__ void land_bitonic(unsigned long long* a, uint32_t len) {
  auto step = [&](uint64_t x) {
    for (uint64_t i = threadIdx.x; i < len; i += blockDim.x) {
      const uint64_t p = i ^ x;
      if (p > i && p < len) {
        const unsigned long long u = a[i], w = a[p];
        if (u > w) {
          a[i] = w;
          a[p] = u;
        }
      }
    }
    __syncthreads();
  };
  for (uint64_t k = 2; k < 2ull * len; k <<= 1) {
    step(k - 1);
    for (uint64_t j = k >> 2; j > 0; j >>= 1) step(j);
  }
}

constexpr uint32_t LAND_SMEM_ROW = 4096;

__global__ void land_sort_cta(uint32_t n, const uint64_t* __restrict__ row_ptr, unsigned long long* __restrict__ key) {
  __shared__ unsigned long long buf[LAND_SMEM_ROW];
  for (uint64_t v = blockIdx.x; v < n; v += gridDim.x) {
    const uint64_t r0 = row_ptr[v], deg = row_ptr[v + 1] - r0;
    if (deg <= 32 || deg > 0xffffffffull) continue;
    if (deg <= LAND_SMEM_ROW) {
      for (uint32_t i = threadIdx.x; i < deg; i += blockDim.x) buf[i] = key[r0 + i];
      __syncthreads();
      land_bitonic(buf, (uint32_t)deg);
      for (uint32_t i = threadIdx.x; i < deg; i += blockDim.x) key[r0 + i] = buf[i];
      __syncthreads();
    } else {
      land_bitonic(key + r0, (uint32_t)deg);
    }
  }
}

// The sorted rows: {neighbour (packed with the weight when col_bits > 0), w - D(h, u)}.
__global__ void land_rows_kernel(uint32_t n, const uint64_t* __restrict__ row_ptr, const uint2* __restrict__ adj,
                                 const unsigned long long* __restrict__ key, uint32_t col_bits,
                                 const uint32_t* __restrict__ e2o, uint2* __restrict__ kadj, uint32_t* __restrict__ kw,
                                 uint32_t* __restrict__ k2o) {
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t v = warp; v < n; v += nwarps) {
    const uint64_t r0 = row_ptr[v], r1 = row_ptr[v + 1];
    for (uint64_t e = r0 + lane; e < r1; e += 32) {
      const unsigned long long k = key[e];
      const uint64_t from = r0 + (uint32_t)k;
      const uint2 x = adj[from];
      kadj[e] = make_uint2(col_bits ? (x.x | (x.y << col_bits)) : x.x, (uint32_t)(k >> 32) ^ 0x80000000u);
      if (kw) kw[e] = x.y;
      k2o[e] = e2o ? e2o[from] : (uint32_t)from;
    }
  }
}

int land_grid(uint64_t warps) {
  return (int)std::max<uint64_t>(1, std::min<uint64_t>((warps + 7) / 8, 152ull * 16));
}

}  // namespace

cudaError_t land_symmetry(const GraphDev& g, unsigned long long* out, cudaStream_t st) {
  land_symmetry_kernel<<<land_grid(g.n), 256, 0, st>>>(g.n, g.row_ptr, g.adj, out);
  return cudaGetLastError();
}

cudaError_t land_judge(const GraphDev& g, const uint32_t* from_h, const uint32_t* probe, uint32_t h,
                       uint32_t nprobe, unsigned long long* out, cudaStream_t st) {
  land_judge_kernel<<<land_grid(g.n), 256, 0, st>>>(g.n, g.row_ptr, g.adj, from_h, probe, h, nprobe, out);
  return cudaGetLastError();
}

cudaError_t land_max(uint64_t count, const uint32_t* tab, uint32_t* out, cudaStream_t st) {
  land_max_kernel<<<land_grid((count + 31) / 32), 256, 0, st>>>(count, tab, out);
  return cudaGetLastError();
}

cudaError_t land_pack(uint32_t n, uint64_t stride, uint32_t rows, const uint32_t* tab, int bits, void* out,
                      cudaStream_t st) {
  const int grid = land_grid((stride * rows + 31) / 32);
  if (bits == 16) land_pack_kernel<<<grid, 256, 0, st>>>(n, stride, rows, tab, static_cast<uint16_t*>(out));
  else land_pack_kernel<<<grid, 256, 0, st>>>(n, stride, rows, tab, static_cast<uint32_t*>(out));
  return cudaGetLastError();
}

cudaError_t land_rows(const GraphDev& g, const uint32_t* from_h, unsigned long long* key, uint32_t col_bits,
                      uint2* kadj, uint32_t* kw, uint32_t* k2o, cudaStream_t st) {
  const int grid = land_grid(g.n);
  land_key_kernel<<<grid, 256, 0, st>>>(g.n, g.row_ptr, g.adj, from_h, key);
  land_sort_warp<<<grid, 256, 0, st>>>(g.n, g.row_ptr, key);
  land_sort_cta<<<(int)std::min<uint64_t>(g.n, 152ull * 4), 512, 0, st>>>(g.n, g.row_ptr, key);
  land_rows_kernel<<<grid, 256, 0, st>>>(g.n, g.row_ptr, g.adj, key, col_bits, g.e2o, kadj, kw, k2o);
  return cudaGetLastError();
}

}  // namespace bcgpu
