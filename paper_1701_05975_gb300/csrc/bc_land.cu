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

// f(v, e) for every entry e of every row v, `chunk` consecutive entries to a
// warp (32 to 256: few enough that small graphs fill the GPU).  A warp per row
// left one warp with a hub's whole row.  With a hub of 4 million neighbours and 8
// million more edges graph creation took 1990 ms, 1560 with the row sorted by the
// whole GPU and 1258 in chunks (317 of them the distances); a star of 4 million 326
// and 208; graphs without such rows as before (Barabasi-Albert 12k 3.0, R-MAT scale 18 236).
uint32_t land_chunk(uint64_t nnz) {
  const uint64_t share = nnz / (152ull * 16 * 8) + 1;  // over the warps of the largest grid
  return (uint32_t)std::min<uint64_t>((share + 31) / 32 * 32, 256);
}
template <typename F>
__device__ __forceinline__ void land_entries(uint32_t n, uint64_t nnz, const uint64_t* __restrict__ row_ptr, uint32_t chunk,
                                             F&& f) {
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t c = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; c * chunk < nnz; c += nwarps) {
    uint64_t e = c * chunk;
    const uint64_t end = min((unsigned long long)(e + chunk), (unsigned long long)nnz);
    uint32_t v = 0, past = n;  // row_ptr[v] <= e < row_ptr[past]
    while (past - v > 1) {
      const uint32_t mid = v + (past - v) / 2;
      if (row_ptr[mid] <= e) v = mid;
      else past = mid;
    }
    for (; e < end; ++v) {
      const uint64_t stop = min((unsigned long long)row_ptr[v + 1], (unsigned long long)end);
      for (uint64_t i = e + lane; i < stop; i += 32) f(v, i);
      e = stop;
    }
  }
}

// out[0], out[1]: sums of entry_hash over the entries and over their reverses.
__global__ void land_symmetry_kernel(uint32_t n, uint64_t nnz, uint32_t chunk, const uint64_t* __restrict__ row_ptr,
                                     const uint2* __restrict__ adj, unsigned long long* out) {
  unsigned long long fwd = 0, rev = 0;
  land_entries(n, nnz, row_ptr, chunk, [&](uint32_t v, uint64_t e) {
    const uint2 x = adj[e];
    fwd += entry_hash(v, x.x, x.y);
    rev += entry_hash(x.x, v, x.y);
  });
  __syncwarp();
  for (int o = 16; o > 0; o >>= 1) {
    fwd += __shfl_xor_sync(0xffffffffu, fwd, o);
    rev += __shfl_xor_sync(0xffffffffu, rev, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&out[0], fwd);
    atomicAdd(&out[1], rev);
  }
}

// Judge the main landmark h on probe sources (distances probe[p * n + v],
// so D(probe p, h) = probe[p * n + h]): out[0] entries of reached rows, out[1] those the
// prefix test keeps.  out[2]: 1 + the largest vertex with entries that the main
// landmark reaches.  out[3]: entries on shortest paths from the probes (tight ones).
__global__ void land_judge_kernel(uint32_t n, uint64_t nnz, uint32_t chunk, const uint64_t* __restrict__ row_ptr,
                                  const uint2* __restrict__ adj, const uint32_t* __restrict__ from_h,
                                  const uint32_t* __restrict__ probe, uint32_t h, uint32_t nprobe,
                                  unsigned long long* out) {
  unsigned long long all = 0, kept = 0, last = 0, tight = 0;
  land_entries(n, nnz, row_ptr, chunk, [&](uint32_t v, uint64_t e) {
    const uint2 x = adj[e];
    const uint32_t hu = from_h[x.x];
    if (from_h[v] != 0xffffffffu) last = v + 1;  // rows come in ascending order
    for (uint32_t p = 0; p < nprobe; ++p) {
      const uint32_t c = probe[(uint64_t)p * n + h], d = probe[(uint64_t)p * n + v];
      if (c == 0xffffffffu || d == 0xffffffffu) continue;
      ++all;
      tight += probe[(uint64_t)p * n + x.x] == d + x.y;
      kept += hu == 0xffffffffu || (long long)x.y - (long long)hu <= (long long)c - (long long)d;
    }
  });
  __syncwarp();
  for (int o = 16; o > 0; o >>= 1) {
    all += __shfl_xor_sync(0xffffffffu, all, o);
    kept += __shfl_xor_sync(0xffffffffu, kept, o);
    tight += __shfl_xor_sync(0xffffffffu, tight, o);
    last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&out[0], all);
    atomicAdd(&out[1], kept);
    atomicMax(&out[2], last);
    atomicAdd(&out[3], tight);
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
__global__ void land_key_kernel(uint32_t n, uint64_t nnz, uint32_t chunk, const uint64_t* __restrict__ row_ptr,
                                const uint2* __restrict__ adj, const uint32_t* __restrict__ from_h,
                                unsigned long long* __restrict__ key) {
  land_entries(n, nnz, row_ptr, chunk, [&](uint32_t v, uint64_t e) {
    const uint2 x = adj[e];
    const uint32_t h = from_h[x.x];
    // both words are below 2^31, so the difference fits 32 bits signed
    const uint32_t k = h == 0xffffffffu ? 0u : (x.y - h) ^ 0x80000000u;
    key[e] = ((unsigned long long)k << 32) | (uint32_t)(e - row_ptr[v]);
  });
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

// Bitonic sort in which every comparison is ascending (the first step of a
// merge compares with the mirrored index), so elements past the end behave as
// +infinity without being stored.  One step: element i against i ^ x.
__device__ __forceinline__ void land_step(unsigned long long* a, uint64_t len, uint64_t x, uint64_t first,
                                          uint64_t stride) {
  for (uint64_t i = first; i < len; i += stride) {
    const uint64_t p = i ^ x;
    if (p > i && p < len) {
      const unsigned long long u = a[i], w = a[p];
      if (u > w) {
        a[i] = w;
        a[p] = u;
      }
    }
  }
}

// The steps of distance j, j / 2, .., 1 by one CTA.
__device__ void land_merge(unsigned long long* a, uint32_t len, uint64_t j) {
  for (; j > 0; j >>= 1) {
    land_step(a, len, j, threadIdx.x, blockDim.x);
    __syncthreads();
  }
}

// a[0, len) by one CTA.
__device__ void land_bitonic(unsigned long long* a, uint32_t len) {
  for (uint64_t k = 2; k < 2ull * len; k <<= 1) {
    land_step(a, len, k - 1, threadIdx.x, blockDim.x);
    __syncthreads();
    land_merge(a, len, k >> 2);
  }
}

constexpr uint32_t LAND_SMEM_ROW = 4096;

// Rows of 33 to `longest` entries, a CTA each.
__global__ void land_sort_cta(uint32_t n, const uint64_t* __restrict__ row_ptr, unsigned long long* __restrict__ key,
                              uint64_t longest) {
  __shared__ unsigned long long buf[LAND_SMEM_ROW];
  for (uint64_t v = blockIdx.x; v < n; v += gridDim.x) {
    const uint64_t r0 = row_ptr[v], deg = row_ptr[v + 1] - r0;
    if (deg <= 32 || deg > longest) continue;
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

// One long row over the whole GPU: blocks of LAND_SMEM_ROW keys sorted (j = 0)
// or merged from distance j down in shared memory, and single steps between them.
__global__ void land_sort_blocks(uint64_t len, unsigned long long* __restrict__ key, uint64_t j) {
  __shared__ unsigned long long buf[LAND_SMEM_ROW];
  const uint64_t b0 = blockIdx.x * (uint64_t)LAND_SMEM_ROW;
  const uint32_t count = (uint32_t)min((unsigned long long)LAND_SMEM_ROW, (unsigned long long)(len - b0));
  for (uint32_t i = threadIdx.x; i < count; i += blockDim.x) buf[i] = key[b0 + i];
  __syncthreads();
  if (j == 0) land_bitonic(buf, count);
  else land_merge(buf, count, j);
  for (uint32_t i = threadIdx.x; i < count; i += blockDim.x) key[b0 + i] = buf[i];
}
__global__ void land_sort_step(uint64_t len, unsigned long long* __restrict__ key, uint64_t x) {
  land_step(key, len, x, blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, (uint64_t)gridDim.x * blockDim.x);
}

void land_sort_grid(uint64_t len, unsigned long long* key, cudaStream_t st) {
  const uint32_t blocks = (uint32_t)((len + LAND_SMEM_ROW - 1) / LAND_SMEM_ROW);
  const int grid = (int)std::min<uint64_t>((len + 511) / 512, 152ull * 8);
  land_sort_blocks<<<blocks, 512, 0, st>>>(len, key, 0);
  for (uint64_t k = 2ull * LAND_SMEM_ROW; k < 2 * len; k <<= 1) {
    land_sort_step<<<grid, 512, 0, st>>>(len, key, k - 1);
    uint64_t j = k >> 2;
    for (; j >= LAND_SMEM_ROW; j >>= 1) land_sort_step<<<grid, 512, 0, st>>>(len, key, j);
    land_sort_blocks<<<blocks, 512, 0, st>>>(len, key, j);
  }
}

// The sorted rows: {neighbour (packed with the weight when col_bits > 0), w - D(h, u)}.
__global__ void land_rows_kernel(uint32_t n, uint64_t nnz, uint32_t chunk, const uint64_t* __restrict__ row_ptr,
                                 const uint2* __restrict__ adj, const unsigned long long* __restrict__ key,
                                 uint32_t col_bits, const uint32_t* __restrict__ e2o, uint2* __restrict__ kadj,
                                 uint32_t* __restrict__ kw, uint32_t* __restrict__ k2o) {
  land_entries(n, nnz, row_ptr, chunk, [&](uint32_t v, uint64_t e) {
    const unsigned long long k = key[e];
    const uint64_t from = row_ptr[v] + (uint32_t)k;
    const uint2 x = adj[from];
    kadj[e] = make_uint2(col_bits ? (x.x | (x.y << col_bits)) : x.x, (uint32_t)(k >> 32) ^ 0x80000000u);
    if (kw) kw[e] = x.y;
    k2o[e] = e2o ? e2o[from] : (uint32_t)from;
  });
}

// Rows longer than this take the whole GPU, if there are at most LAND_GRID_ROWS of them.
constexpr uint64_t LAND_GRID_ROW = 32768;
constexpr uint32_t LAND_GRID_ROWS = 64;

int land_grid(uint64_t warps) {
  return (int)std::max<uint64_t>(1, std::min<uint64_t>((warps + 7) / 8, 152ull * 16));
}

}  // namespace

cudaError_t land_symmetry(const GraphDev& g, unsigned long long* out, cudaStream_t st) {
  const uint32_t chunk = land_chunk(g.nnz);
  land_symmetry_kernel<<<land_grid(g.nnz / chunk + 1), 256, 0, st>>>(g.n, g.nnz, chunk, g.row_ptr, g.adj, out);
  return cudaGetLastError();
}

cudaError_t land_judge(const GraphDev& g, const uint32_t* from_h, const uint32_t* probe, uint32_t h,
                       uint32_t nprobe, unsigned long long* out, cudaStream_t st) {
  const uint32_t chunk = land_chunk(g.nnz);
  land_judge_kernel<<<land_grid(g.nnz / chunk + 1), 256, 0, st>>>(g.n, g.nnz, chunk, g.row_ptr, g.adj, from_h, probe, h,
                                                                  nprobe, out);
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

cudaError_t land_rows(const GraphDev& g, const uint64_t* host_row_ptr, const uint32_t* from_h, unsigned long long* key,
                      uint32_t col_bits, uint2* kadj, uint32_t* kw, uint32_t* k2o, cudaStream_t st) {
  const uint32_t chunk = land_chunk(g.nnz);
  const int grid = land_grid(g.nnz / chunk + 1);
  land_key_kernel<<<grid, 256, 0, st>>>(g.n, g.nnz, chunk, g.row_ptr, g.adj, from_h, key);
  land_sort_warp<<<land_grid(g.n), 256, 0, st>>>(g.n, g.row_ptr, key);
  // a hub's row is sorted by the whole GPU, unless there are so many of them
  // that a CTA each keeps it as busy
  uint32_t rows = 0;
  for (uint32_t v = 0; v < g.n; ++v) rows += host_row_ptr[v + 1] - host_row_ptr[v] > LAND_GRID_ROW;
  const uint64_t longest = rows <= LAND_GRID_ROWS ? LAND_GRID_ROW : g.nnz;
  land_sort_cta<<<(int)std::min<uint64_t>(g.n, 152ull * 4), 512, 0, st>>>(g.n, g.row_ptr, key, longest);
  for (uint32_t v = 0; rows && longest < g.nnz && v < g.n; ++v) {
    const uint64_t deg = host_row_ptr[v + 1] - host_row_ptr[v];
    if (deg > longest) land_sort_grid(deg, key + host_row_ptr[v], st);
  }
  land_rows_kernel<<<grid, 256, 0, st>>>(g.n, g.nnz, chunk, g.row_ptr, g.adj, key, col_bits, g.e2o, kadj, kw, k2o);
  return cudaGetLastError();
}

}  // namespace bcgpu
