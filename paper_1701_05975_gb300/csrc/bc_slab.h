// Per-source slabs: what they hold for each schedule, and where the sweep
// schedule keeps its arrays.
#pragma once

#include <algorithm>
#include <cstdint>

#include "bc_common.h"

namespace bcgpu {

// Graphs of up to this many vertices run the sweep schedule from shared memory:
// three 256-thread teams to an SM at 1536 (46 bytes per vertex).  Against slabs,
// all sources, best team of each: Erdos-Renyi 600 184 / 257 us, 1024 386 / 451,
// 1500 818 / 929, 2048 1356 / 1461; BA 1500 501 / 549, 2048 843 / 676; 45 x 45 grid
// 2673 / 1737 (two teams to an SM there).
constexpr uint32_t SWEEP_SMEM_N = 1536;
// The vertex bits are in shared memory while 1024 threads' worth of teams
// keep theirs within this many bytes of an SM's 227 KB.
constexpr uint32_t SWEEP_BITS_MAX = 212u << 10;

inline uint64_t align256(uint64_t x) { return (x + 255) & ~uint64_t(255); }

// Vertices from this id on are neither a row's owner nor any entry's neighbour:
// the sweep schedule's vertex bits cover the ids below it.  A row's neighbours
// count as much as the row: a CSR that stores an edge in one direction only is
// accepted, and its targets need not have rows.
inline uint32_t active_vertices(uint32_t n, const uint64_t* row_ptr, const uint32_t* col) {
  uint32_t last = n;
  while (last > 0 && row_ptr[last] == row_ptr[last - 1]) --last;
  if (last < n)
    for (uint64_t e = 0; e < row_ptr[n]; ++e) last = std::max(last, col[e] + 1);
  return last;
}

// Whether the sweep schedule's 32-bit counts hold: vertex ids in signed words,
// DAG lists of every entry plus two words per vertex, and room for a walk's last
// stride.  Larger graphs run the strict schedule.
inline bool sweep_counts_fit(uint32_t n, uint64_t nnz) {
  return n < 0x80000000u && nnz + 2ull * n < (1ull << 32) - (1u << 16);
}

// What a workspace's slabs hold: the layouts and the values their arrays keep
// between sources differ by schedule.
enum SlabKind : int { SLAB_STRICT = 0, SLAB_SWEEP = 1, SLAB_NONE = 2 };

inline SlabLayout make_layout(uint32_t n, int dist_bits, SlabKind kind) {
  SlabLayout L{};
  uint64_t off = 0;
  const uint64_t grain = kind == SLAB_NONE ? 16 : 256;
  auto take = [&](uint64_t bytes) {
    const uint64_t at = off;
    off += (bytes + grain - 1) & ~(grain - 1);
    return at;
  };
  if (kind == SLAB_NONE) {
    // every per-source array in a CTA's shared memory, queue entries in 16 bits
    L.off_sig = take((uint64_t)n * 16);
    L.off_d = take((uint64_t)n * (dist_bits / 8));
    L.off_acc = take((uint64_t)n * 4);
    L.pair_cap = 3 * n + 64;
    L.off_pairs = take(((uint64_t)L.pair_cap + 8) * 4);
    L.off_pend = take((((uint64_t)n + 31) / 32) * 12);
    for (uint64_t* q : {&L.off_near, &L.off_far, &L.off_far2, &L.off_ends, &L.off_S}) *q = take(((uint64_t)n + 2) * 2);
    L.smem = (uint32_t)off;
    L.stride = 256;  // nothing of it is in the slab
    return L;
  }
  const uint64_t w = (uint64_t)n * 4, w2 = ((uint64_t)n + 2) * 4;
  L.off_d = take((uint64_t)n * (dist_bits / 8));
  if (kind == SLAB_SWEEP) {
    L.off_sig = take((uint64_t)n * 16);
    L.off_near = take(w2);
    L.off_far = take(w2);
    L.off_far2 = take(w);
    L.off_ends = take(w);
    L.off_S = take(w);
    L.off_acc = take(w);
    L.off_pend = take((((uint64_t)n + 31) / 32) * 12);
    // DAG lists (two words per vertex with successors, then the successors):
    // 8 n words cover six DAG edges per vertex; a source beyond that walks
    // the rows again instead
    L.pair_cap = (uint32_t)std::min<uint64_t>(8ull * n + 64, 0xffffffffull);
    L.off_pairs = take(((uint64_t)L.pair_cap + 8) * 4);
    L.stride = off;
    return L;
  }
  L.off_sig = take((uint64_t)n * 8);
  L.off_S = take(w);
  L.off_ends = take(w2);
  L.off_near = take(w);
  L.off_far = take(w);
  L.off_far2 = take(w);
  L.off_acc = take((uint64_t)n * 8);
  L.off_pend = take(w2);
  // DAG edge list: 2 n pairs covers every graph whose shortest-path DAG has at
  // most two in-edges per vertex on average (sources beyond it fall back to
  // the per-entry backward scan)
  L.pair_cap = (uint32_t)std::min<uint64_t>(2ull * n + 64, 0xffffffffull);
  L.off_pairs = take((uint64_t)L.pair_cap * 8);
  L.off_pair_e = take((uint64_t)L.pair_cap * 4);
  L.stride = off;
  return L;
}

// The values every slab holds between sources: distances INF, backward
// accumulators (strict) or vertex records and bits (sweep) zero; other arrays are
// written before they are read.
inline cudaError_t init_slabs(char* slabs, const SlabLayout& lay, SlabKind kind, uint32_t slots, uint32_t n, int dist_bits,
                       cudaStream_t st, const uint32_t* gate = nullptr) {
  if (kind == SLAB_NONE) return cudaSuccess;
  cudaError_t e = launch_fill_slabs(slabs, lay.stride, slots, lay.off_d, align256((uint64_t)n * (dist_bits / 8)),
                                    0xffffffffu, st, gate);
  if (e != cudaSuccess) return e;
  if (kind == SLAB_SWEEP) {
    e = launch_fill_slabs(slabs, lay.stride, slots, lay.off_sig, align256((uint64_t)n * 16), 0u, st, gate);
    if (e != cudaSuccess) return e;
    return launch_fill_slabs(slabs, lay.stride, slots, lay.off_pend, align256((((uint64_t)n + 31) / 32) * 8), 0u, st,
                             gate);
  }
  return launch_fill_slabs(slabs, lay.stride, slots, lay.off_acc, align256((uint64_t)n * 8), 0u, st, gate);
}

// Teams of `team` threads that an SM holds: by the registers the kernels are
// compiled for (64 a thread; 64-bit distance words leave room for 7/8 of them up
// to 256 threads), and by the bytes of shared memory a team keeps its source in
// (0: in a slab), 3 KB more for its own state and the system's share.
inline uint32_t sweep_teams_per_sm(int dist_bits, uint32_t team, uint32_t smem) {
  const uint32_t by_regs = (dist_bits == 64 && team <= 256 ? 896u : 1024u) / team;
  return smem ? std::min<uint32_t>(by_regs, (228u << 10) / (smem + 3072u)) : by_regs;
}

// Memory form of a sweep plan whose distance width and team are set: n
// vertices, the ones from act_n on without entries.
inline void sweep_place(SweepPlan& p, uint32_t n, uint32_t act_n, bool allow_smem) {
  p.mem = 0;
  p.smem_bytes = 0;
  if (p.team < 128) return;
  const uint64_t bits = ((uint64_t)act_n + 31) / 32 * 8;
  if (allow_smem && n <= SWEEP_SMEM_N) {
    p.mem = 2;
    p.group = 1;
    p.smem_bytes = make_layout(n, p.dist_bits, SLAB_NONE).smem;
  } else if (bits <= (uint64_t)SWEEP_BITS_MAX * p.team / 1024) {
    p.mem = 1;
    p.smem_bytes = (uint32_t)bits;
  }
}

}  // namespace bcgpu
