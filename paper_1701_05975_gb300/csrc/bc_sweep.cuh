// Sweep schedule of the batched kernel (BC_ALGO_DELTA): one team of threads
// per source, many sources in flight, sources pulled from a device counter.
//
// Per source (arxiv 1701.05975, Sec. 2.1, with distances found before any
// path is counted):
//   1. distances: rounds of frontier relaxation (atomicMin on the distance
//      word).  With landmarks every distance starts at the upper bound
//      min_l D(s, l) + D(l, v), one coalesced pass over a small table, and
//      only vertices that beat the bound are ever relaxed; without them
//      improved vertices wait in buckets of the split width (delta-stepping).
//   2. shortest-path DAG: one walk over the reached vertices keeps the tight
//      entries d(v) + w = d(u) as a compact list per vertex; two bits per
//      vertex tell which vertices have several predecessors.  A second pass
//      over the lists replaces the successors that have no successor and one
//      predecessor by a count: each adds exactly 1 to its predecessor's
//      dependency (sigma(v) * 1 / sigma(v)), so neither its sigma nor its
//      record is ever touched.
//   3. sigma down the DAG in hop-depth levels: a vertex with one predecessor
//      takes its sigma by a plain store, one with several by atomics, and the
//      last predecessor releases it into the next level.
//   4. Algorithm 3 over those levels in reverse: every vertex pulls
//      (1 + delta) / sigma from its listed successors, no atomics but the
//      final add into BC.
// Frontiers and levels that hold a fair share of the vertices are put into
// vertex order (from a bit per vertex), so that neighbouring threads read
// neighbouring records, rows and lists.
//
// Landmark pruning (the triangle inequality on the highest-degree vertex h):
// an entry v -> u of weight w can lie on a shortest path from s only if
//   d(v) + w <= D(s, h) + D(h, u),  i.e.  w - D(h, u) <= D(s, h) - d(v).
// The left side is a constant of the entry, so each row is stored in its order
// and a walk stops at the first entry above D(s, h) - d(v).  An entry on a
// shortest path never fails the test (d(v) + w = d(s, u) <= D(s, h) + D(h, u)),
// so distances, sigma and the DAG are exact.  Same idea as the landmark bounds
// of A* search (Goldberg and Harrelson, SODA 2005), here as a row order.
//
// What bounds it (GB300, per pass; the strict schedule on the same graphs in
// brackets): R-MAT scale 20, 4096 sources: 220 ms (855), 1.0 TB of DRAM traffic
// (3.9) at 0.63-0.67 of the measured bandwidth: random distance gathers of the
// DAG build (35% of the cycles) and of the rounds (22%), 2.2 gathers per DAG edge.
// Barabasi-Albert 65k, 2048 sources: 15 ms (72), 31% DAG build, 40% the passes
// over the lists, latency of their dependent loads.  Erdos-Renyi 262k, 256 sources:
// 39 ms (83): no landmarks, every entry walked 2.2 times; 152 teams hold 256
// sources in two unequal waves.  512 x 512 grid, 512 sources: 32 ms (110): 1530 rounds
// and 2 x 805 levels of ~300 vertices each, ~7 us a round (six dependent L2 round
// trips and a barrier).  1024 vertices in shared memory, 1024 sources: 0.39-0.42 ms
// (0.94): 608 teams for 1024 sources, ~35 steps of ~9 k cycles.
//
// Why these forms (BA 65k / R-MAT scale 20, ms, each against the one before):
// predecessor counts and round stamps by atomics on the records 30.9 / 441; two bits
// per vertex in shared memory instead, frontiers in vertex order, leaves as counts
// 21.1 / 252; rows in tiers of one thread (4 entries), eight lanes (16) and whole
// warps, atomics of one kind issued together 17.1 / 225; folding and lists in the
// same tiers 14.9 / 222 (0 / 1 / 2 / 3 passes: 18.9 / 16.6 / 15.5 / 14.9 and
// 232 / 221 / 222 / 225).  64 landmarks against 8 / 16 / 32: R-MAT 288 / 273 / 260 / 252.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "bc_common.h"
#include "bc_team.cuh"

namespace bcgpu {
namespace {

constexpr int SW_UNR = 4;              // entries in flight per thread
constexpr int SW_STEPS = 4;            // eight threads per row: SW_UNR * SW_STEPS * 8 entries, then whole warps
constexpr uint32_t SW_SECOND = 16;     // one thread per row: FIRST entries, eight threads SW_SECOND more, then whole warps
constexpr int32_t SW_NO_BOUND = 0x7fffffff;  // no entry's test word exceeds it
constexpr uint32_t SW_LIST = 4;        // DAG lists: one thread's work up to this length,
constexpr uint32_t SW_LIST8 = 64;      // ... eight threads' up to this many more, then a warp's
constexpr uint32_t SW_SCAN = 8;        // the pass over the lists before sigma: one thread up to this length
constexpr int SW_FOLDS = 3;            // ... and its repetitions
constexpr uint32_t SW_WARP_MAX = 2048; // longer rows and lists are the whole team's work
constexpr uint32_t SW_TEAM_CAP = 64;   // rows handed to the whole team per pass (the rest stay with a warp)
constexpr uint32_t SW_HEAD = 2;        // words before a DAG list: successors listed, successors counted
constexpr uint32_t SW_ORDER = 64;      // frontiers above n / SW_ORDER are put into vertex order
constexpr uint32_t SW_DEEP = 256;      // ... and levels, and vertices folded, where the distances took fewer rounds
                                       // than this (random and scale-free graphs take 8-62, grids from 32 x 32 on 65;
                                       // folding costs the 512 x 512 grid 10%)

// Where a team's arrays are.
enum : int {
  MEM_GLOBAL = 0,  // the slab
  MEM_BITS = 1,    // the slab, the two bits per vertex in shared memory
  MEM_ALL = 2,     // shared memory
  MEM_CHECK = 3,   // the slab; an undirected graph whose rows are not symmetric: every source is checked
};

// Per-vertex record, one 32-byte sector holds two.  Sigma pass: aux's low
// word counts the predecessors left beyond the last (vertices with several
// predecessors only).  Backward: aux = delta.  Zero between sources.
struct __align__(16) SweepNode {
  double sig;
  unsigned long long aux;
};

template <typename D, int TEAM>
struct SweepShared {
  uint32_t src_idx;
  uint32_t qlen[3];   // next frontier / level lengths, rotating so that one barrier ends a round
  uint32_t nwide[3];  // rows left to whole warps
  uint32_t nteam[3];  // rows left to the whole team
  uint32_t tpos;
  uint32_t S_len, def_len, ndef, dag_len, dag_lists, dag_over, nkeep, nfold;
  unsigned long long cyc[4];
  long long tmark;
  uint32_t team_v[SW_TEAM_CAP], team_e[SW_TEAM_CAP];
  uint32_t land[SWEEP_MAX_LAND];
  D red[2 * (TEAM / 32) + 2];
  uint32_t scan[TEAM / 32 + 1];
  double acc[TEAM / 32];
};

template <typename D, int TEAM, bool PRUNE, int MEM, int G>
struct SweepTeam {
  using Sh = SweepShared<D, TEAM>;
  static constexpr bool SM = MEM == MEM_ALL;
  static constexpr bool CHECK = MEM == MEM_CHECK;
  using Idx = typename std::conditional<SM, uint16_t, uint32_t>::type;
  static constexpr int NW = TEAM / 32;
  static constexpr uint32_t FIRST = 4;  // entries that one thread walks before its warp helps

  const BatchArgs& a;
  Sh& sh;
  const int t;
  D* d;
  SweepNode* node;
  uint32_t* off;     // DAG list of each reached vertex (0: none)
  Idx *qa, *qb, *S, *def, *wide;
  uint32_t* succ;
  uint32_t succ_cap;
  uint32_t *bits0, *bits1;  // one bit per vertex each, zero between sources
  uint32_t* bits2;          // ... has successors (written by the DAG build over all vertices)
  // per source
  uint32_t s;
  int32_t C;      // D(s, h), or SW_NO_BOUND
  uint32_t nrelax, nscan, nreach;
  uint32_t sel;   // rotates over qlen / nwide / nteam
  bool seeded, stream;
  uint64_t width;  // bucket width, all ones = one bucket

  __device__ SweepTeam(const BatchArgs& args, Sh& shared, int thread) : a(args), sh(shared), t(thread) {}

  template <typename T>
  static __device__ __forceinline__ T ld(const T* p) {
    if constexpr (SM) {
      return *reinterpret_cast<const volatile T*>(p);
    } else {
      return ldcg(p);
    }
  }
  static __device__ __forceinline__ SweepNode ld_node(const SweepNode* p) {
    uint4 x;
    if constexpr (SM) x = *reinterpret_cast<const uint4*>(p);
    else x = __ldcg(reinterpret_cast<const uint4*>(p));
    SweepNode r;
    r.sig = __longlong_as_double((long long)((unsigned long long)x.x | ((unsigned long long)x.y << 32)));
    r.aux = (unsigned long long)x.z | ((unsigned long long)x.w << 32);
    return r;
  }
  static __device__ __forceinline__ uint32_t* count_of(SweepNode* p) { return reinterpret_cast<uint32_t*>(p) + 2; }

  static __device__ __forceinline__ uint32_t ld_bits(const uint32_t* p) {
    if constexpr (MEM == MEM_GLOBAL || CHECK) return ldcg(p);
    else return *reinterpret_cast<const volatile uint32_t*>(p);
  }
  static __device__ __forceinline__ bool test_bit(const uint32_t* b, uint32_t v) {
    return (ld_bits(&b[v >> 5]) >> (v & 31)) & 1u;
  }
  static __device__ __forceinline__ bool set_bit(uint32_t* b, uint32_t v) {  // true: it was clear
    const uint32_t m = 1u << (v & 31);
    return !(atomicOr(&b[v >> 5], m) & m);
  }
  static __device__ __forceinline__ void clear_bit(uint32_t* b, uint32_t v) { atomicAnd(&b[v >> 5], ~(1u << (v & 31))); }

  // One slot of a counter per calling thread, one atomic for the lanes that
  // reach it together.
  static __device__ __forceinline__ uint32_t push_pos(uint32_t* ctr) {
    const unsigned m = __activemask();
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(ctr, (uint32_t)__popc(m));
    base = __shfl_sync(m, base, leader);
    return base + __popc(m & ((1u << lane) - 1u));
  }

  // A slot of a counter for every set flag of a converged warp, one atomic for
  // them all, and the values stored there.
  template <int N>
  static __device__ __forceinline__ void push_many(uint32_t* ctr, Idx* out, const bool (&on)[N], const uint32_t (&val)[N]) {
    uint32_t b[N], total = 0;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      b[q] = __ballot_sync(FULL, on[q]);
      total += __popc(b[q]);
    }
    if (total == 0) return;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t pos = 0;
    if (lane == 0) pos = atomicAdd(ctr, total);
    pos = __shfl_sync(FULL, pos, 0);
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if (on[q]) out[pos + __popc(b[q] & below)] = (Idx)val[q];
      pos += __popc(b[q]);
    }
  }

  // The set bits in ascending order into out; CLEAR: and the bits cleared.
  // Every warp takes one contiguous share of the words.  Ends synchronised;
  // returns how many.
  template <bool CLEAR>
  __device__ __forceinline__ uint32_t ordered(uint32_t* bits, Idx* out) {
    const uint32_t words = (a.g.act_n + 31) / 32, lane = threadIdx.x & 31, w = (uint32_t)t >> 5;
    const uint32_t share = ((words + NW - 1) / NW + 31) & ~31u;
    const uint32_t w0 = min(w * share, words), w1 = min(w0 + share, words);
    uint32_t c = 0;
    for (uint32_t i = w0 + lane; i < w1; i += 32) c += __popc(ld_bits(&bits[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    if (lane == 0) sh.scan[w] = c;
    team_sync<TEAM>();
    const uint32_t share_c = lane < NW ? sh.scan[lane] : 0u;
    uint32_t base = lane < w ? share_c : 0u, total = share_c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      base += __shfl_xor_sync(FULL, base, o);
      total += __shfl_xor_sync(FULL, total, o);
    }
    for (uint32_t i0 = w0; i0 < w1; i0 += 32) {
      const uint32_t i = i0 + lane;
      uint32_t x = 0;
      if (i < w1) {
        x = ld_bits(&bits[i]);
        if (CLEAR && x) bits[i] = 0;
      }
      const uint32_t p = __popc(x), inc = warp_incl_scan(p);
      uint32_t pos = base + inc - p;
      while (x) {
        out[pos++] = (Idx)(i * 32 + __ffs(x) - 1);
        x &= x - 1;
      }
      base += __shfl_sync(FULL, inc, 31);
    }
    team_sync<TEAM>();
    return total;
  }

  // ---- row entries ---------------------------------------------------------

  struct Row {
    uint64_t r0;
    uint32_t deg;
    D dv;
    int32_t lim;
  };
  __device__ __forceinline__ Row row_of(uint32_t v) const {
    Row r;
    r.dv = ld(&d[v]);
    r.r0 = __ldg(&a.g.row_ptr[v]);
    r.deg = (uint32_t)(__ldg(&a.g.row_ptr[v + 1]) - r.r0);
    r.lim = PRUNE && C != SW_NO_BOUND ? C - (int32_t)r.dv : SW_NO_BOUND;
    return r;
  }
  // Entry e of the row as {neighbour, weight}; false past the row or its prefix.
  __device__ __forceinline__ bool entry(const Row& r, uint32_t e, uint32_t end, uint2& x) const {
    x = make_uint2(0, 0);
    if (e >= end) return false;
    if constexpr (PRUNE) {
      const uint2 y = __ldg(&a.g.kadj[r.r0 + e]);
      if ((int32_t)y.y > r.lim) return false;
      if (a.g.kw) {
        x = make_uint2(y.x, __ldg(&a.g.kw[r.r0 + e]));
      } else {
        x = make_uint2(y.x & ((1u << a.g.col_bits) - 1u), y.x >> a.g.col_bits);
      }
    } else {
      x = __ldg(&a.g.adj[r.r0 + e]);
    }
    return true;
  }
  __device__ __forceinline__ uint32_t entry_col(uint64_t e) const {
    if constexpr (PRUNE) {
      const uint32_t x = __ldg(&a.g.kadj[e].x);
      return a.g.kw ? x : (x & ((1u << a.g.col_bits) - 1u));
    } else {
      return __ldg(&a.g.adj[e].x);
    }
  }
  // Caller's index of walked entry e (edge output).
  __device__ __forceinline__ uint64_t entry_out(uint64_t e) const {
    if constexpr (PRUNE) return __ldg(&a.g.k2o[e]);
    return a.g.e2o ? __ldg(&a.g.e2o[e]) : (uint32_t)e;
  }
  // First entry at or after lo that the prefix test drops (the rows are in
  // the test's order): a 32-way search by one warp.
  __device__ __forceinline__ uint32_t prefix_end(const Row& r, uint32_t lo) const {
    if constexpr (!PRUNE) return r.deg;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t hi = r.deg;
    while (hi - lo > 32) {
      const uint32_t step = (hi - lo + 31) / 32;
      const uint32_t p = min(lo + (lane + 1) * step - 1, hi - 1);
      const bool pass = (int32_t)__ldg(&a.g.kadj[r.r0 + p].y) <= r.lim;
      const uint32_t c = __popc(__ballot_sync(FULL, pass));
      const uint32_t nlo = min(lo + c * step, hi), nhi = min(lo + (c + 1) * step, hi);
      lo = nlo;
      hi = nhi;
    }
    const bool pass = lo + lane < hi && (int32_t)__ldg(&a.g.kadj[r.r0 + lo + lane].y) <= r.lim;
    return lo + __popc(__ballot_sync(FULL, pass));
  }

  // `lanes` threads (whole warps; this is number l) visit entries [p, end) of
  // a row, SW_UNR each at a time: visit<N>(v, row, ok, x, du, e, step) is
  // called by converged warps with entries e, e + step, ...
  template <typename Visit>
  __device__ __forceinline__ void walk_range(uint32_t v, const Row& r, uint32_t p, uint32_t end, uint32_t l,
                                             uint32_t lanes, Visit&& visit) {
    for (uint32_t b = p + (l & ~31u); b < end; b += lanes * SW_UNR) {
      const uint32_t e0 = b + (l & 31u);
      uint2 x[SW_UNR];
      bool ok[SW_UNR];
#pragma unroll
      for (int q = 0; q < SW_UNR; ++q) ok[q] = entry(r, e0 + q * lanes, end, x[q]);
      D du[SW_UNR];
#pragma unroll
      for (int q = 0; q < SW_UNR; ++q) du[q] = ok[q] ? ld(&d[x[q].x]) : 0;
      visit(v, r, ok, x, du, e0, lanes);
    }
  }

  // Another lane's row.
  static __device__ __forceinline__ Row shfl_row(const Row& r, int src) {
    Row q;
    q.r0 = __shfl_sync(FULL, (unsigned long long)r.r0, src);
    q.deg = __shfl_sync(FULL, r.deg, src);
    q.dv = shfl_d(r.dv, src);
    q.lim = PRUNE ? __shfl_sync(FULL, r.lim, src) : SW_NO_BOUND;
    return q;
  }
  static __device__ __forceinline__ D shfl_d(D x, int src) {
    if constexpr (sizeof(D) == 8) return (D)__shfl_sync(FULL, (unsigned long long)x, src);
    else return __shfl_sync(FULL, x, src);
  }
  // Rows that one warp takes at a time: all 32 lanes' worth, or an even share
  // of a short list, so that no warp idles while another walks long rows.
  static __device__ __forceinline__ uint32_t rows_per_warp(uint32_t len) { return min(32u, (len + NW - 1) / NW); }
  // Lane of the (lane / 8)-th row in m, or -1.
  static __device__ __forceinline__ int tier_row(uint32_t m) {
    for (uint32_t k = (threadIdx.x & 31) >> 3; k > 0; --k) m &= m - 1;
    return m ? __ffs(m) - 1 : -1;
  }

  // Visit every walkable entry of the rows get(0) .. get(len - 1): G = 1: one
  // thread per row for FIRST entries, then eight lanes of its warp for
  // SW_SECOND more; G = 8: eight threads per row.  The rest of longer rows goes
  // to whole warps, and to the whole team above SW_WARP_MAX.  Ends with the
  // team synchronised.
  template <typename Get, typename Visit>
  __device__ __forceinline__ void walk(uint32_t len, Get&& get, Visit&& visit) {
    constexpr uint32_t P0 = G == 1 ? FIRST + SW_SECOND : SW_UNR * SW_STEPS * G;
    const uint32_t lane = threadIdx.x & 31;
    if constexpr (G == 1) {
      const uint32_t rpw = rows_per_warp(len);
      for (uint32_t base = ((uint32_t)t >> 5) * rpw; base < len; base += NW * rpw) {
        const uint32_t v = lane < rpw && base + lane < len ? get(base + lane) : NONE;
        Row r{};
        if (v != NONE) r = row_of(v);
        bool more;
        {
          uint2 x[FIRST];
          bool ok[FIRST];
#pragma unroll
          for (uint32_t q = 0; q < FIRST; ++q) ok[q] = entry(r, q, r.deg, x[q]);
          D du[FIRST];
#pragma unroll
          for (uint32_t q = 0; q < FIRST; ++q) du[q] = ok[q] ? ld(&d[x[q].x]) : 0;
          visit(v, r, ok, x, du, 0u, 1u);
          more = r.deg > FIRST && (!PRUNE || ok[FIRST - 1]);
        }
        uint32_t m = __ballot_sync(FULL, more);
        while (m) {
          const int src = tier_row(m);
          const Row q = shfl_row(r, src < 0 ? 0 : src);
          const uint32_t qv = __shfl_sync(FULL, v, src < 0 ? 0 : src);
          m &= m - 1;
          m &= m - 1;
          m &= m - 1;
          m &= m - 1;
          const uint32_t e = FIRST + (lane & 7);
          uint2 x[2];
          bool ok[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) ok[j] = entry(q, e + 8 * j, src < 0 ? 0u : q.deg, x[j]);
          D du[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) du[j] = ok[j] ? ld(&d[x[j].x]) : 0;
          visit(qv, q, ok, x, du, e, 8u);
          if ((lane & 7) == 7 && ok[1] && q.deg > P0) wide[push_pos(&sh.nwide[sel])] = (Idx)qv;
          __syncwarp();
        }
      }
    } else {
      const uint32_t l = (uint32_t)t % G;
      constexpr uint32_t NG = TEAM / G;
      for (uint32_t base = ((uint32_t)t - lane) / G; base < len; base += NG) {
        const uint32_t i = base + lane / G;
        const uint32_t v = i < len ? get(i) : NONE;
        Row r{};
        if (v != NONE) r = row_of(v);
        uint32_t e0 = l;
#pragma unroll 1
        for (int step = 0; step < SW_STEPS && __any_sync(FULL, e0 - l < r.deg); ++step) {
          uint2 x[SW_UNR];
          bool ok[SW_UNR];
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q) ok[q] = entry(r, e0 + q * G, r.deg, x[q]);
          D du[SW_UNR];
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q) du[q] = ok[q] ? ld(&d[x[q].x]) : 0;
          visit(v, r, ok, x, du, e0, (uint32_t)G);
          e0 += SW_UNR * G;
        }
        if (r.deg > P0 && l == 0) wide[push_pos(&sh.nwide[sel])] = (Idx)v;
        __syncwarp();
      }
    }
    team_sync<TEAM>();
    const uint32_t nw = sh.nwide[sel];
    if (nw) {
      for (uint32_t i = (uint32_t)t >> 5; i < nw; i += NW) {
        const uint32_t v = ld(&wide[i]);
        const Row r = row_of(v);
        const uint32_t end = prefix_end(r, P0);
        if (TEAM > 32 && end - P0 > SW_WARP_MAX) {
          uint32_t pos = 0;
          if (lane == 0) pos = atomicAdd(&sh.nteam[sel], 1u);
          pos = __shfl_sync(FULL, pos, 0);
          if (pos < SW_TEAM_CAP) {
            if (lane == 0) {
              sh.team_v[pos] = v;
              sh.team_e[pos] = end;
            }
            continue;
          }
        }
        walk_range(v, r, P0, end, lane, 32, visit);
      }
      team_sync<TEAM>();
      if constexpr (TEAM > 32) {
        const uint32_t nt = min(sh.nteam[sel], SW_TEAM_CAP);
        for (uint32_t i = 0; i < nt; ++i) {
          const uint32_t v = sh.team_v[i];
          walk_range(v, row_of(v), P0, sh.team_e[i], (uint32_t)t, TEAM, visit);
        }
        if (nt) team_sync<TEAM>();
      }
    }
    rotate();
  }

  // The counters of the pass that just ended are read by every thread until
  // the next barrier; the ones after next are cleared for their use then.
  __device__ __forceinline__ void rotate() {
    sel = sel == 2 ? 0 : sel + 1;
    const uint32_t clear = sel == 2 ? 0 : sel + 1;
    if (t == 0) {
      sh.qlen[clear] = 0;
      sh.nwide[clear] = 0;
      sh.nteam[clear] = 0;
    }
  }

  // ---- 1. distances ---------------------------------------------------------

  // d(v) = min over the landmarks of D(s, l) + D(l, v) (the table holds exact
  // distances; 16-bit words where every sum fits below 0x7fff).
  __device__ __forceinline__ void seed_distances() {
    const uint32_t nl = a.g.nland;
    const uint64_t stride = a.g.land_stride;
    if (a.g.land_bits == 16) {
      const uint16_t* in = static_cast<const uint16_t*>(a.g.land_in);
      for (uint32_t l = t; l < nl; l += TEAM) sh.land[l] = __ldg(&in[l * stride + s]) * 0x10001u;
      team_sync<TEAM>();
      const uint4* tab = static_cast<const uint4*>(a.g.land_out);
      const uint64_t st8 = stride / 8;
      const uint32_t n8 = (a.g.land_n + 7) / 8;
      for (uint32_t b = t; b < n8; b += TEAM) {
        uint32_t m[4] = {0x7fff7fffu, 0x7fff7fffu, 0x7fff7fffu, 0x7fff7fffu};
#pragma unroll 8
        for (uint32_t l = 0; l < nl; ++l) {
          const uint4 x = __ldg(&tab[l * st8 + b]);
          const uint32_t c = sh.land[l];
          m[0] = __viaddmin_u16x2(x.x, c, m[0]);
          m[1] = __viaddmin_u16x2(x.y, c, m[1]);
          m[2] = __viaddmin_u16x2(x.z, c, m[2]);
          m[3] = __viaddmin_u16x2(x.w, c, m[3]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t lo = m[j] & 0xffffu, hi = m[j] >> 16;
          const uint32_t v = b * 8 + 2 * j;
          if (v < a.g.n) d[v] = lo == 0x7fffu ? dinf<D>() : (D)lo;
          if (v + 1 < a.g.n) d[v + 1] = hi == 0x7fffu ? dinf<D>() : (D)hi;
        }
      }
    } else {
      const uint32_t* in = static_cast<const uint32_t*>(a.g.land_in);
      for (uint32_t l = t; l < nl; l += TEAM) sh.land[l] = __ldg(&in[l * stride + s]);
      team_sync<TEAM>();
      const uint32_t* tab = static_cast<const uint32_t*>(a.g.land_out);
      for (uint32_t v = t; v < a.g.land_n; v += TEAM) {
        uint32_t m = 0xffffffffu;
#pragma unroll 8
        for (uint32_t l = 0; l < nl; ++l) {
          // both below 2^31, so the sum of two finite words does not wrap
          const uint32_t x = __ldg(&tab[l * stride + v]), c = sh.land[l];
          if (x != 0xffffffffu && c != 0xffffffffu) m = min(m, x + c);
        }
        d[v] = m == 0xffffffffu ? dinf<D>() : (D)m;
      }
    }
    team_sync<TEAM>();
  }

  __device__ __forceinline__ int distances(uint32_t& rounds, uint32_t& advances) {
    const D INF = dinf<D>();
    D bound = (seeded || width == ~0ull) ? INF : sat_add<D>((D)0, width);
    const uint32_t order_min = TEAM > 32 ? a.g.n / SW_ORDER + TEAM : ~0u;
    uint32_t len = 1;
    Idx *cur = qa, *nxt = qb;
    uint32_t *bcur = bits0, *bnxt = bits1;
    bool sorted = true;  // the current frontier's bits are clear already
    for (;;) {
      ++rounds;
      uint32_t* qn = &sh.qlen[sel];
      Idx* out = nxt;
      walk(len,
           [&](uint32_t i) {
             const uint32_t v = (uint32_t)ld(&cur[i]);
             if (!sorted && (G == 1 || t % G == 0)) clear_bit(bcur, v);
             return v;
           },
           [&](uint32_t, const Row& r, auto& ok, auto& x, auto& du, uint32_t, uint32_t) {
             constexpr int N = sizeof(ok) / sizeof(ok[0]);
             D nd[N], old[N];
             uint32_t u[N];
             bool on[N];
             // the atomics of one kind are all in flight before any is waited for
#pragma unroll
             for (int q = 0; q < N; ++q) {
               nscan += ok[q];
               nd[q] = r.dv + (D)x[q].y;
               u[q] = x[q].x;
               on[q] = ok[q] && nd[q] < du[q];
               nrelax += on[q];
               old[q] = on[q] ? atomic_min_d(&d[u[q]], nd[q]) : 0;
             }
             bool better[N];
#pragma unroll
             for (int q = 0; q < N; ++q) {
               better[q] = on[q] && nd[q] < old[q];
               on[q] = better[q] && nd[q] < bound && set_bit(bnxt, u[q]);
             }
             push_many(qn, out, on, u);
             if (!seeded) {
#pragma unroll
               for (int q = 0; q < N; ++q) on[q] = better[q] && old[q] == INF;
               push_many(&sh.S_len, S, on, u);
               if (bound != INF) {
#pragma unroll
                 for (int q = 0; q < N; ++q) on[q] = on[q] && nd[q] >= bound;
                 push_many(&sh.def_len, def, on, u);
               }
             }
           });
      len = *qn;
      Idx* tq = cur;
      cur = nxt;
      nxt = tq;
      uint32_t* tb = bcur;
      bcur = bnxt;
      bnxt = tb;
      sorted = len >= order_min;
      if (sorted) ordered<true>(bcur, cur);
      while (len == 0) {
        const uint32_t dl = sh.def_len;
        if (dl == 0) return DEV_OK;
        // next bucket: the deferred vertices within one width of the smallest
        D lo = INF, dummy = INF;
        for (uint32_t j = t; j < dl; j += TEAM) {
          const D du = ld(&d[ld(&def[j])]);
          if (du >= bound) lo = dmin(lo, du);
        }
        team_min2<D, TEAM>(lo, dummy, sh.red);
        const D nb = lo == INF ? bound : sat_add<D>(lo, width);
        if (t == 0) sh.ndef = 0;
        team_sync<TEAM>();
        for (uint32_t j = t; j < dl; j += TEAM) {
          const uint32_t u = ld(&def[j]);
          const D du = ld(&d[u]);
          if (du >= bound) {  // below it: already relaxed in an earlier bucket
            if (du < nb) cur[push_pos(&sh.qlen[sel])] = (Idx)u;
            else wide[push_pos(&sh.ndef)] = (Idx)u;
          }
        }
        ++advances;
        team_sync<TEAM>();
        len = sh.qlen[sel];
        const uint32_t kept = sh.ndef;
        tq = def;
        def = wide;
        wide = tq;
        bound = nb;
        sorted = true;  // these carry no bits
        team_sync<TEAM>();
        if (t == 0) {
          sh.def_len = kept;
          sh.qlen[sel] = 0;
        }
        team_sync<TEAM>();
        if ((uint64_t)rounds + advances > a.phase_cap) return DEV_ERR_TIMEOUT;
      }
      if ((uint64_t)rounds + advances > a.phase_cap) {
        if (!sorted)  // the slab's bits go back to zero
          for (uint32_t i = t; i < len; i += TEAM) clear_bit(bcur, ld(&cur[i]));
        team_sync<TEAM>();
        return DEV_ERR_TIMEOUT;
      }
    }
  }

  // ---- 2. shortest-path DAG ----------------------------------------------------

  // u has one more predecessor than its first.
  __device__ __forceinline__ void several(uint32_t u) {
    set_bit(bits1, u);
    atomicAdd(count_of(&node[u]), 1u);
  }
  // A tight entry into u, listed at pos (0: the lists are full).  bits0: u
  // has a predecessor, bits1: several.
  __device__ __forceinline__ void emit(uint64_t e, uint32_t u, uint32_t pos) {
    if (!set_bit(bits0, u)) several(u);
    if (pos != 0) succ[pos] = a.ebc ? (uint32_t)e : u;
  }

  // Reached vertex number i of `count`.
  __device__ __forceinline__ uint32_t reached_count() const { return stream ? (seeded ? a.g.land_n : a.g.act_n) : sh.S_len; }
  __device__ __forceinline__ uint32_t reached_vertex(uint32_t i) const { return stream ? i : (uint32_t)ld(&S[i]); }

  // Tight entries of every reached row as a list.  G threads per row; longer
  // rows by one warp or the whole team in two passes (count, fill).
  __device__ __forceinline__ void build_dag() {
    const D INF = dinf<D>();
    const uint32_t len = reached_count();
    const uint32_t l = (uint32_t)t % G, lane = threadIdx.x & 31;
    constexpr uint32_t NG = TEAM / G;
    for (uint32_t base = 0; base < len; base += NG) {
      const uint32_t i = base + (uint32_t)t / G;
      uint32_t v = i < len ? reached_vertex(i) : NONE;
      Row r{};
      if (v != NONE) {
        r = row_of(v);
        if (r.dv == INF) {
          v = NONE;
          r.deg = 0;
        } else if (l == 0) {
          ++nreach;
        }
      }
      uint32_t mask = 0;
      bool more;
      if constexpr (G == 1) {
        uint2 x[FIRST];
        bool ok[FIRST];
#pragma unroll
        for (uint32_t q = 0; q < FIRST; ++q) ok[q] = entry(r, q, r.deg, x[q]);
        D du[FIRST];
#pragma unroll
        for (uint32_t q = 0; q < FIRST; ++q) du[q] = ok[q] ? ld(&d[x[q].x]) : INF;
#pragma unroll
        for (uint32_t q = 0; q < FIRST; ++q)
          if (ok[q]) {
            ++nscan;
            if (du[q] == r.dv + (D)x[q].y) mask |= 1u << q;
          }
        more = r.deg > FIRST && (!PRUNE || ok[FIRST - 1]);
        uint32_t m = __ballot_sync(FULL, more);
        while (m) {
          const int src = tier_row(m);
          const Row y = shfl_row(r, src < 0 ? 0 : src);
          uint2 z[2];
          bool in[2], fit[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) in[k] = entry(y, FIRST + (lane & 7) + 8 * k, src < 0 ? 0u : y.deg, z[k]);
#pragma unroll
          for (int k = 0; k < 2; ++k) fit[k] = in[k] && ld(&d[z[k].x]) == y.dv + (D)z[k].y;
          nscan += in[0] + in[1];
          const uint32_t f0 = __ballot_sync(FULL, fit[0]), f1 = __ballot_sync(FULL, fit[1]);
          const uint32_t on = __ballot_sync(FULL, (lane & 7) == 7 && in[1] && y.deg > FIRST + SW_SECOND);
          // the rows' own lanes collect their bits
          const uint32_t k = __popc(m & ((1u << lane) - 1u));
          if (((m >> lane) & 1u) && k < 4) {
            mask |= (((f0 >> (8 * k)) & 0xffu) << FIRST) | (((f1 >> (8 * k)) & 0xffu) << (FIRST + 8));
            more = (on >> (8 * k + 7)) & 1u;
          }
          m &= m - 1;
          m &= m - 1;
          m &= m - 1;
          m &= m - 1;
        }
      } else {
        more = r.deg > 0;
        uint32_t e0 = l;
#pragma unroll 1
        for (int step = 0; step < SW_STEPS && more; ++step) {
          uint2 x[SW_UNR];
          bool ok[SW_UNR];
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q) ok[q] = entry(r, e0 + q * G, r.deg, x[q]);
          D du[SW_UNR];
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q) du[q] = ok[q] ? ld(&d[x[q].x]) : INF;
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q)
            if (ok[q]) {
              ++nscan;
              if (du[q] == r.dv + (D)x[q].y) mask |= 1u << (step * SW_UNR + q);
            }
          e0 += SW_UNR * G;
          more = e0 - l < r.deg;
        }
      }
      // every lane of the warp is here: place the lists of the warp's rows
      __syncwarp();
      if (more) {
        mask = 0;
        if (l == 0) wide[push_pos(&sh.nwide[sel])] = (Idx)v;
      }
      __syncwarp();
      const uint32_t c = __popc(mask);
      uint32_t total = c;
#pragma unroll
      for (int o = 1; o < G; o <<= 1) total += __shfl_xor_sync(FULL, total, o);
      const uint32_t head = (l == 0 && total) ? SW_HEAD : 0u;
      const uint32_t inc = warp_incl_scan(c + head);
      uint32_t start = 0;
      const uint32_t wsum = __shfl_sync(FULL, inc, 31);
      const uint32_t has = __ballot_sync(FULL, head != 0);
      if (lane == 31 && wsum) {
        start = atomicAdd(&sh.dag_len, wsum);
        atomicAdd(&sh.dag_lists, __popc(has));
      }
      start = __shfl_sync(FULL, start, 31);
      const bool fits = start + wsum <= succ_cap;
      if (!fits && lane == 0 && wsum) sh.dag_over = 1;
      uint32_t pos = start + inc - (c + head);
      if (l == 0 && v != NONE && !more) off[v] = (head && fits) ? pos : 0u;
      if (head && fits) {
        succ[pos] = total;
        succ[pos + 1] = 0;
      }
      if (G == 1 && stream && lane == 0 && i < len) bits2[i >> 5] = has;
      pos += head;
      while (__any_sync(FULL, mask != 0)) {
        uint32_t e[SW_UNR], u[SW_UNR];
#pragma unroll
        for (int q = 0; q < SW_UNR; ++q) {
          e[q] = mask ? l + (__ffs(mask) - 1) * G : NONE;
          mask &= mask - 1;
        }
#pragma unroll
        for (int q = 0; q < SW_UNR; ++q) u[q] = e[q] != NONE ? entry_col(r.r0 + e[q]) : 0u;
        bool again[SW_UNR];
#pragma unroll
        for (int q = 0; q < SW_UNR; ++q) again[q] = e[q] != NONE && !set_bit(bits0, u[q]);
#pragma unroll
        for (int q = 0; q < SW_UNR; ++q)
          if (e[q] != NONE) {
            if (again[q]) several(u[q]);
            if (fits) succ[pos++] = a.ebc ? (uint32_t)(r.r0 + e[q]) : u[q];
          }
      }
    }
    team_sync<TEAM>();
    const uint32_t nw = sh.nwide[sel];
    for (uint32_t i = (uint32_t)t >> 5; i < nw; i += NW) {
      const uint32_t v = ld(&wide[i]);
      const Row r = row_of(v);
      const uint32_t end = prefix_end(r, 0);
      if (TEAM > 32 && end > SW_WARP_MAX) {
        uint32_t pos = 0;
        if (lane == 0) pos = atomicAdd(&sh.nteam[sel], 1u);
        pos = __shfl_sync(FULL, pos, 0);
        if (pos < SW_TEAM_CAP) {
          if (lane == 0) {
            sh.team_v[pos] = v;
            sh.team_e[pos] = end;
          }
          continue;
        }
      }
      uint32_t c = 0;
      walk_range(v, r, 0, end, lane, 32, [&](uint32_t, const Row& rr, auto& ok, auto& x, auto& du, uint32_t, uint32_t) {
#pragma unroll
        for (int q = 0; q < SW_UNR; ++q) c += ok[q] && du[q] == rr.dv + (D)x[q].y;
      });
      if (lane == 0) nscan += end;
      const uint32_t inc = warp_incl_scan(c);
      const uint32_t total = __shfl_sync(FULL, inc, 31);
      uint32_t start = 0;
      if (lane == 0) {
        if (total) start = atomicAdd(&sh.dag_len, total + SW_HEAD);
        start = list_head(v, start, total);
      }
      start = __shfl_sync(FULL, start, 0);
      uint32_t pos = start ? start + SW_HEAD + inc - c : 0u;
      if (total)
        walk_range(v, r, 0, end, lane, 32, [&](uint32_t, const Row& rr, auto& ok, auto& x, auto& du, uint32_t e, uint32_t step) {
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q)
            if (ok[q] && du[q] == rr.dv + (D)x[q].y) {
              emit(rr.r0 + e + q * step, x[q].x, pos);
              pos += pos != 0;
            }
        });
    }
    if (nw) team_sync<TEAM>();
    if constexpr (TEAM > 32) {
      const uint32_t nt = nw ? min(sh.nteam[sel], SW_TEAM_CAP) : 0u;
      for (uint32_t i = 0; i < nt; ++i) {
        const uint32_t v = sh.team_v[i], end = sh.team_e[i];
        const Row r = row_of(v);
        uint32_t c = 0;
        walk_range(v, r, 0, end, (uint32_t)t, TEAM, [&](uint32_t, const Row& rr, auto& ok, auto& x, auto& du, uint32_t, uint32_t) {
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q) c += ok[q] && du[q] == rr.dv + (D)x[q].y;
        });
        if (t == 0) nscan += end;
        uint32_t total;
        const uint32_t ex = team_excl_scan<TEAM>(c, &total, sh.scan);
        if (t == 0) {
          uint32_t start = 0;
          if (total) start = atomicAdd(&sh.dag_len, total + SW_HEAD);
          sh.tpos = list_head(v, start, total);
        }
        team_sync<TEAM>();
        const uint32_t start = sh.tpos;
        uint32_t pos = start ? start + SW_HEAD + ex : 0u;
        if (total)
          walk_range(v, r, 0, end, (uint32_t)t, TEAM, [&](uint32_t, const Row& rr, auto& ok, auto& x, auto& du, uint32_t e, uint32_t step) {
#pragma unroll
            for (int q = 0; q < SW_UNR; ++q)
              if (ok[q] && du[q] == rr.dv + (D)x[q].y) {
                emit(rr.r0 + e + q * step, x[q].x, pos);
                pos += pos != 0;
              }
          });
        team_sync<TEAM>();
      }
    }
    rotate();
  }
  // One thread: v's list of `total` successors at `start`; 0 when it has none or does not fit.
  __device__ __forceinline__ uint32_t list_head(uint32_t v, uint32_t start, uint32_t total) {
    if (total) atomicAdd(&sh.dag_lists, 1u);
    if (total && start + total + SW_HEAD > succ_cap) {
      sh.dag_over = 1;
      total = 0;
    }
    if (total) {
      succ[start] = total;
      succ[start + 1] = 0;
    }
    off[v] = total ? start : 0u;
    if (G == 1 && stream && total) atomicOr(&bits2[v >> 5], 1u << (v & 31));
    return total ? start : 0u;
  }

  // 32-bit finaliser of MurmurHash3 (A. Appleby, public domain).
  static __device__ __forceinline__ uint32_t hash(uint32_t x) {
    x = (x ^ (x >> 16)) * 0x85ebca6bu;
    x = (x ^ (x >> 13)) * 0xc2b2ae35u;
    return x ^ (x >> 16);
  }
  // Whether every reached vertex has as many predecessors by its own row
  // (d(u) + w = d(v)) as by theirs (the DAG): the sums of a hash of each DAG edge's
  // target, taken both ways.  An entry on a shortest path without a reverse
  // entry makes them differ.  Ends synchronised.
  __device__ bool rows_agree() {
    const D INF = dinf<D>();
    if (t == 0) sh.tpos = 0;
    team_sync<TEAM>();
    uint32_t sum = 0;
    walk(reached_count(),
         [&](uint32_t i) {
           const uint32_t v = reached_vertex(i);
           return ld(&d[v]) == INF ? NONE : v;
         },
         [&](uint32_t v, const Row& r, auto& ok, auto& x, auto& du, uint32_t, uint32_t) {
           constexpr int N = sizeof(ok) / sizeof(ok[0]);
#pragma unroll
           for (int q = 0; q < N; ++q) {
             if (!ok[q] || du[q] == INF) continue;
             if (du[q] == r.dv + (D)x[q].y) sum += hash(x[q].x);
             if (du[q] + (D)x[q].y == r.dv) sum -= hash(v);
           }
         });
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
    if ((t & 31) == 0) atomicAdd(&sh.tpos, sum);
    team_sync<TEAM>();
    const bool agree = sh.tpos == 0;
    team_sync<TEAM>();
    return agree;
  }

  // Replace the listed successors that have no successor themselves and one
  // predecessor by a count; then fold, a few times over: a vertex with one
  // predecessor whose successors are all counted has its dependency (the
  // count), so it goes into BC and its predecessor counts it too.  bits0
  // becomes "has successors and is not folded" on the way and is zero at the
  // end.
  __device__ __forceinline__ void drop_leaves(int folds) {
    const uint32_t lane = threadIdx.x & 31, all = reached_count();
    // the vertices with successors: as bits, and as a list in vertex order
    uint32_t len = all;
    if (stream) {
      if (G == 1) {
        for (uint32_t w = t; w < (all + 31) / 32; w += TEAM) bits0[w] = ld(&bits2[w]);
      } else {
        for (uint32_t base = (uint32_t)t & ~31u; base < all; base += TEAM) {
          const uint32_t v = base + lane;
          const bool has = v < all && (test_bit(bits0, v) || v == s) && ld(&off[v]) != 0;
          const uint32_t m = __ballot_sync(FULL, has);
          if (lane == 0) bits0[base >> 5] = m;
        }
      }
      team_sync<TEAM>();
      len = ordered<false>(bits0, S);
    } else {
      for (uint32_t i = t; i < all; i += TEAM) {
        const uint32_t v = ld(&S[i]);
        if (ld(&off[v]) == 0) clear_bit(bits0, v);
      }
      team_sync<TEAM>();
    }
    const Idx* list = S;
    Idx *keep = qa, *spare = qb;
    for (int pass = 0;; ++pass) {
      if (t == 0) sh.nkeep = sh.nfold = 0;
      team_sync<TEAM>();
      const bool last = pass >= folds;
      for (uint32_t base = (uint32_t)t - lane; base < len; base += TEAM) {
        const uint32_t i = base + lane;
        uint32_t v = 0, o = 0, n = 0;
        if (i < len) {
          v = ld(&list[i]);
          o = ld(&off[v]);
          if (o) n = ld(&succ[o]);
        }
        if (n > SW_SCAN) {
          wide[push_pos(&sh.nwide[sel])] = (Idx)v;
          n = 0;
        }
        uint32_t kept = 0, gone = 0;
        for (uint32_t j0 = 0; j0 < n; j0 += SW_UNR) {
          uint32_t x[SW_UNR];
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q) x[q] = j0 + q < n ? ld(&succ[o + SW_HEAD + j0 + q]) : NONE;
#pragma unroll
          for (int q = 0; q < SW_UNR; ++q)
            if (x[q] != NONE) {
              if (listed(x[q])) {
                if (kept != j0 + q) succ[o + SW_HEAD + kept] = x[q];
                ++kept;
              } else {
                gone += counted(x[q], pass);
              }
            }
        }
        if (kept != n) {
          succ[o] = kept;
          succ[o + 1] = pass == 0 ? gone : gone + ld(&succ[o + 1]);
        }
        __syncwarp();
        if (!last) {
          const bool fold[1] = {n > 0 && kept == 0 && v != s && !test_bit(bits1, v)};
          const bool stay[1] = {kept > 0};
          const uint32_t val[1] = {v};
          push_many(&sh.nfold, def, fold, val);
          push_many(&sh.nkeep, keep, stay, val);
        }
      }
      team_sync<TEAM>();
      const uint32_t nw = sh.nwide[sel];
      for (uint32_t i = (uint32_t)t >> 5; i < nw; i += NW) {
        const uint32_t v = ld(&wide[i]);
        const uint32_t o = ld(&off[v]);
        const uint32_t n = ld(&succ[o]);
        uint32_t kept = 0, gone = 0;
        for (uint32_t j0 = 0; j0 < n; j0 += 128) {
          uint32_t x[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = j0 + q * 32 + lane < n ? ld(&succ[o + SW_HEAD + j0 + q * 32 + lane]) : NONE;
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const bool stays = x[q] != NONE && listed(x[q]);
            if (x[q] != NONE && !stays) gone += counted(x[q], pass);
            const uint32_t m = __ballot_sync(FULL, stays);
            if (stays) succ[o + SW_HEAD + kept + __popc(m & ((1u << lane) - 1u))] = x[q];
            kept += __popc(m);
          }
          __syncwarp();
        }
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) gone += __shfl_xor_sync(FULL, gone, k);
        if (lane == 0) {
          succ[o] = kept;
          succ[o + 1] += gone;
          if (!last) {
            if (kept) keep[atomicAdd(&sh.nkeep, 1u)] = (Idx)v;
            else if (v != s && !test_bit(bits1, v)) def[atomicAdd(&sh.nfold, 1u)] = (Idx)v;
          }
        }
      }
      if (nw) team_sync<TEAM>();
      rotate();
      const uint32_t nf = sh.nfold;
      // one more pass only where it removes a fair share of what is left
      if (last || nf < len / 12) break;
      for (uint32_t i = t; i < nf; i += TEAM) {
        const uint32_t v = ld(&def[i]);
        clear_bit(bits0, v);
        add_bc(v, (double)ld(&succ[ld(&off[v]) + 1]));
      }
      len = sh.nkeep;
      list = keep;
      Idx* tmp = keep;
      keep = spare;
      spare = tmp;
      team_sync<TEAM>();
    }
    team_sync<TEAM>();
    clear_bits0();
  }
  __device__ __forceinline__ uint32_t succ_vertex(uint32_t x) const { return a.ebc ? entry_col(x) : x; }
  __device__ __forceinline__ void add_bc(uint32_t v, double delta) {
    atomicAdd(&a.bc[a.g.n2o ? __ldg(&a.g.n2o[v]) : v], delta);
  }
  // Whether list word x stays listed: its vertex has several predecessors, or
  // successors of its own that are not folded.
  __device__ __forceinline__ bool listed(uint32_t x) const {
    const uint32_t u = succ_vertex(x);
    return test_bit(bits1, u) || test_bit(bits0, u);
  }
  // What a word leaving its list adds to the dependency: its vertex, and on
  // later passes (where it is a folded one) what was counted below it.
  __device__ __forceinline__ uint32_t counted(uint32_t x, int pass) {
    const uint32_t c = pass == 0 ? 1u : 1u + ld(&succ[ld(&off[succ_vertex(x)]) + 1]);
    if (a.ebc) atomicAdd(&a.ebc[entry_out(x)], (double)c);
    return c;
  }
  // bits0 back to zero (it holds reached vertices only).  Ends synchronised.
  __device__ __forceinline__ void clear_bits0() {
    const uint32_t len = reached_count();
    if (stream) {
      for (uint32_t w = t; w < (len + 31) / 32; w += TEAM) bits0[w] = 0;
    } else {
      for (uint32_t i = t; i < len; i += TEAM) bits0[ld(&S[i]) >> 5] = 0;
    }
    team_sync<TEAM>();
  }

  // ---- 3. sigma ----------------------------------------------------------------

  // One predecessor of u is done.  Returns true when it was the last, with
  // u's record ready for the levels below (aux = 0).
  __device__ __forceinline__ bool release(uint32_t u, double sv, bool multi) {
    if (!multi) {
      node[u].sig = sv;
      return true;
    }
    atomicAdd(&node[u].sig, sv);
    if (atomicSub(count_of(&node[u]), 1u) != 0u) return false;
    node[u].aux = 0ull;
    return true;
  }

  // Levels of the DAG from the source; order holds them back to back, lvl
  // their bounds.  A vertex without successors needs no level of its own
  // unless `all` asks for it.  Returns the number of levels.
  __device__ __forceinline__ uint32_t sigma_levels(Idx* order, Idx* lvl, bool rows, bool all, bool shallow) {
    if (t == 0) {
      node[s].sig = 1.0;
      order[0] = (Idx)s;
      lvl[0] = 0;
      lvl[1] = 1;
    }
    team_sync<TEAM>();
    const uint32_t order_min = (TEAM > 32 && shallow) ? a.g.n / (4 * SW_ORDER) + TEAM : ~0u;
    uint32_t nlev = 1, l0 = 0, l1 = 1;
    for (;;) {
      uint32_t* qn = &sh.qlen[sel];
      Idx* out = order + l1;
      // successors u of converged warps, each with its predecessor's sigma
      auto push = [&](auto& on, auto& u, double sv) {
        constexpr int N = sizeof(on) / sizeof(on[0]);
        bool look[N];
#pragma unroll
        for (int q = 0; q < N; ++q) {
          const bool multi = on[q] && test_bit(bits1, u[q]);
          // after drop_leaves a listed successor with one predecessor has successors itself; of the
          // others, look
          look[q] = !all && multi;
          if (on[q]) on[q] = release(u[q], sv, multi);
        }
#pragma unroll
        for (int q = 0; q < N; ++q) {
          if (on[q] && look[q]) on[q] = ld(&off[u[q]]) != 0;
          if (on[q] && shallow) set_bit(bits0, u[q]);
        }
        push_many(qn, out, on, u);
      };
      if (rows) {
        walk(l1 - l0, [&](uint32_t i) { return (uint32_t)ld(&order[l0 + i]); },
             [&](uint32_t v, const Row& r, auto& ok, auto& x, auto& du, uint32_t, uint32_t) {
               constexpr int N = sizeof(ok) / sizeof(ok[0]);
               bool on[N];
               uint32_t u[N];
               bool any = false;
#pragma unroll
               for (int q = 0; q < N; ++q) {
                 on[q] = ok[q] && du[q] == r.dv + (D)x[q].y;
                 u[q] = x[q].x;
                 any |= on[q];
               }
               push(on, u, any ? ld(&node[v].sig) : 0.0);
             });
      } else {
        const uint32_t lane = threadIdx.x & 31, rpw = rows_per_warp(l1 - l0);
        for (uint32_t b = l0 + ((uint32_t)t >> 5) * rpw; b < l1; b += NW * rpw) {
          uint32_t v = 0, o = 0, len = 0;
          double sv = 0.0;
          if (lane < rpw && b + lane < l1) {
            v = ld(&order[b + lane]);
            o = ld(&off[v]);
            sv = ld(&node[v].sig);
            if (o) len = ld(&succ[o]);
          }
          if (len > SW_LIST + SW_LIST8) {
            wide[push_pos(&sh.nwide[sel])] = (Idx)v;
            len = 0;
          }
          __syncwarp();
          if (__any_sync(FULL, len > 0)) {
            bool on[SW_LIST];
            uint32_t u[SW_LIST];
#pragma unroll
            for (uint32_t q = 0; q < SW_LIST; ++q) {
              on[q] = q < len;
              u[q] = on[q] ? succ_vertex(ld(&succ[o + SW_HEAD + q])) : 0u;
            }
            push(on, u, sv);
          }
          uint32_t m = __ballot_sync(FULL, len > SW_LIST);
          while (m) {
            const int src = tier_row(m);
            const uint32_t qo = __shfl_sync(FULL, o, src < 0 ? 0 : src);
            uint32_t ql = __shfl_sync(FULL, len, src < 0 ? 0 : src);
            const double qs = __shfl_sync(FULL, sv, src < 0 ? 0 : src);
            if (src < 0) ql = 0;
            for (uint32_t k = SW_LIST + (lane & 7); __any_sync(FULL, k < ql); k += 16) {
              bool on[2];
              uint32_t u[2];
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                on[q] = k + 8 * q < ql;
                u[q] = on[q] ? succ_vertex(ld(&succ[qo + SW_HEAD + k + 8 * q])) : 0u;
              }
              push(on, u, qs);
            }
            m &= m - 1;
            m &= m - 1;
            m &= m - 1;
            m &= m - 1;
          }
        }
        team_sync<TEAM>();
        wide_lists([&](uint32_t v, uint32_t o, uint32_t len, uint32_t l, uint32_t lanes) {
          const double sv = ld(&node[v].sig);
          for (uint32_t b = l & ~31u; b < len; b += lanes * SW_UNR) {
            bool on[SW_UNR];
            uint32_t u[SW_UNR];
#pragma unroll
            for (int q = 0; q < SW_UNR; ++q) {
              const uint32_t j = b + (l & 31u) + q * lanes;
              on[q] = j < len;
              u[q] = on[q] ? succ_vertex(ld(&succ[o + SW_HEAD + j])) : 0u;
            }
            push(on, u, sv);
          }
        });
        rotate();
      }
      const uint32_t next = *qn;
      if (next == 0) break;
      if (shallow) {
        if (next >= order_min) {
          ordered<true>(bits0, order + l1);
        } else {
          for (uint32_t i = t; i < next; i += TEAM) clear_bit(bits0, ld(&order[l1 + i]));
        }
      }
      ++nlev;
      l0 = l1;
      l1 += next;
      if (t == 0) lvl[nlev] = (Idx)l1;
    }
    team_sync<TEAM>();
    return nlev;
  }

  // The vertices in the wide list with their DAG lists: one warp each, the
  // whole team for lists above SW_WARP_MAX.  Ends synchronised.
  template <typename F>
  __device__ __forceinline__ void wide_lists(F&& f) {
    const uint32_t nw = sh.nwide[sel];
    if (nw == 0) return;
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t i = (uint32_t)t >> 5; i < nw; i += NW) {
      const uint32_t v = ld(&wide[i]);
      const uint32_t o = ld(&off[v]);
      const uint32_t len = ld(&succ[o]);
      if (TEAM > 32 && len > SW_WARP_MAX) {
        uint32_t pos = 0;
        if (lane == 0) pos = atomicAdd(&sh.nteam[sel], 1u);
        pos = __shfl_sync(FULL, pos, 0);
        if (pos < SW_TEAM_CAP) {
          if (lane == 0) sh.team_v[pos] = v;
          continue;
        }
      }
      f(v, o, len, lane, 32u);
    }
    team_sync<TEAM>();
    if constexpr (TEAM > 32) {
      const uint32_t nt = min(sh.nteam[sel], SW_TEAM_CAP);
      for (uint32_t i = 0; i < nt; ++i) {
        const uint32_t v = sh.team_v[i];
        const uint32_t o = ld(&off[v]);
        f(v, o, ld(&succ[o]), (uint32_t)t, (uint32_t)TEAM);
      }
      if (nt) team_sync<TEAM>();
    }
  }

  // ---- 4. dependencies -----------------------------------------------------------

  // c(u) = (1 + delta(u)) / sigma(u); most vertices have one shortest path.
  static __device__ __forceinline__ double coeff(const SweepNode& u) {
    const double x = 1.0 + __longlong_as_double((long long)u.aux);
    return u.sig == 1.0 ? x : x / u.sig;
  }
  __device__ __forceinline__ void finish(uint32_t v, double delta) {
    node[v].aux = (unsigned long long)__double_as_longlong(delta);
    if (v != s) add_bc(v, delta);
  }
  __device__ __forceinline__ double pull(uint32_t x, const SweepNode& u, double sig) {
    const double c = coeff(u);
    if (a.ebc) atomicAdd(&a.ebc[entry_out(x)], sig * c);
    return c;
  }

  __device__ __forceinline__ void dependencies(const Idx* order, const Idx* lvl, uint32_t nlev, bool rows) {
    const int last = a.ebc ? 0 : 1;
    uint32_t b1 = ld(&lvl[nlev]);
    for (int lev = (int)nlev - 1; lev >= last; --lev) {
      const uint32_t b0 = ld(&lvl[lev]);
      if (rows) {
        // the sums collect in aux (zero after the sigma pass)
        walk(b1 - b0, [&](uint32_t i) { return (uint32_t)ld(&order[b0 + i]); },
             [&](uint32_t v, const Row& r, auto& ok, auto& x, auto& du, uint32_t e, uint32_t step) {
               constexpr int N = sizeof(ok) / sizeof(ok[0]);
#pragma unroll
               for (int q = 0; q < N; ++q)
                 if (ok[q] && du[q] == r.dv + (D)x[q].y) {
                   const double c = coeff(ld_node(&node[x[q].x]));
                   atomicAdd(reinterpret_cast<double*>(&node[v].aux), c);
                   if (a.ebc) atomicAdd(&a.ebc[entry_out(r.r0 + e + q * step)], ld(&node[v].sig) * c);
                 }
             });
        for (uint32_t i = b0 + t; i < b1; i += TEAM) {
          const uint32_t v = ld(&order[i]);
          const SweepNode nd = ld_node(&node[v]);
          if (nd.aux) finish(v, nd.sig * __longlong_as_double((long long)nd.aux));
        }
        team_sync<TEAM>();
      } else {
        const uint32_t lane = threadIdx.x & 31, rpw = rows_per_warp(b1 - b0);
        for (uint32_t b = b0 + ((uint32_t)t >> 5) * rpw; b < b1; b += NW * rpw) {
          uint32_t v = 0, o = 0, len = 0, below = 0;
          double sig = 0.0, acc = 0.0;
          if (lane < rpw && b + lane < b1) {
            v = ld(&order[b + lane]);
            o = ld(&off[v]);
            sig = ld(&node[v].sig);
            if (o) {
              len = ld(&succ[o]);
              below = ld(&succ[o + 1]);
            }
          }
          if (len > SW_LIST + SW_LIST8) {
            wide[push_pos(&sh.nwide[sel])] = (Idx)v;
            len = o = 0;
          }
          __syncwarp();
          {
            uint32_t x[SW_LIST];
#pragma unroll
            for (uint32_t q = 0; q < SW_LIST; ++q) x[q] = q < len ? ld(&succ[o + SW_HEAD + q]) : NONE;
#pragma unroll
            for (uint32_t h = 0; h < SW_LIST; h += 2) {
              SweepNode u0{1.0, 0ull}, u1{1.0, 0ull};
              if (h < len) u0 = ld_node(&node[succ_vertex(x[h])]);
              if (h + 1 < len) u1 = ld_node(&node[succ_vertex(x[h + 1])]);
              if (h < len) acc += pull(x[h], u0, sig);
              if (h + 1 < len) acc += pull(x[h + 1], u1, sig);
            }
          }
          uint32_t m = __ballot_sync(FULL, len > SW_LIST);
          while (m) {
            const int src = tier_row(m);
            const uint32_t qo = __shfl_sync(FULL, o, src < 0 ? 0 : src);
            uint32_t ql = __shfl_sync(FULL, len, src < 0 ? 0 : src);
            const double qs = __shfl_sync(FULL, sig, src < 0 ? 0 : src);
            if (src < 0) ql = 0;
            double part = 0.0;
            for (uint32_t k = SW_LIST + (lane & 7); k < ql; k += 8) {
              const uint32_t x = ld(&succ[qo + SW_HEAD + k]);
              part += pull(x, ld_node(&node[succ_vertex(x)]), qs);
            }
            __syncwarp();
#pragma unroll
            for (int k = 4; k > 0; k >>= 1) part += __shfl_xor_sync(FULL, part, k);
            // the lists' own lanes collect their sums
            const uint32_t k = __popc(m & ((1u << lane) - 1u));
            part = __shfl_sync(FULL, part, (k & 3) * 8);
            if (((m >> lane) & 1u) && k < 4) acc += part;
            m &= m - 1;
            m &= m - 1;
            m &= m - 1;
            m &= m - 1;
          }
          if (o) finish(v, sig * acc + (double)below);
        }
        team_sync<TEAM>();
        wide_lists([&](uint32_t v, uint32_t o, uint32_t len, uint32_t l, uint32_t lanes) {
          const double sig = ld(&node[v].sig);
          double acc = 0.0;
          for (uint32_t j = l; j < len; j += lanes) {
            const uint32_t x = ld(&succ[o + SW_HEAD + j]);
            acc += pull(x, ld_node(&node[succ_vertex(x)]), sig);
          }
#pragma unroll
          for (int k = 16; k > 0; k >>= 1) acc += __shfl_xor_sync(FULL, acc, k);
          if (TEAM > 32 && lanes > 32) {
            if ((t & 31) == 0) sh.acc[t >> 5] = acc;
            team_sync<TEAM>();
            if (t == 0) {
              acc = 0.0;
              for (int w = 0; w < NW; ++w) acc += sh.acc[w];
              finish(v, sig * acc + (double)ld(&succ[o + 1]));
            }
            team_sync<TEAM>();
          } else if (l == 0) {
            finish(v, sig * acc + (double)ld(&succ[o + 1]));
          }
        });
        rotate();
      }
      b1 = b0;
    }
    team_sync<TEAM>();
  }

  // ---- one source -----------------------------------------------------------------

  __device__ __forceinline__ void lap(int section) {
    if (t == 0) {
      const long long now = clock64();
      sh.cyc[section] += (unsigned long long)(now - sh.tmark);
      sh.tmark = now;
    }
  }

  __device__ __forceinline__ void fill_distances() {
    for (uint32_t v = t; v < a.g.n; v += TEAM) d[v] = dinf<D>();
  }

  // Records back to zero: the vertices in the levels and those with several
  // predecessors (bits1, cleared too); every reached one where the lists
  // keep them all.
  __device__ __forceinline__ void clear_records(const Idx* order, uint32_t count, bool every) {
    const SweepNode zero{0.0, 0ull};
    const uint32_t len = reached_count();
    if (every) {
      for (uint32_t i = t; i < len; i += TEAM) node[reached_vertex(i)] = zero;
    } else {
      for (uint32_t i = t; i < count; i += TEAM) node[ld(&order[i])] = zero;
    }
    if (stream) {
      for (uint32_t w = t; w < (len + 31) / 32; w += TEAM) {
        uint32_t x = ld_bits(&bits1[w]);
        if (x == 0) continue;
        bits1[w] = 0;
        while (x && !every) {
          node[w * 32 + __ffs(x) - 1] = zero;
          x &= x - 1;
        }
      }
    } else {
      for (uint32_t i = t; i < len; i += TEAM) {
        const uint32_t v = ld(&S[i]);
        if (!every && test_bit(bits1, v)) node[v] = zero;
      }
      team_sync<TEAM>();
      for (uint32_t i = t; i < len; i += TEAM) bits1[ld(&S[i]) >> 5] = 0;
    }
  }

  // A source without entries (outside the vertex bits): it reaches itself.
  __device__ __forceinline__ bool run_alone(uint32_t idx) {
    if (a.flags & RUN_DIST_ONLY) {
      uint32_t* out = a.dist_out + (uint64_t)idx * a.g.n;
      for (uint32_t v = t; v < a.g.n; v += TEAM) out[v] = v == s ? 0u : 0xffffffffu;
    }
    if (t == 0) {
      if (a.flags & RUN_FORWARD_ONLY) {
        d[s] = 0;
        node[s].sig = 1.0;
        qa[0] = (Idx)s;
        qb[0] = 0;
        qb[1] = 1;
        if (a.debug_out) a.debug_out[0] = a.debug_out[1] = 1;
      }
      if (a.stats) {
        atomicAdd(&a.stats[STAT_SOURCES], 1ull);
        atomicAdd(&a.stats[STAT_REACHED], 1ull);
        atomicAdd(&a.stats[STAT_LEVELS], 1ull);
      }
    }
    return !(a.flags & RUN_FORWARD_ONLY);
  }

  // Returns false when the run stops here (a cap hit or the test hook).
  __device__ bool run(uint32_t source, uint32_t idx, bool& dirty) {
    const D INF = dinf<D>();
    s = source;
    if (s >= a.g.act_n) return run_alone(idx);
    nrelax = nscan = nreach = 0;
    C = SW_NO_BOUND;
    bool in_land = false;
    if constexpr (PRUNE) {
      uint32_t c;
      if (a.g.land_bits == 16) {
        c = __ldg(static_cast<const uint16_t*>(a.g.land_in) + s);
        in_land = c != 0x7fffu;
      } else {
        c = __ldg(static_cast<const uint32_t*>(a.g.land_in) + s);
        in_land = c != 0xffffffffu;
      }
      if (in_land) C = (int32_t)c;  // a source that does not reach the landmark walks whole rows
    }
    seeded = PRUNE && in_land && width == ~0ull;
    if (dirty && !seeded) {
      fill_distances();
      dirty = false;
      team_sync<TEAM>();
    }
    if (t == 0) {
      sh.S_len = seeded ? 0u : 1u;
      sh.def_len = 0;
      sh.dag_len = 1;  // offset 0 means no list
      sh.dag_lists = 0;
      sh.dag_over = 0;
      sh.cyc[0] = sh.cyc[1] = sh.cyc[2] = sh.cyc[3] = 0;
      sh.tmark = clock64();
      qa[0] = (Idx)s;
      S[0] = (Idx)s;
    }
    if (seeded) {
      seed_distances();
      dirty = true;
    }
    if (t == 0) d[s] = 0;
    team_sync<TEAM>();
    lap(0);
    uint32_t rounds = 0, advances = 0, nlev = 0;
    int err = distances(rounds, advances);
    lap(1);
    const uint32_t reached = seeded ? 0u : sh.S_len;
    stream = seeded || reached > a.g.n / 2;
    const bool dist_only = (a.flags & RUN_DIST_ONLY) != 0;
    bool over = false, every = false;
    if (err == DEV_OK && !dist_only) {
      build_dag();
      team_sync<TEAM>();
      over = sh.dag_over != 0;
      if constexpr (CHECK) {
        if (!rows_agree()) err = DEV_ERR_INTERNAL;
      }
      const bool all = over || (a.flags & RUN_FORWARD_ONLY);
      const bool drop = !all && (!CHECK || err == DEV_OK);
      every = !drop;
      if (drop) {
        drop_leaves(rounds < SW_DEEP ? SW_FOLDS : 0);
      } else {
        clear_bits0();
      }
      lap(0);
      if (!CHECK || err == DEV_OK) nlev = sigma_levels(qa, qb, over, all, rounds < SW_DEEP);
      lap(2);
      if (a.phase_cap < (uint64_t)rounds + advances + nlev) err = DEV_ERR_TIMEOUT;
      if (a.flags & RUN_FORWARD_ONLY) {
        if (t == 0 && a.debug_out) {
          a.debug_out[0] = nlev;
          a.debug_out[1] = ld(&qb[nlev]);
        }
      } else if (err == DEV_OK) {
        dependencies(qa, qb, nlev, over);
        lap(3);
      }
      if (a.flags & RUN_FORWARD_ONLY) {
        // the caller reads the slab and restores distances and records
        const uint32_t words = (a.g.act_n + 31) / 32;
        for (uint32_t w = t; w < words; w += TEAM) bits1[w] = 0;
        if (err != DEV_OK && t == 0) atomicCAS(a.err, DEV_OK, err);
        return false;
      }
      clear_records(qa, nlev ? (uint32_t)ld(&qb[nlev]) : 0u, every);
    }
    if (err == DEV_OK && dist_only) {
      uint32_t* out = a.dist_out + (uint64_t)idx * a.g.n;
      for (uint32_t v = t; v < a.g.n; v += TEAM) out[v] = (uint32_t)ld(&d[v]);
      team_sync<TEAM>();
    }
    if (err != DEV_OK && t == 0) atomicCAS(a.err, DEV_OK, err);
    // distances back to INF (seeded ones are overwritten by the next seeds)
    if (!seeded) {
      if (stream) {
        for (uint32_t v = t; v < a.g.n; v += TEAM) d[v] = INF;
      } else {
        for (uint32_t i = t; i < reached; i += TEAM) d[ld(&S[i])] = INF;
      }
    }
    if (a.stats) {
      unsigned long long relax = nrelax, scanned = nscan, seen = nreach;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        relax += __shfl_xor_sync(FULL, relax, o);
        scanned += __shfl_xor_sync(FULL, scanned, o);
        seen += __shfl_xor_sync(FULL, seen, o);
      }
      if ((t & 31) == 0) {
        atomicAdd(&a.stats[STAT_RELAX], relax);
        atomicAdd(&a.stats[STAT_ENTRIES], scanned);
        atomicAdd(&a.stats[STAT_REACHED], seen);
      }
      if (t == 0) {
        atomicAdd(&a.stats[STAT_SOURCES], 1ull);
        atomicAdd(&a.stats[STAT_PHASES], (unsigned long long)rounds);
        atomicAdd(&a.stats[STAT_REFILLS], (unsigned long long)advances);
        atomicAdd(&a.stats[STAT_DAG_EDGES], (unsigned long long)(sh.dag_len - 1 - SW_HEAD * sh.dag_lists));
        atomicAdd(&a.stats[STAT_LEVELS], (unsigned long long)nlev);
        atomicAdd(&a.stats[STAT_PAIR_OVERFLOW], (unsigned long long)(over ? 1 : 0));
        atomicAdd(&a.stats[STAT_CYC_EXPAND], sh.cyc[1]);
        atomicAdd(&a.stats[STAT_CYC_REFILL], sh.cyc[0]);
        atomicAdd(&a.stats[STAT_CYC_SETTLE], sh.cyc[2]);
        atomicAdd(&a.stats[STAT_CYC_BACKWARD], sh.cyc[3]);
      }
    }
    team_sync<TEAM>();
    return err == DEV_OK;
  }
};

// Resident CTAs per SM that the register budget is compiled for: 64 registers
// per thread, as in the strict kernel (a 64-bit distance word gets 7/8).
template <typename D, int TEAM, int BLOCK>
__host__ __device__ constexpr int sweep_min_blocks() {
  return TEAM == 32 ? 2 : (sizeof(D) == 4 ? 1024 / BLOCK : (BLOCK <= 256 ? 896 / BLOCK : 1024 / BLOCK));
}

template <typename D, int TEAM, int BLOCK, bool PRUNE, int MEM, int G>
__global__ void __launch_bounds__(BLOCK, (sweep_min_blocks<D, TEAM, BLOCK>())) bc_sweep_kernel(const BatchArgs a) {
  static_assert(TEAM == 32 || TEAM == BLOCK, "a CTA holds either warp teams or one team");
  constexpr bool SM = MEM == MEM_ALL, SMEM = SM || MEM == MEM_BITS;
  static_assert(!SMEM || TEAM == BLOCK, "the shared-memory forms hold one team per CTA");
  constexpr int NTEAMS = BLOCK / TEAM;
  __shared__ SweepShared<D, TEAM> shared_teams[NTEAMS];
  extern __shared__ __align__(16) unsigned char sweep_arrays[];
  using T = SweepTeam<D, TEAM, PRUNE, MEM, G>;
  using Idx = typename T::Idx;
  const int team = threadIdx.x / TEAM;
  const int t = threadIdx.x % TEAM;
  const uint32_t slot = blockIdx.x * NTEAMS + team;
  if (slot >= a.nslots) return;  // a whole team leaves together
  SweepShared<D, TEAM>& sh = shared_teams[team];
  T w(a, sh, t);
  w.sel = 0;
  w.width = a.width_dev ? (uint64_t)__ldg(a.width_dev) : a.width;
  if (t < 3) sh.qlen[t] = sh.nwide[t] = sh.nteam[t] = 0;
  bool dirty = false;
  const uint32_t words = (a.g.act_n + 31) / 32;
  char* base = SM ? reinterpret_cast<char*>(sweep_arrays) : a.slabs + (uint64_t)slot * a.lay.stride;
  w.d = reinterpret_cast<D*>(base + a.lay.off_d);
  w.node = reinterpret_cast<SweepNode*>(base + a.lay.off_sig);
  w.qa = reinterpret_cast<Idx*>(base + a.lay.off_near);
  w.qb = reinterpret_cast<Idx*>(base + a.lay.off_far);
  w.def = reinterpret_cast<Idx*>(base + a.lay.off_far2);
  w.wide = reinterpret_cast<Idx*>(base + a.lay.off_ends);
  w.S = reinterpret_cast<Idx*>(base + a.lay.off_S);
  w.off = reinterpret_cast<uint32_t*>(base + a.lay.off_acc);
  w.succ = reinterpret_cast<uint32_t*>(base + a.lay.off_pairs);
  w.succ_cap = a.lay.pair_cap;
  w.bits0 = reinterpret_cast<uint32_t*>(MEM == MEM_BITS ? reinterpret_cast<char*>(sweep_arrays) : base + a.lay.off_pend);
  w.bits1 = w.bits0 + words;
  w.bits2 = reinterpret_cast<uint32_t*>(base + a.lay.off_pend) + 2 * words;
  if constexpr (SM) {
    const SweepNode zero{0.0, 0ull};
    for (uint32_t v = t; v < a.g.n; v += TEAM) w.node[v] = zero;
    w.fill_distances();
  }
  if constexpr (SMEM)
    for (uint32_t i = t; i < 2 * words; i += TEAM) w.bits0[i] = 0;
  team_sync<TEAM>();
  for (;;) {
    if (t == 0) sh.src_idx = atomicAdd(a.counter, 1u);
    team_sync<TEAM>();
    const uint32_t idx = sh.src_idx;
    team_sync<TEAM>();
    if (idx >= a.k) break;
    uint32_t s = __ldg(&a.sources[idx]);
    if (s >= a.g.n) {
      if (t == 0) atomicCAS(a.err, DEV_OK, DEV_ERR_INVALID);
      continue;
    }
    if (a.g.o2n) s = __ldg(&a.g.o2n[s]);
    if (!w.run(s, idx, dirty)) break;
  }
  // distances left by a seeded source: the next launch expects INF
  if (!SM && dirty && !(a.flags & RUN_FORWARD_ONLY)) w.fill_distances();
}

// Launch (a != nullptr) or occupancy, which also raises the kernel's dynamic
// shared memory limit: a plan is asked for its occupancy before it is launched.
template <typename D, int TEAM, int BLOCK, bool PRUNE, int MEM, int G>
cudaError_t sweep_one(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  auto* k = bc_sweep_kernel<D, TEAM, BLOCK, PRUNE, MEM, G>;
  if (a) {
    k<<<grid, BLOCK, p.smem_bytes, st>>>(*a);
    return cudaGetLastError();
  }
  if (MEM == MEM_ALL || MEM == MEM_BITS) {
    // always the device's limit, so plans of different sizes (and threads) do not disturb each other
    int dev = 0, optin = 0;
    cudaFuncAttributes fa{};
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e != cudaSuccess) return e;
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, BLOCK, p.smem_bytes);
}

template <typename D, bool PRUNE, int MEM, int G>
cudaError_t sweep_team(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  switch (p.team) {
    case 32:
      if constexpr (MEM == MEM_GLOBAL || MEM == MEM_CHECK) return sweep_one<D, 32, 256, PRUNE, MEM, G>(p, a, grid, st, occ);
      return cudaErrorInvalidValue;
    case 128: return sweep_one<D, 128, 128, PRUNE, MEM, G>(p, a, grid, st, occ);
    case 256: return sweep_one<D, 256, 256, PRUNE, MEM, G>(p, a, grid, st, occ);
    case 512: return sweep_one<D, 512, 512, PRUNE, MEM, G>(p, a, grid, st, occ);
    case 1024:
      if constexpr (sizeof(D) == 4) return sweep_one<D, 1024, 1024, PRUNE, MEM, G>(p, a, grid, st, occ);
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace
}  // namespace bcgpu
