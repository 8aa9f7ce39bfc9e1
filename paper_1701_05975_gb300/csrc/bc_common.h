// Internal declarations shared by the CUDA translation units of libbcgpu.
// Not part of the public ABI (that is include/bcgpu.h).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace bcgpu {

// 64-bit finaliser of SplitMix64 (Steele, Lea and Flood, "Fast splittable
// pseudorandom number generators", OOPSLA 2014).
__host__ __device__ inline uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
// Hash of one directed entry (a -> b, weight w).  The sums mod 2^64 over all
// entries and over their reverses are equal for a symmetric CSR, and for
// another only with probability about 2^-64.
__host__ __device__ inline uint64_t entry_hash(uint32_t a, uint32_t b, uint32_t w) {
  return mix64((((uint64_t)a << 32) | b) ^ mix64((uint64_t)w + 0x9e3779b97f4a7c15ull));
}

// Graph as the kernels see it (Sec. 3.1: CSR plus a parallel weight array,
// here interleaved as one 8-byte {col, w} record per entry).
struct GraphDev {
  uint32_t n;
  uint64_t nnz;
  const uint64_t* row_ptr;  // [n + 1]
  const uint2* adj;         // [nnz] {neighbour, weight}; nullptr where adjp and kadj serve both schedules
  const uint32_t* adjp;     // [nnz] neighbour | weight << col_bits (where both fit 32 bits): the strict schedule's
  uint32_t col_bits;        // bits of the neighbour id in an adjp word
  const uint32_t* dnode;    // [n] Delta_node(v) = min incident (directed: outgoing) weight, UINT32_MAX if none
  // Undirected graphs (nullptr otherwise): the second smallest incident weight
  // (UINT32_MAX below two entries) and the neighbour of the smallest one
  // (UINT32_MAX if none): once that neighbour is settled, every edge from v to
  // a vertex still unsettled weighs at least dnode2[v].
  const uint32_t* dnode2;
  const uint32_t* dnode_arg;
  // Directed graphs only (nullptr otherwise): the in-edge CSR, same entry
  // form as the out-edge one, and the minimum incoming weight per vertex.
  const uint64_t* in_row_ptr;
  const uint2* in_adj;
  const uint32_t* in_adjp;
  const uint32_t* dnode_in;
  // Optional relabeling (graph prep orders vertices by decreasing degree so
  // the state of high-degree vertices is contiguous).  Internal ids are
  // "new"; the caller's ids are "old".  All three are nullptr when the graph
  // keeps the caller's order.
  const uint32_t* o2n;      // [n] old id -> new id (applied to sources)
  const uint32_t* n2o;      // [n] new id -> old id (applied to BC output)
  const uint32_t* e2o;      // [nnz] new CSR entry -> old CSR entry (edge BC output)
  // Landmarks of the sweep schedule (kadj == nullptr: none).  h is the main
  // landmark; land_out[l][v] = D(landmark l, v) and land_in[l][v] =
  // D(v, landmark l) in 16- or 32-bit words (the same table for undirected
  // graphs); kadj holds every row in ascending order of its second word.
  const uint2* kadj;        // [nnz] {neighbour | weight << col_bits, w - D(h, neighbour)}; {neighbour, ...} with kw
  const uint32_t* kw;       // [nnz] weights, where neighbour and weight do not fit one word
  const uint32_t* k2o;      // [nnz] kadj entry -> caller's entry
  const void* land_out;
  const void* land_in;
  uint64_t land_stride;     // words per table row (a multiple of 8)
  uint32_t land_bits;       // 16 (0x7fff: unreachable) or 32 (0xffffffff: unreachable)
  uint32_t nland;
  uint32_t land_n;          // vertices from this id on are unreachable from and to h
  uint32_t act_n;           // vertices from this id on have no entries (sweep schedule)
};

constexpr uint32_t SWEEP_MAX_LAND = 64;

// Byte offsets of the per-source arrays inside one slab (one slab per source
// in flight).
// Strict schedule.  d: distances (all INF between sources), sig: sigma during
// the forward pass and the coefficient c = (1 + delta) / sigma during the
// backward pass, S: settle order (the level lists of Algorithm 1's S/ends),
// ends: level boundaries, nearq / farq / farq2: candidate queues (reached,
// unsettled vertices below the split, between the split and split2, above
// split2), acc: per-vertex sum of successor coefficients during the backward
// pass (zero between sources); pend: end of each level's range in the DAG edge
// list; pairs: the shortest-path DAG edges (u -> v) found while pulling sigma,
// in level order of v (capacity pair_cap; on overflow the backward pass falls
// back to scanning every CSR entry).
// Sweep schedule.  d: distances (INF between sources), sig: 16-byte vertex
// records (zero between sources), near / far: frontiers, then the level lists
// and their bounds, far2: deferred vertices, ends: rows left to whole warps,
// S: reached vertices, acc: DAG list offsets, pend: three bits per vertex (two of
// them zero between sources), pairs: compact DAG lists (capacity pair_cap words).
struct SlabLayout {
  uint64_t stride;
  uint64_t off_d, off_sig, off_S, off_ends, off_near, off_far, off_far2, off_acc, off_pend, off_pairs;
  uint64_t off_pair_e;  // entry walked by each DAG edge (edge output); 0 = not in this layout
  uint32_t pair_cap;
  uint32_t smem;  // sweep schedule in shared memory: the offsets are into it, and this many bytes
};

enum : uint32_t {
  RUN_FORWARD_ONLY = 1u,  // stop after distances / sigma / levels (test hook)
  RUN_DIST_ONLY = 2u,     // sweep schedule: write distances to dist_out and stop there
};

// Per-source schedules of the batched kernel.
enum : uint32_t {
  ALGO_STRICT = 1,  // strict settle batches (Sec. 3.2), sigma pulled per batch
  ALGO_DELTA = 2,   // sweep schedule: distances first, then sigma and delta over DAG hop levels
};

enum : int {
  DEV_OK = 0,
  DEV_ERR_INVALID = 1,  // out-of-range source
  DEV_ERR_TIMEOUT = 4,  // phase cap hit
  DEV_ERR_INTERNAL = 5, // a consistency check failed (reported as BC_ERR_CUDA)
};

// Per-run counters (summed over sources).
enum : int {
  STAT_SOURCES = 0,
  STAT_PHASES,
  STAT_REFILLS,
  STAT_REACHED,
  STAT_RELAX,
  STAT_ENTRIES,
  STAT_DAG_EDGES,
  STAT_PAIR_OVERFLOW,
  STAT_CYC_EXPAND,    // SM clock cycles (team leader) spent per section
  STAT_CYC_REFILL,
  STAT_CYC_SETTLE,
  STAT_CYC_BACKWARD,
  STAT_NEAR_SCANNED,  // near / far queue entries read by the threshold, settle and refill passes
  STAT_FAR_SCANNED,
  STAT_LEVELS,        // levels of the backward pass
  STAT_COUNT
};

struct BatchArgs {
  GraphDev g;
  const uint32_t* sources;
  uint32_t k;
  uint32_t* counter;  // [0]: next source index (zeroed before launch)
  double* bc;         // [n] raw sum of delta (scale applied afterwards)
  double* ebc;        // [nnz] raw per-entry shares, or nullptr
  const uint32_t* esm; // edge output with the DAG edge list: walked entry -> output entry, or nullptr
  char* slabs;
  SlabLayout lay;
  uint32_t nslots;
  uint64_t width;      // near/far split width (sweep schedule: bucket width, all ones = one bucket)
  uint32_t settle_in;  // apply the strict IN criterion too
  uint32_t refine;     // bound each candidate's edges to unsettled vertices by dnode2 once dnode_arg is settled
  uint64_t phase_cap;  // cap on phases + refills per source
  int* err;            // DEV_* status word
  unsigned long long* stats;  // [STAT_COUNT] or nullptr
  uint32_t warp_deg;   // forward expansion: rows with >= warp_deg entries get a warp each
  uint32_t team_deg;   // ... and rows with >= team_deg entries the whole team
  uint32_t hot_n;      // ids below hot_n are gathered with an L2 evict-last hint
  uint32_t flags;      // RUN_*
  uint32_t* debug_out; // RUN_FORWARD_ONLY: [0] = levels, [1] = reached
  uint32_t* dist_out;  // RUN_DIST_ONLY: [k][n] distances
  const unsigned long long* width_dev;  // sweep schedule: bucket width in device memory (nullptr: width)
};

// Strict schedule (bc_batched.cu).  team: 32, 128, 256, 512 or (32-bit
// distances) 1024 threads per source.
cudaError_t launch_batched(const BatchArgs& a, int dist_bits, int team, int grid, cudaStream_t st);
int batched_block_threads(int team);
cudaError_t batched_occupancy(int dist_bits, int team, int* blocks_per_sm);

// Bucket width of the sweep schedule without landmark bounds: 4 max_w /
// (average degree), twice that below an average degree of 6.  Rounds against
// entries walked again: Erdos-Renyi 262k (degree 16) 39.5 / 40.6 / 45.8 ms at
// 1/8, 1/4 (this) and 1/2 max_w; 200 x 200 and 512 x 512 grids 6.2 and 32.9 ms at
// 1 max_w, 5.8 and 32.5 at 2 (this), 5.6 and 33.4 at 4.
__host__ __device__ inline unsigned long long sweep_bucket_width(uint32_t max_w, uint32_t n, uint64_t nnz) {
  if (nnz == 0) return 1;
  const double deg = (double)nnz / n;
  const double w = (deg < 6.0 ? 8.0 : 4.0) * max_w / (deg < 1.0 ? 1.0 : deg);
  return w < 1.0 ? 1ull : (unsigned long long)w;
}

// Sweep schedule (bc_sweep*.cu): the kernel variant and its dynamic shared memory.
struct SweepPlan {
  int dist_bits = 32;
  int team = 256;
  bool prune = false;   // rows in landmark order (kadj)
  int mem = 0;          // 0: slab, 1: slab with the vertex bits in shared memory, 2: all in shared memory,
                        // 3: slab, every source's rows checked against their reverses
  int group = 1;        // threads per row: 1 or 8
  uint32_t smem_bytes = 0;
};
cudaError_t launch_sweep(const BatchArgs& a, const SweepPlan& p, int grid, cudaStream_t st);
cudaError_t sweep_occupancy(const SweepPlan& p, int* blocks_per_sm);
// One instantiation set each (a == nullptr: occupancy into *occ).
cudaError_t sweep32_prune_global(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep32_prune_bits(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep32_prune_all(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep32_full1_global(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep32_full8_global(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep32_full1_bits(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep32_full8_bits(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep32_full1_all(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep64_full1_global(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep64_full8_global(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep64_full1_bits(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep64_full8_bits(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep32_check(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep64_check(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);
cudaError_t sweep64_full1_all(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ);

// Settings of one batched run.
struct RunCfg {
  uint32_t team;
  uint64_t width;
  uint32_t settle_in;
  uint32_t refine;  // settled-neighbour refinement of Delta_node (undirected graphs)
  uint64_t phase_cap;
  uint32_t max_slots;
  double mem_fraction;
  uint32_t mode;
  uint32_t warp_deg;
  uint32_t team_deg;
  uint32_t algo;  // ALGO_STRICT or ALGO_DELTA
  bool algo_auto; // not asked for by the configuration or the caller
  uint32_t hot_n;
  SweepPlan sweep;  // ALGO_DELTA
};

// Landmark preparation (bc_land.cu); g.adj holds the rows walked.
cudaError_t land_symmetry(const GraphDev& g, unsigned long long* out, cudaStream_t st);
cudaError_t land_judge(const GraphDev& g, const uint32_t* from_h, const uint32_t* probe, uint32_t h,
                       uint32_t nprobe, unsigned long long* out, cudaStream_t st);
cudaError_t land_max(uint64_t count, const uint32_t* tab, uint32_t* out, cudaStream_t st);
cudaError_t land_pack(uint32_t n, uint64_t stride, uint32_t rows, const uint32_t* tab, int bits, void* out,
                      cudaStream_t st);
cudaError_t land_rows(const GraphDev& g, const uint64_t* host_row_ptr, const uint32_t* from_h, unsigned long long* key,
                      uint32_t col_bits, uint2* kadj, uint32_t* kw, uint32_t* k2o, cudaStream_t st);

// Graph preparation and small helpers (bc_prep.cu).
// dnode2 / dnode_arg may be nullptr (not computed).
cudaError_t launch_prep(uint32_t n, uint64_t nnz, const uint64_t* row_ptr, const uint32_t* col, const uint32_t* w,
                        uint2* adj, uint32_t* dnode, uint32_t* dnode2, uint32_t* dnode_arg, cudaStream_t st);
// Packed form: adjp[e] = col[e] | w[e] << col_bits (caller checked that both fit).
cudaError_t launch_pack32(uint64_t nnz, const uint32_t* col, const uint32_t* w, uint32_t col_bits, uint32_t* adjp,
                          cudaStream_t st);
cudaError_t launch_fill_u64(uint64_t* p, uint64_t count, uint64_t value, cudaStream_t st);
cudaError_t launch_scale(double* p, uint64_t count, double scale, cudaStream_t st);
cudaError_t launch_check_sources(const uint32_t* src, uint32_t k, uint32_t n, int* err, cudaStream_t st);
// Fill `bytes` (a multiple of 4) at offset `off` of every slot of a slab array;
// nothing if *gate, a source counter, is parked (nullptr: always).
constexpr uint32_t PARKED = 0x80000000u;  // a source counter from here on hands out no source
cudaError_t launch_fill_slabs(char* base, uint64_t stride, uint32_t nslots, uint64_t off, uint64_t bytes,
                              uint32_t value, cudaStream_t st, const uint32_t* gate = nullptr);

// Record a message for bc_last_error() on the calling thread; returns code.
int set_error(int code, const char* msg);

// The paper's thread mappings (bc_paper.cu): node-parallel or work-efficient
// expansion with VW threads per vertex, Delta_i and settle over all V.
struct PaperWork {
  uint32_t n = 0;
  void* d = nullptr;
  double* sig = nullptr;
  uint32_t* S = nullptr;
  uint8_t* U = nullptr;
  uint8_t* F = nullptr;
  void* ctr = nullptr;
  void* host_ctr = nullptr;  // pinned
};
PaperWork* paper_create(uint32_t n, int dist_bits, cudaError_t* e);
void paper_destroy(PaperWork* w);
uint64_t paper_bytes(uint32_t n, int dist_bits);
cudaError_t paper_run(PaperWork* w, const GraphDev& g, int dist_bits, const uint32_t* host_sources,
                      const uint32_t* host_o2n, uint32_t k, double* bc, bool node_parallel, int vwarp,
                      uint64_t phase_cap, int sm_count, cudaStream_t st, int* status, unsigned long long* stats);

}  // namespace bcgpu

struct bc_graph;

namespace bcgpu {

// Serving support (implemented in bc_api.cu, used by the scheduler in
// bc_serve.cu).  A lease is one request's workspace (slabs, source list,
// device accumulator), held from serve_open to serve_finish; the request's
// sources run as a sequence of source batches (serve_batch), each one
// persistent launch that adds into the accumulator, on whichever stream the
// scheduler picks.  The last batch also scales the sum and copies it to
// pinned host memory; serve_finish hands it to the caller and releases the
// workspace.
struct ServeLease;
struct ServePlan {
  RunCfg run;           // settings at admission: the lease's slabs and kernel belong to them
  uint32_t max_slots;   // sources the GPU holds at once for this team size
  uint64_t slot_bytes;  // device bytes per source in flight
  uint64_t fixed_bytes; // per-request device bytes besides the slabs
};
// budget: device bytes a request may take (a strict slab is smaller than a sweep one).
int serve_plan(bc_graph* g, uint32_t k, uint64_t budget, ServePlan* out);
// Reserve a workspace of up to slot_cap slabs and stage the sources (on st).
int serve_open(bc_graph* g, const ServePlan& plan, const uint32_t* sources, uint32_t k, uint32_t slot_cap, cudaStream_t st,
               ServeLease** out);
uint32_t serve_slot_cap(const ServeLease* l);  // slabs actually held
// Enqueue sources [first, first + count) with `slots` of them in flight; the
// last batch also applies `scale` and stages the result for serve_finish.
int serve_batch(ServeLease* l, uint32_t first, uint32_t count, uint32_t slots, bool last, double scale,
                cudaStream_t st);
bool serve_ready(ServeLease* l);         // the latest batch has completed
int serve_batch_status(ServeLease* l);   // its device status (waits for it)
int serve_finish(ServeLease* l, double* out_bc);  // out_bc may be null (failed request); releases the lease
int graph_device(const bc_graph* g);
uint32_t graph_n(const bc_graph* g);
uint64_t graph_nnz(const bc_graph* g);
void graph_serving_ref(bc_graph* g, int delta);

// Plain form (bc_plain.cu): one source at a time over the whole GPU.
struct PlainWork;
PlainWork* plain_create(uint32_t n, int dist_bits, cudaError_t* e);
void plain_destroy(PlainWork* w);
uint64_t plain_bytes(uint32_t n, int dist_bits);
// Runs sources[0..k) (HOST list) one after another; adds raw delta into bc.
// Returns DEV_* status through *dev_status.
// host_o2n: the graph's old -> new id map on the host (nullptr: no relabeling).
cudaError_t plain_run(PlainWork* w, const GraphDev& g, int dist_bits, const uint32_t* host_sources,
                      const uint32_t* host_o2n, uint32_t k, double* bc, uint64_t width, uint32_t settle_in,
                      uint64_t phase_cap, int sm_count, cudaStream_t st, int* dev_status,
                      unsigned long long* host_stats);

}  // namespace bcgpu
