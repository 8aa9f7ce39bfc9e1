// bc_compute_noalloc: batched BC with no device allocation at call time.
//
// Who needs it: callers that must not allocate device memory while they run,
// for example a host thread with real-time limits, code that runs while
// another framework owns the device allocator, or a process whose memory is
// fully reserved up front.  Such callers cannot create a bc_graph_t (that
// allocates), so this entry point takes the caller's device CSR directly.
//
// All scratch (the packed adjacency, Delta_node, the control block and the
// per-source slabs) lives in one file-scope device array of
// BC_NOALLOC_SCRATCH_BYTES.  Every GPU that loads the library holds this
// array until the process exits.  The host code never uses the symbol itself
// as an address: once per device, with that device current, it asks the
// runtime for the array's device address (cudaGetSymbolAddress) and passes that
// pointer to the kernels.  The first call on a device does this set-up, so it
// should come before any stream capture.  The address is cached per device
// together with the unique id of the context it was looked up in; a call
// that finds another context current (for example after cudaDeviceReset)
// looks the address up again.
//
// All calls share the array, and it keeps whatever the last call left there.
// Each call therefore re-initialises what must start at a known value: the
// control block, and in slabs the distance words (INF) and the vertex records
// and bits of the sweep schedule or the backward accumulators of the strict one (0).
//
// Both schedules are enqueued where either may be the faster one: the largest
// weight decides, and only the device knows it.  The kernel and the fills of the one
// not chosen find its source counter parked and leave.
// Two calls whose work overlaps on the GPU (different streams, or different
// host threads, without ordering between them) race on the array.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <mutex>

#include "../../include/bcgpu.h"
#include "bc_common.h"
#include "bc_slab.h"

namespace bcgpu {
namespace {

static __device__ __align__(256) unsigned char g_noalloc_scratch[BC_NOALLOC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_na_mu;

// The scratch array's device address on each device, and the unique id of the
// context it was looked up in (0: unknown, look it up again).
struct NaAddr {
  unsigned long long ctx_id;
  char* ptr;
};
NaAddr g_na_addr[kMaxDevices] = {};

// cuCtxGetCurrent and cuCtxGetId, reached through the runtime's driver entry
// point query so the library needs no link-time dependency on the driver.
using CtxGetCurrentFn = int (*)(void** ctx);
using CtxGetIdFn = int (*)(void* ctx, unsigned long long* id);

// Unique id of the calling thread's current context, or 0 when none is
// current yet or the driver does not offer the query.
unsigned long long current_ctx_id() {
  static const CtxGetCurrentFn get_cur = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<CtxGetCurrentFn>(f);
  }();
  static const CtxGetIdFn get_id = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<CtxGetIdFn>(f);
  }();
  if (!get_cur || !get_id) return 0;
  void* ctx = nullptr;
  if (get_cur(&ctx) != 0 || !ctx) return 0;
  unsigned long long id = 0;
  if (get_id(ctx, &id) != 0) return 0;
  return id;
}

struct NaCtl {
  uint32_t counter[2];  // sources handed out by the sweep kernel and by the strict one
  int err;
  uint32_t debug[2];
  unsigned long long stats[STAT_COUNT];
  // sums over all entries (v -> u, w) of hash(v, u, w) and of hash(u, v, w):
  // equal for a symmetric CSR (the two multisets are the same)
  unsigned long long sym[2];
  unsigned long long width;  // sweep schedule: bucket width, from the largest weight
  uint32_t max_w;
  uint32_t blocks_done;      // of the validation kernel
};

// The device status word carries DEV_* codes; the caller reads them as BC_* codes.
static_assert(DEV_OK == BC_OK && DEV_ERR_INVALID == BC_ERR_INVALID && DEV_ERR_TIMEOUT == BC_ERR_TIMEOUT,
              "device status codes must equal the ABI codes they are reported as");

constexpr uint64_t kCtlBytes = 256;
static_assert(sizeof(NaCtl) <= kCtlBytes, "control block must fit its reserved bytes");

// Strict slabs that the validation kernel initialises on the side (slots 0: none).
struct NaFill {
  char* slabs;
  uint64_t stride, off_acc;  // distances (INF) at 0, accumulators (0) at off_acc
  uint32_t slots;
};

// Validates the caller's CSR while packing it (every read stays inside the
// caller's arrays whatever their contents) and computes Delta_node.  On any
// violation it records DEV_ERR_INVALID and parks the source counters far above
// any source index, so the kernels that follow do no work.  It also
// sums, mod 2^64, a hash of every entry (v -> u, w) and of its reverse
// (u -> v, w): an asymmetric CSR (some entry without its reverse entry of the same
// weight) makes the two sums differ; the block that ends last compares them and
// rejects it like any other invalid input.  That block also derives what follows from
// the largest weight: the sweep schedule's bucket width, by the same rule as for
// a prepared graph, and the schedule: the strict one from `strict_from` to `strict_to`.
// Blocks from `rows` on fill the strict slabs meanwhile: as launches of their own the fills,
// the check and the strict kernel cost a call 12 us (of 155 at 300 vertices), this way 1.
__global__ void na_validate_prep(uint32_t n, uint64_t nnz, const uint64_t* __restrict__ row_ptr,
                                 const uint32_t* __restrict__ col, const uint32_t* __restrict__ w,
                                 const uint32_t* __restrict__ src, uint32_t k, uint2* __restrict__ adj,
                                 uint32_t* __restrict__ dnode, NaCtl* ctl, uint32_t strict_from, uint32_t strict_to,
                                 uint32_t rows, NaFill fill) {
  if (blockIdx.x < rows) {
    const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const uint64_t nth = (uint64_t)rows * blockDim.x;
    bool bad = false;
    uint32_t heaviest = 0;
    unsigned long long fwd = 0, rev = 0;
    if (tid == 0 && (row_ptr[0] != 0 || row_ptr[n] != nnz)) bad = true;
    for (uint64_t v = tid; v < n; v += nth) {
      const uint64_t r0 = row_ptr[v], r1 = row_ptr[v + 1];
      uint32_t m = 0xffffffffu;
      if (r0 > r1 || r1 > nnz) {
        bad = true;
      } else {
        for (uint64_t e = r0; e < r1; ++e) {
          const uint32_t c = col[e], ww = w[e];
          if (c >= n || ww == 0) bad = true;
          adj[e] = make_uint2(c < n ? c : 0u, ww);
          m = min(m, ww);
          heaviest = max(heaviest, ww);
          fwd += entry_hash((uint32_t)v, c, ww);
          rev += entry_hash(c, (uint32_t)v, ww);
        }
      }
      dnode[v] = m;
    }
    for (uint64_t i = tid; i < k; i += nth)
      if (src[i] >= n) bad = true;
    for (int o = 16; o > 0; o >>= 1) {
      fwd += __shfl_xor_sync(0xffffffffu, fwd, o);
      rev += __shfl_xor_sync(0xffffffffu, rev, o);
      heaviest = max(heaviest, __shfl_xor_sync(0xffffffffu, heaviest, o));
    }
    if ((threadIdx.x & 31) == 0) {
      atomicMax(&ctl->max_w, heaviest);
      atomicAdd(&ctl->sym[0], fwd);
      atomicAdd(&ctl->sym[1], rev);
    }
    if (bad) {
      atomicCAS(&ctl->err, DEV_OK, DEV_ERR_INVALID);
      atomicExch(&ctl->counter[0], PARKED);
      atomicExch(&ctl->counter[1], PARKED);
    }
  } else {
    // few slabs: several blocks to each
    const uint32_t blocks = gridDim.x - rows, parts = max(1u, blocks / fill.slots);
    for (uint64_t j = blockIdx.x - rows; j < (uint64_t)fill.slots * parts; j += blocks) {
      char* slab = fill.slabs + j / parts * fill.stride;
      uint64_t* d = reinterpret_cast<uint64_t*>(slab);
      uint64_t* acc = reinterpret_cast<uint64_t*>(slab + fill.off_acc);
      for (uint64_t v = j % parts * blockDim.x + threadIdx.x; v < n; v += (uint64_t)parts * blockDim.x) {
        d[v] = ~0ull;
        acc[v] = 0;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&ctl->blocks_done, 1u) == gridDim.x - 1) {
      __threadfence();
      const uint32_t max_w = atomicMax(&ctl->max_w, 0u);
      ctl->width = sweep_bucket_width(max_w, n, nnz);
      atomicExch(&ctl->counter[max_w >= strict_from && max_w <= strict_to ? 0 : 1], PARKED);
      if (atomicAdd(&ctl->sym[0], 0ull) != atomicAdd(&ctl->sym[1], 0ull)) {
        atomicCAS(&ctl->err, DEV_OK, DEV_ERR_INVALID);
        atomicExch(&ctl->counter[0], PARKED);
        atomicExch(&ctl->counter[1], PARKED);
      }
    }
  }
}

// Largest weight at which the strict schedule is the faster one here, where the sweep
// has neither landmarks nor 32-bit words: one unit of weight per entry of a row up to
// 500 vertices, two up to 1300, then with the square of the degree (the shared-memory form
// holds three teams to an SM, and slabs fewer sources than the strict schedule's).
// Strict / sweep time of this call, all sources: Erdos-Renyi of degree 8 n = 1024
// 0.85 / 1.02 / 1.34 at weights to 4 / 16 / 32, of degree 16 0.92 / 1.13 / 1.44 at 16 / 32 / 64,
// of degree 32 0.65 / 0.81 / 1.07 at 32 / 64 / 128; n = 4096, degree 8 1.03 / 1.25 at 16 /
// 32, degree 16 0.85 / 0.97 at 64 / 128, degree 32 0.63 / 0.82 at 128 / 300; R-MAT 2^12 of
// degree 27 0.29 at 8.  Few sources leave the narrow strict teams alone on their SMs: half
// of it.  Sparse rows: grids 0.78 / 0.90 / 1.07 at 3 / 4 / 6.  At unit weights the strict
// schedule's list of DAG edges outgrows its slab and costs a second scan (1.12 at n = 4096,
// degree 8; below 1300 vertices the sweep's list in shared memory does, too).
uint32_t na_strict_to(uint32_t n, uint64_t nnz, uint32_t k) {
  const double deg = (double)nnz / n;
  const bool few = k < 608 && k < n;
  if (deg < 6.0) return n > 500 && !few ? 4u : 0u;
  const double w = n <= 500 ? deg : (n <= 1300 ? 2.0 * deg : 0.25 * deg * deg);
  return (uint32_t)std::min(few ? 0.5 * w : w, 4.0e9);
}

int na_fail(int code, const char* msg) { return set_error(code, msg); }

}  // namespace
}  // namespace bcgpu

using namespace bcgpu;

extern "C" int bc_compute_noalloc(const uint64_t* d_row_ptr, const uint32_t* d_col_idx, const uint32_t* d_w,
                                  uint32_t n, uint64_t nnz, const uint32_t* d_sources, uint32_t k, double scale,
                                  double* d_out_bc, int* d_status, void* stream) {
  if (n == 0 || n > 0xfffffff0u) return na_fail(BC_ERR_INVALID, "bc_compute_noalloc: n must be in [1, 2^32 - 16]");
  if (!d_row_ptr || !d_out_bc || !d_status) return na_fail(BC_ERR_INVALID, "bc_compute_noalloc: null pointer");
  if (nnz > 0 && (!d_col_idx || !d_w)) return na_fail(BC_ERR_INVALID, "bc_compute_noalloc: null col_idx or w");
  if (k > 0 && !d_sources) return na_fail(BC_ERR_INVALID, "bc_compute_noalloc: null sources");
  if (nnz >= (1ull << 32)) return na_fail(BC_ERR_INVALID, "bc_compute_noalloc: nnz must be below 2^32");
  if (k >= 0x80000000u) return na_fail(BC_ERR_INVALID, "bc_compute_noalloc: k must be below 2^31");
  SlabLayout strict_lay = make_layout(n, 64, SLAB_STRICT);
  strict_lay.stride = strict_lay.off_pair_e;  // its last array is for edge output, which this call has not
  strict_lay.off_pair_e = 0;
  const uint64_t off_adj = kCtlBytes;
  const uint64_t off_dnode = off_adj + align256(std::max<uint64_t>(nnz, 1) * 8);
  const uint64_t off_slabs = off_dnode + align256((uint64_t)n * 4);
  if (off_slabs + strict_lay.stride > BC_NOALLOC_SCRATCH_BYTES) {
    char msg[256];
    snprintf(msg, sizeof msg,
             "bc_compute_noalloc: graph needs %llu scratch bytes for one source, above the fixed maximum of %llu "
             "(BC_NOALLOC_SCRATCH_BYTES); use bc_graph_create + bc_compute_async",
             (unsigned long long)(off_slabs + strict_lay.stride), (unsigned long long)BC_NOALLOC_SCRATCH_BYTES);
    return na_fail(BC_ERR_NOMEM, msg);
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return na_fail(BC_ERR_CUDA, cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return na_fail(BC_ERR_INVALID, "bc_compute_noalloc: device index too large");
  char* base = nullptr;
  {
    // set-up, once per device and context: the array's device address
    std::lock_guard<std::mutex> lk(g_na_mu);
    NaAddr& ad = g_na_addr[dev];
    const unsigned long long cur = current_ctx_id();
    if (!ad.ptr || cur == 0 || cur != ad.ctx_id) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);  // makes the device's context current if needed
      if (e != cudaSuccess) return na_fail(BC_ERR_CUDA, cudaGetErrorString(e));
      ad.ptr = static_cast<char*>(p);
      ad.ctx_id = current_ctx_id();
    }
    base = ad.ptr;
  }
  int sms = 0;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return na_fail(BC_ERR_CUDA, cudaGetErrorString(e));
  bc_config cfg;
  bc_get_config(&cfg);
  const double avg_deg = (double)nnz / n;
  // the sweep schedule unless a knob of the strict one is set; its slab is a
  // little larger, so a graph of which just one strict slab fits stays strict
  SweepPlan plan;
  plan.dist_bits = 64;
  plan.team = 256;
  plan.group = avg_deg >= 12.0 ? 8 : 1;
  sweep_place(plan, n, n, true);
  const SlabKind kind = plan.mem == 2 ? SLAB_NONE : SLAB_SWEEP;
  const SlabLayout lay = make_layout(n, 64, kind);
  const bool sweep = cfg.algorithm != BC_ALGO_STRICT && !cfg.bucket_width && !cfg.settle_in && !cfg.warp_degree &&
                     !cfg.team_degree && off_slabs + lay.stride <= BC_NOALLOC_SCRATCH_BYTES;
  const uint32_t strict_to =
      !sweep ? 0xffffffffu : (cfg.algorithm == BC_ALGO_DELTA ? 0u : na_strict_to(n, nnz, k));
  const uint32_t strict_from = !sweep ? 0u : (n > 1300 && avg_deg >= 6.0 && avg_deg < 12.0 ? 2u : 1u);
  const int team = avg_deg >= 20.0 ? 512 : (avg_deg >= 12.0 ? 256 : 128);
  // sources in flight and CTAs of each schedule
  auto in_flight = [&](uint64_t stride, uint32_t threads, int bps, uint32_t* slots, int* grid) {
    const uint32_t per_block = (uint32_t)(batched_block_threads((int)threads) / (int)threads);
    uint64_t s = (uint64_t)std::max(bps, 1) * sms * per_block;
    s = std::min<uint64_t>(s, (BC_NOALLOC_SCRATCH_BYTES - off_slabs) / stride);
    *slots = (uint32_t)std::min<uint64_t>(s, std::max<uint32_t>(k, 1));
    *grid = (int)((*slots + per_block - 1) / per_block);
  };
  uint32_t slots = 0, strict_slots = 0;
  int grid = 0, strict_grid = 0, bps = 0;
  if (strict_to) {
    e = batched_occupancy(64, team, &bps);
    if (e != cudaSuccess) return na_fail(BC_ERR_CUDA, cudaGetErrorString(e));
    in_flight(strict_lay.stride, (uint32_t)team, bps, &strict_slots, &strict_grid);
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  NaCtl* ctl = reinterpret_cast<NaCtl*>(base);
  uint2* adj = reinterpret_cast<uint2*>(base + off_adj);
  uint32_t* dnode = reinterpret_cast<uint32_t*>(base + off_dnode);
  char* slabs = base + off_slabs;

  // strict slabs that share no memory with sweep ones are filled while the input is validated
  const bool fill_early = strict_to && (!sweep || kind == SLAB_NONE);
  e = cudaMemsetAsync(ctl, 0, sizeof(NaCtl), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(d_out_bc, 0, (size_t)n * 8, st);
  if (e == cudaSuccess) {
    const uint64_t work = std::max<uint64_t>(n, k);
    const uint32_t rows = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((work + 255) / 256, (uint64_t)sms * 8));
    const NaFill fill{slabs, strict_lay.stride, strict_lay.off_acc, fill_early ? strict_slots : 0u};
    na_validate_prep<<<rows + (fill.slots ? 4u * sms : 0u), 256, 0, st>>>(
        n, nnz, d_row_ptr, d_col_idx, d_w, d_sources, k, adj, dnode, ctl, strict_from, strict_to, rows, fill);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && sweep) {  // asked for while the GPU validates
    e = sweep_occupancy(plan, &bps);
    in_flight(lay.stride, (uint32_t)plan.team, bps, &slots, &grid);
  }
  BatchArgs a{};
  a.g.n = n;
  a.g.nnz = nnz;
  a.g.row_ptr = d_row_ptr;
  a.g.adj = adj;
  a.g.adjp = nullptr;
  a.g.dnode = dnode;
  a.g.act_n = n;
  a.sources = d_sources;
  a.k = k;
  a.bc = d_out_bc;
  a.ebc = nullptr;
  a.slabs = slabs;
  a.phase_cap = cfg.phase_cap ? cfg.phase_cap : 4ull * n + 64;  // phases + refills <= 4n + 2
  a.err = &ctl->err;
  a.stats = ctl->stats;
  a.flags = 0;
  a.debug_out = ctl->debug;
  if (e == cudaSuccess && strict_to) {
    a.counter = &ctl->counter[1];
    a.lay = strict_lay;
    a.nslots = strict_slots;
    a.width = cfg.bucket_width ? cfg.bucket_width : 64;
    a.settle_in = cfg.settle_in == 2 ? 0u : 1u;
    a.warp_deg = cfg.warp_degree ? cfg.warp_degree : 32u;
    a.team_deg = std::max<uint32_t>(cfg.team_degree ? cfg.team_degree : 8u * team, a.warp_deg);
    if (!fill_early) e = init_slabs(slabs, strict_lay, SLAB_STRICT, strict_slots, n, 64, st, a.counter);
    if (e == cudaSuccess) e = launch_batched(a, 64, team, strict_grid, st);
  }
  if (e == cudaSuccess && sweep) {
    a.counter = &ctl->counter[0];
    a.lay = lay;
    a.nslots = slots;
    a.width_dev = &ctl->width;
    e = init_slabs(slabs, lay, kind, slots, n, 64, st, strict_to ? a.counter : nullptr);
    if (e == cudaSuccess) e = launch_sweep(a, plan, grid, st);
  }
  if (e == cudaSuccess && scale != 1.0) e = launch_scale(d_out_bc, n, scale, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_status, &ctl->err, sizeof(int), cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return na_fail(BC_ERR_CUDA, cudaGetErrorString(e));
  return BC_OK;
}
