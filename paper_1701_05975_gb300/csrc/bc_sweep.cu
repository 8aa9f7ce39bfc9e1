// Variant choice of the sweep schedule (device code in bc_sweep.cuh, several
// translation units so that the instantiation sets compile in parallel).
#include "bc_common.h"

namespace bcgpu {
namespace {

cudaError_t dispatch(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  using Fn = cudaError_t (*)(const SweepPlan&, const BatchArgs*, int, cudaStream_t, int*);
  // [distance width and row order][memory form]
  static const Fn prune32[3] = {sweep32_prune_global, sweep32_prune_bits, sweep32_prune_all};
  static const Fn full32[3] = {sweep32_full1_global, sweep32_full1_bits, sweep32_full1_all};
  static const Fn wide32[3] = {sweep32_full8_global, sweep32_full8_bits, sweep32_full1_all};
  static const Fn full64[3] = {sweep64_full1_global, sweep64_full1_bits, sweep64_full1_all};
  static const Fn wide64[3] = {sweep64_full8_global, sweep64_full8_bits, sweep64_full1_all};
  if (p.mem == 3) return p.dist_bits == 32 ? sweep32_check(p, a, grid, st, occ) : sweep64_check(p, a, grid, st, occ);
  if (p.mem < 0 || p.mem > 3) return cudaErrorInvalidValue;
  const Fn* row = p.dist_bits == 32 ? (p.prune ? prune32 : (p.group == 8 ? wide32 : full32))
                                    : (p.group == 8 ? wide64 : full64);
  return row[p.mem](p, a, grid, st, occ);
}

}  // namespace

cudaError_t launch_sweep(const BatchArgs& a, const SweepPlan& p, int grid, cudaStream_t st) {
  if (grid <= 0) return cudaSuccess;
  return dispatch(p, &a, grid, st, nullptr);
}

cudaError_t sweep_occupancy(const SweepPlan& p, int* blocks_per_sm) { return dispatch(p, nullptr, 0, nullptr, blocks_per_sm); }

}  // namespace bcgpu
