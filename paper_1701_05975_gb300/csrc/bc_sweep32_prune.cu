// Sweep schedule, one instantiation set (see bc_sweep.cu).
#include "bc_sweep.cuh"

cudaError_t bcgpu::sweep32_prune_global(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  return sweep_team<uint32_t, true, MEM_GLOBAL, 1>(p, a, grid, st, occ);
}

cudaError_t bcgpu::sweep32_prune_bits(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  return sweep_team<uint32_t, true, MEM_BITS, 1>(p, a, grid, st, occ);
}

cudaError_t bcgpu::sweep32_prune_all(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  return sweep_team<uint32_t, true, MEM_ALL, 1>(p, a, grid, st, occ);
}
