// Sweep schedule, one instantiation set (see bc_sweep.cu).
#include "bc_sweep.cuh"

cudaError_t bcgpu::sweep32_full1_global(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  return sweep_team<uint32_t, false, MEM_GLOBAL, 1>(p, a, grid, st, occ);
}

cudaError_t bcgpu::sweep32_full1_bits(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  return sweep_team<uint32_t, false, MEM_BITS, 1>(p, a, grid, st, occ);
}

cudaError_t bcgpu::sweep32_full1_all(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  return sweep_team<uint32_t, false, MEM_ALL, 1>(p, a, grid, st, occ);
}
