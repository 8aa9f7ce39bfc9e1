// Sweep schedule, one instantiation set (see bc_sweep.cu).
#include "bc_sweep.cuh"

cudaError_t bcgpu::sweep32_check(const SweepPlan& p, const BatchArgs* a, int grid, cudaStream_t st, int* occ) {
  return sweep_team<uint32_t, false, MEM_CHECK, 1>(p, a, grid, st, occ);
}
