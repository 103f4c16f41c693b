// The trajectory kernel for operators written as vectors (physical dimension 4).
#include "traj_impl.cuh"

extern "C" cudaError_t tnrc_op_prepare(int smem) {
  return cudaFuncSetAttribute(tnrc::traj_kernel<1, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

extern "C" cudaError_t tnrc_op_occupancy(int warps, size_t smem, int* per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, tnrc::traj_kernel<1, 4>, warps * 32, smem);
}

extern "C" cudaError_t tnrc_op_launch(const tnrc::TrajParams* p, int grid, size_t smem, cudaStream_t st) {
  tnrc::traj_kernel<1, 4><<<grid, p->warps * 32, smem, st>>>(*p);
  return cudaGetLastError();
}
