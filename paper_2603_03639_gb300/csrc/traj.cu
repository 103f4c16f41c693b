// Launchers of the trajectory kernel (traj_impl.cuh): qubit states; the operator
// form (physical dimension 4) is compiled in traj_op.cu, in parallel with this file.
#include "traj_impl.cuh"

extern "C" cudaError_t tnrc_op_prepare(int smem);
extern "C" cudaError_t tnrc_op_occupancy(int warps, size_t smem, int* per_sm);
extern "C" cudaError_t tnrc_op_launch(const tnrc::TrajParams* p, int grid, size_t smem, cudaStream_t st);

// host-side launcher; tnrc_create (and the allocation-free entry point) raise
// the shared-memory limit with tnrc_traj_prepare before any launch or capture
extern "C" cudaError_t tnrc_traj_prepare() {
  cudaError_t e = cudaFuncSetAttribute(tnrc::traj_kernel<1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tnrc::traj_kernel<2, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  if (e == cudaSuccess) e = tnrc_op_prepare(226 * 1024);
  return e;
}

// Resident CTAs per SM of the trajectory kernel for this launch shape (the
// size of a pooled launch's region pool is SMs times this).
extern "C" cudaError_t tnrc_traj_occupancy(int phys_dim, int min_blocks, int warps, size_t smem, int* per_sm) {
  if (phys_dim == 4)
    return tnrc_op_occupancy(warps, smem, per_sm);
  if (min_blocks == 2)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, tnrc::traj_kernel<2, 2>, warps * 32, smem);
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, tnrc::traj_kernel<1, 2>, warps * 32, smem);
}

extern "C" cudaError_t tnrc_launch_traj(const tnrc::TrajParams* p, int grid, size_t smem, cudaStream_t st) {
  (void)cudaGetLastError();  // report only this launch below
  // operators (physical dimension 4) have only the build without a register limit
  if (p->phys_dim == 4) return tnrc_op_launch(p, grid, smem, st);
  if (p->min_blocks == 2)
    tnrc::traj_kernel<2, 2><<<grid, p->warps * 32, smem, st>>>(*p);
  else
    tnrc::traj_kernel<1, 2><<<grid, p->warps * 32, smem, st>>>(*p);
  return cudaGetLastError();
}

extern "C" size_t tnrc_traj_smem(int warps, int slab_elems) {
  return (size_t)warps * slab_elems * sizeof(double2) + (size_t)warps * tnrc::kMaxDim * 2 * (sizeof(double) + sizeof(int)) +
         (size_t)warps * 64 * sizeof(double2);
}
