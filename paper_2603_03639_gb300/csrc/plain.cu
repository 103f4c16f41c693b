#include "traj_impl.cuh"

namespace tnrc {

// ---------------------------------------------------------------------------
// The plain GPU path: one trajectory at a time, one launch per step, the
// bonds of a layer spread over CTAs of one warp each (the whole GPU for one
// trajectory, as far as its layers have bonds).  It runs the same device
// functions as the batched kernel and gives bitwise the same results; it is
// the baseline that the persistent batched launch is measured against.
// ---------------------------------------------------------------------------
struct PlainShared {
  double2* slab;
  double* sig;
  double* qn;
  int* perm;
  int* piv;
  double2* small;
};

__device__ inline void plain_warp(const TrajParams& p, WarpCtx& w, int scratch_index, int* order, int* next,
                                  int warp, WideShared* wide = nullptr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* slabs = reinterpret_cast<double2*>(smem_raw);
  double* sig = reinterpret_cast<double*>(slabs + (size_t)p.warps * p.slab_elems);
  double* qns = sig + (size_t)p.warps * kMaxDim;
  int* perms = reinterpret_cast<int*>(qns + (size_t)p.warps * kMaxDim);
  int* pivs = perms + (size_t)p.warps * kMaxDim;
  double2* smalls = reinterpret_cast<double2*>(pivs + (size_t)p.warps * kMaxDim);
  w.region = 0;   // the one environment region
  w.slab = slabs + (size_t)warp * p.slab_elems;
  w.scratch = p.warp_scratch + (size_t)scratch_index * p.scratch_elems;
  w.sig2 = sig + (size_t)warp * kMaxDim;
  w.perm = perms + (size_t)warp * kMaxDim;
  w.qn = qns + (size_t)warp * kMaxDim;
  w.piv = pivs + (size_t)warp * kMaxDim;
  w.small = smalls + (size_t)warp * 64;
  w.lane = threadIdx.x & 31;
  w.cta_slab = slabs;
  w.cta_scratch = w.scratch;
  w.cta_small = smalls;
  w.cta_sig2 = sig;
  w.cta_qn = qns;
  w.cta_perm = perms;
  w.cta_piv = pivs;
  w.wide = wide;
  w.sweeps = w.updates = w.capcuts = 0;
  w.alg = 0;
  w.disc = 0.0;
  w.maxk = 0;
  for (int i = 0; i < kNumPhases; ++i) w.ph[i] = 0;
  w.order = order;
  w.next = next;
}

// Copy a full slot (one CTA).
template <int kD>
__global__ void plain_copy_kernel(TrajParams p, const unsigned char* src, unsigned char* dst) {
  copy_slot<kD>(p, p.full, src, p.full, dst);
}

// What CTA j of a layer's launch takes: one of the nw wide bonds each (they
// come first; the return value is the bond, or -1), then the groups of two of
// the other bonds, which are packed to the front of the order (nb of them,
// group of entry e).  The grouping of the batched launch, so the results are
// the same.
template <int kD>
__device__ int plain_share(const TrajParams& p, const int* D, int j, int& nb, int& e, WarpCtx& w) {
  int wide = -1, nw = 0, left = 0;
  for (int i = 0; i < nb; ++i) {
    const int b = w.order[i];
    if (wide_update<kD>(p, D, b, w.wide->total)) {
      if (nw++ == j) wide = b;
    } else {
      __syncwarp();
      if (w.lane == 0) w.order[left] = b;
      ++left;
    }
  }
  __syncwarp();
  nb = left;
  e = group_size(p) * (j - nw);
  return wide;
}

// Forward layer l of trajectory (s, .) on `slot`.
template <int kD>
__global__ void __launch_bounds__(32) plain_fwd_kernel(TrajParams p, unsigned char* slot, int s, int l) {
  __shared__ int s_order[128], s_next;
  __shared__ WideShared s_wide;
  WarpCtx w;
  plain_warp(p, w, blockIdx.x, s_order, &s_next, 0, &s_wide);
  const int parity = layer_parity(p, l);
  int nb = (p.N - 1 - parity + 1) / 2, e;
  order_layer(p, slot_dims(slot), parity, w);   // reads outer bond dimensions only, which no update changes
  __syncwarp();
  const int wide = plain_share<kD>(p, slot_dims(slot), blockIdx.x, nb, e, w);
  if (wide >= 0)
    wide_update_cta<kD>(p, p.full, slot, wide, layer_rec(p, s, l, wide).G, false, true, true, w);
  else if (e < nb)
    forward_group<kD>(p, p.full, slot, s, l, e, nb, false, true, true, w);
  if (w.lane == 0) atomicAdd(&p.counters[1], (unsigned long long)w.sweeps);
}

// O_t = <t_p | a_t> (one warp).
template <int kD>
__global__ void __launch_bounds__(32) plain_overlap_kernel(TrajParams p, const unsigned char* tg,
                                                           const unsigned char* a, int t) {
  __shared__ int s_order[1], s_next;
  WarpCtx w;
  plain_warp(p, w, 0, s_order, &s_next, 0);
  const double2 O = warp_overlap<kD>(p, p.full, tg, p.full, a, w);
  if (w.lane == 0) p.O[t] = O;
}

// Environments of <c|.|a_l> for layer l (two warps: left and right sweeps).
template <int kD>
__global__ void __launch_bounds__(64) plain_envs_kernel(TrajParams p, const unsigned char* cslot,
                                                        const unsigned char* aslot) {
  __shared__ int s_order[1], s_next;
  WarpCtx w;
  const int warp = threadIdx.x >> 5;
  plain_warp(p, w, warp, s_order, &s_next, warp);
  if (threadIdx.x == 0) {
    env_left(p, w.region)[0] = make_double2(1.0, 0.0);
    env_right(p, w.region)[(size_t)p.N * p.chi * p.chi] = make_double2(1.0, 0.0);
  }
  __syncthreads();
  layer_envs<kD>(p, p.full, cslot, slot_view(aslot, p.full), w, warp);
}

// Gradient and costate update of the bonds of layer l (CTA j: the j-th
// group of two bonds, as in the batched launch).
template <int kD>
__global__ void __launch_bounds__(32) plain_bwd_kernel(TrajParams p, unsigned char* cslot, const unsigned char* aslot,
                                                       int s, int l, int t) {
  __shared__ int s_order[128], s_next;
  __shared__ WideShared s_wide;
  WarpCtx w;
  plain_warp(p, w, blockIdx.x, s_order, &s_next, 0, &s_wide);
  const int parity = layer_parity(p, l);
  int nb = (p.N - 1 - parity + 1) / 2, e;
  const int* D = slot_dims(cslot);
  double* row = p.gsp + (size_t)t * p.K * p.C * p.N;
  order_layer(p, D, parity, w);
  __syncwarp();
  const int wide = plain_share<kD>(p, D, blockIdx.x, nb, e, w);
  if (wide >= 0) {
    double2* th = wide_home<kD>(p, kD * D[wide], kD * D[wide + 2], w).T;
    bond_gradient<kD>(p, p.full, cslot, slot_view(aslot, p.full), s, l, wide, p.O[t], row, w, th, true);
    __syncthreads();
    wide_update_cta<kD>(p, p.full, cslot, wide, layer_rec(p, s, l, wide).G, true, false, true, w, true);
  } else if (e < nb) {
    costate_group<kD>(p, p.full, cslot, slot_view(aslot, p.full), s, l, e, nb, p.O[t], row, w);
  }
  if (w.lane == 0) atomicAdd(&p.counters[1], (unsigned long long)w.sweeps);
}

}  // namespace tnrc

// Host launchers of the plain path (see above).  `op`: 0 copy, 1 forward
// layer, 2 overlap, 3 environments, 4 gradient and costate update.
extern "C" cudaError_t tnrc_launch_plain(const tnrc::TrajParams* p, int op, const unsigned char* a,
                                         unsigned char* b, int s, int l, int t, size_t smem, cudaStream_t st) {
  (void)cudaGetLastError();
  const int nb = (p->N - 1 - ((l + p->first_parity) & 1) + 1) / 2;
  const bool d4 = p->phys_dim == 4;
  switch (op) {
    case 0:
      if (d4) tnrc::plain_copy_kernel<4><<<1, 256, 0, st>>>(*p, a, b);
      else tnrc::plain_copy_kernel<2><<<1, 256, 0, st>>>(*p, a, b);
      break;
    case 1:
      if (d4) tnrc::plain_fwd_kernel<4><<<nb, 32, smem, st>>>(*p, b, s, l);
      else tnrc::plain_fwd_kernel<2><<<nb, 32, smem, st>>>(*p, b, s, l);
      break;
    case 2:
      if (d4) tnrc::plain_overlap_kernel<4><<<1, 32, smem, st>>>(*p, a, b, t);
      else tnrc::plain_overlap_kernel<2><<<1, 32, smem, st>>>(*p, a, b, t);
      break;
    case 3:
      if (d4) tnrc::plain_envs_kernel<4><<<1, 64, smem, st>>>(*p, b, a);
      else tnrc::plain_envs_kernel<2><<<1, 64, smem, st>>>(*p, b, a);
      break;
    case 4:
      if (d4) tnrc::plain_bwd_kernel<4><<<nb, 32, smem, st>>>(*p, b, a, s, l, t);
      else tnrc::plain_bwd_kernel<2><<<nb, 32, smem, st>>>(*p, b, a, s, l, t);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

extern "C" cudaError_t tnrc_plain_prepare() {
  cudaError_t e = cudaSuccess;
  const int lim = 226 * 1024;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tnrc::plain_fwd_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tnrc::plain_fwd_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tnrc::plain_overlap_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tnrc::plain_overlap_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tnrc::plain_envs_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tnrc::plain_envs_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tnrc::plain_bwd_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tnrc::plain_bwd_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  return e;
}
