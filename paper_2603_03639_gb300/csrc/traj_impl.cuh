// Persistent trajectory kernel: one CTA evaluates one trajectory (noise sample
// s, input p) at a time and takes the next one from a device work counter.
//
//   forward  (Sec. II): the truncated layers of the time discretisation, each
//            a set of disjoint two-site gates with their parity alternating --
//            for the second-order split A(dt/2) B(dt) A(dt/2) per Trotter step
//            the 2S+1 layers A_0, B_0, A_0A_1, B_1, ..., B_{S-1}, A_{S-1} (half
//            layers at a step boundary merged into one gate: the state is
//            compressed once per time step), for the first-order slice of
//            Eq. circuit two layers per step (odd bonds; even bonds with the
//            single-site rotations folded in).  Every two-site gate is
//            followed by the truncated SVD; the warps of the CTA share the
//            disjoint bonds of a layer, largest first, and work together on a
//            bond that is a large part of its layer.
//   overlap  (Sec. II state form): O = <t_p | a(T)> by a transfer-matrix sweep.
//   gradient (App. A): the costate b_l = L_{l+1}^dag .. L_L^dag t is propagated
//            backwards with the same truncated update; for every gate of layer
//            l, dO/du += tr(Q_u rho) with rho the mixed two-site density of
//            <b_l|.|a_l> from left/right environments and Q_u from the layer
//            gate table; the forward states a_l come from the packed history
//            of the forward pass (or are recomputed segment by segment from
//            checkpoints when the history does not fit).
// Each trajectory writes its own O and its own gradient row, so results do not
// depend on which CTA ran it or on what else ran in the launch.
//
// What bounds it: with the SVDs in integers (fx.cuh) neither the FP64 pipe nor
// DRAM is busy for long (profiles/traj_kernel_cnot50_counters.txt); a warp waits
// for the results of its own instructions (fixed latencies a third
// of the stalls, then shared and L2 loads, barriers and instruction fetch), two
// warps to a scheduler, which the 220 KB of shared memory for theta and
// R^dagger allow.  Every function is out of line and no runtime loop unrolled:
// inlined and unrolled the kernel overran the instruction cache, which cost
// 45 % of the stalls (50-qubit CNOT, 304 trajectories: 742 ms, then 386 ms).
#pragma once
#include "svd_fx.cuh"

namespace tnrc {

// device counters: [0] updates [1] Jacobi sweeps [2] max bond [3] algorithmic
// FP64 flops [4] trajectories whose packed history did not fit and that were
// redone with checkpoints [5 + d] forward updates that left bond dimension d
constexpr int kCtrHist = 5;

struct WarpCtx {
  double2* slab;       // shared, slab_elems
  double2* scratch;    // global, scratch_elems
  double* sig2;        // shared, kMaxDim
  double* qn;          // shared, kMaxDim (SvdBufs)
  int* perm;           // shared, kMaxDim
  int* piv;            // shared, kMaxDim
  double2* small;      // shared, 64 complex (four 4x4 matrices)
  int lane;
  long long sweeps;
  long long updates;
  double disc;
  int maxk;
  unsigned long long alg;   // algorithmic flops counted by lane 0
  long long capcuts;        // cuts decided by the cap chi (forward and costate updates)
  long long ph[kNumPhases]; // phase cycles (TNRC_PHASE_TIMERS builds)
  int* order;               // shared, CTA-wide: bonds of the current layer by decreasing cost
  int* next;                // shared, CTA-wide: next entry of `order` to take
  int region;               // the CTA's work region (scratch, environments, slots)
  // updates shared by the CTA's warps: the whole shared slab, the first warp's
  // arrays and scratch, and a few words
  double2 *cta_slab, *cta_scratch, *cta_small;
  double *cta_sig2, *cta_qn;
  int *cta_perm, *cta_piv;
  struct WideShared* wide;
};

struct WideShared {
  double part[kWarps];
  FxQrShared qr;
  long long total;   // cost of the current layer
  int k;
};

// Algorithmic flops of one two-site update with theta of m x n (m = 2 Dl,
// n = 2 Dr), inner bond Dc and k kept values: contraction 8 m Dc n, gate
// 128 Dl Dr, thin SVD 4 (14 a b^2 + 8 b^3) (a = max(m, n), b = min(m, n);
// Golub-Van Loan count, x4 for complex), split 8 m n k.
__device__ __forceinline__ unsigned long long update_flops(int m, int n, int Dc, int k) {
  const unsigned long long a = m > n ? m : n, b = m > n ? n : m;
  return 8ull * m * Dc * n + 32ull * m * n + 4ull * (14ull * a * b * b + 8ull * b * b * b) + 8ull * m * n * k;
}

// Bonds of truncated layer l have parity (l + first_parity) & 1; the record of
// bond b in layer l of sample s is layer_off[l] + b / 2 within the sample.
__device__ __forceinline__ int layer_parity(const TrajParams& p, int l) { return (l + p.first_parity) & 1; }

__device__ __forceinline__ const LayerGate& layer_rec(const TrajParams& p, int s, int l, int b) {
  return p.lgates[(size_t)s * p.recs_per_sample + p.layer_off[l] + (b >> 1)];
}

// ---------------------------------------------------------------------------
// Physical dimension kD: 2 for qubit states; 4 for operators written as
// vectors (site index s = 2 out + in, the MPO of Sec. II), where the 4x4 gate
// acts on the two out indices and leaves the in indices alone.  With
// kI = kD / 2, s = o kI + i.
// ---------------------------------------------------------------------------
// Two-site update of bond b: theta = lam_{b-1} G (B_b B_{b+1}), truncated SVD,
// B_{b+1} <- Y_k^dag, B_b <- Phi Y_k / |S_k|, lam_b <- S_k / |S_k|.
// The SVD (svd_fx.cuh, in integers): theta = Q R by pivoted Gram-Schmidt (Q not
// kept; R has r rows, r the numerical rank), then one-sided Jacobi on the r
// columns of R^dagger: R^dagger V = Z S, so theta = (Q V) S Z^dagger and Y = Z.
// ---------------------------------------------------------------------------
// Per-matrix work arrays of the SVD (shared, per warp): squared singular values
// (row exponents during the QR), column norms of the QR and then the columns'
// exponents, exponents of R^dagger and then the rank order, QR column order and
// then the columns' shifts.
struct SvdBufs {
  double* sig2;
  double* qn;
  int* perm;
  int* piv;
};

// Phase 1 of a two-site update of bond b: Phi = G (B_b B_{b+1}) and theta =
// lam_{b-1} Phi, both row-major: row (al s1), column (s2 ga).  With have_pre the
// product B_b B_{b+1} is in T already.  By one warp, or (cta) by every thread of
// the CTA; returns this thread's part of |theta|_F^2.  gs: 16 shared elements.
//
// Three passes of one element per thread each: product, gate, Schmidt values.
// A thread that took a whole (al, ga) through all three left half the lanes idle
// in its second round (36 pairs on 32 lanes at bonds of 6): 10,200 cycles an
// update on 8 qubits, 5,200 in passes; 250,000 and 57,500 in the operator form.
template <int kD>
__device__ __noinline__ double theta_build(const TrajParams& p, const Lay& Y, unsigned char* slot, int b,
                                           const double2* G, bool adjoint, double2* T, double2* Phi, bool have_pre,
                                           double2* gs, bool cta) {
  constexpr int kI = kD / 2, kDD = kD * kD;
  const int ti = cta ? (int)threadIdx.x : (int)(threadIdx.x & 31), nt = cta ? (int)blockDim.x : 32;
  const int* D = slot_dims(slot);
  const int Dl = D[b], Dc = D[b + 1], Dr = D[b + 2];
  const int n = kD * Dr, total = kD * Dl * n;
  const double2* sites = slot_sites(slot, Y.L);
  const double* lam = slot_lam(slot, Y.L) + (size_t)(b > 0 ? b - 1 : 0) * Y.L.chi;
  const double2* A = sites + Y.site_off[b];
  const double2* Bt = sites + Y.site_off[b + 1];
  if (ti < 16) gs[ti] = adjoint ? cconj(G[(ti & 3) * 4 + (ti >> 2)]) : G[ti];
  if (!have_pre) {
#pragma unroll 1
    for (int u = ti; u < total; u += nt) {
      const int row = u / n, col = u - row * n;
      double2 acc = make_double2(0.0, 0.0);
#pragma unroll 2
      for (int be = 0; be < Dc; ++be) cfma(acc, A[(size_t)row * Dc + be], Bt[(size_t)be * n + col]);
      T[u] = acc;
    }
  }
  if (cta) __syncthreads(); else __syncwarp();
#pragma unroll 1
  for (int u = ti; u < total; u += nt) {
    const int q = u / Dr, ga = u - q * Dr, al = q / kDD, ss = q - al * kDD;
    const int s1 = ss / kD, s2 = ss - s1 * kD;
    const double2* g = gs + ((s1 / kI) * 2 + s2 / kI) * 4;
    const double2* t = T + ((size_t)al * kDD + (s1 % kI) * kD + s2 % kI) * Dr + ga;
    double2 v = make_double2(0.0, 0.0);
#pragma unroll
    for (int p1 = 0; p1 < 2; ++p1)
#pragma unroll
      for (int p2 = 0; p2 < 2; ++p2) cfma(v, g[p1 * 2 + p2], t[(p1 * kI * kD + p2 * kI) * Dr]);
    Phi[u] = v;
  }
  if (cta) __syncthreads(); else __syncwarp();
  double fro = 0.0;
#pragma unroll 1
  for (int u = ti; u < total; u += nt) {
    const double ll = (b > 0) ? lam[u / (kDD * Dr)] : 1.0;
    const double2 th = cscale(Phi[u], ll);
    T[u] = th;
    fro += cabs2(th);
  }
  return fro;
}

// Phase 3 of a two-site update of bond b, by one warp, after the SVD left
// R^dagger V = Z S in X (r columns of length n, real values X 2^ex[j]): rank and
// truncate, lam_b <- S_k / |S_k|.  Keeps k = max(1, min(chi, #{sigma_j > eps
// sigma_max})); bf.perm[i] = column of rank i, by decreasing sigma with ties to
// the smaller index.  nrm[j] (r entries) receives what normalises column j: y =
// 1 / |X_j| for X_j shifted by the number in bf.piv[j].  Returns k; inv_kn =
// 1 / |S_k|.  In integers but for the squared values that are ranked and the
// Schmidt values themselves: with FP64 sums, roots and quotients this took 8,500
// cycles of a small update's 65,000.
struct ColNorm {
  long long n2, y;
};
template <int kD>
__device__ __noinline__ int theta_rank(const TrajParams& p, const Lay& Y, unsigned char* slot, int b, const int4* X,
                                       int ldx, const int* ex, ColNorm* nrm, int r, int sw, bool record, bool count,
                                       WarpCtx& w, SvdBufs bf, double& inv_kn) {
  const int lane = w.lane;
  const int* D = slot_dims(slot);
  const int m = kD * D[b], n = kD * D[b + 2];
  {
    const int lg = fx_lanes(r, 32), gi = lane >> lg, lig = lane & ((1 << lg) - 1), groups = 32 >> lg;
#pragma unroll 1
    for (int c0 = 0; c0 < r; c0 += groups) {
      const int c = c0 + gi;
      FxSquares nn{0, 0, 0};
      if (c < r)
#pragma unroll 1
        for (int i = lig; i < n; i += 1 << lg) {
          const int4 a = X[c * ldx + i];
          fx_square(nn, fx_re(a));
          fx_square(nn, fx_im(a));
        }
      const long long N = fx_group_sum(fx_sum(nn), lg, lg);
      if (c < r && lig == 0) nrm[c].n2 = N;
    }
  }
  __syncwarp();
  // sigma_j^2 = n2 2^(56 + 2 e), n2 in [2^54, 2^56), e = ex - shift
  int emax = -100000;
  double mx = 0.0;
#pragma unroll 1
  for (int j = lane; j < r; j += 32) {
    long long N = nrm[j].n2;
    int z = 0;
    double sq = 0.0;
    if (N > 0) {
      z = (55 - (63 - __clzll(N))) >> 1;
      N = z >= 0 ? N << (2 * z) : N >> (-2 * z);
      emax = max(emax, ex[j] - z);
      sq = fx_scale((double)N, 56 + 2 * (ex[j] - z));
      nrm[j].y = fx_rsqrt(N);
    } else {
      nrm[j].y = 0;
    }
    nrm[j].n2 = N;
    bf.piv[j] = z;
    bf.sig2[j] = sq;
    mx = fmax(mx, sq);
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    const long long v = __shfl_xor_sync(0xffffffffu, __double_as_longlong(mx), o);
    if (v > __double_as_longlong(mx)) mx = __longlong_as_double(v);
  }
  __syncwarp();
  const double cut2 = p.eps * p.eps * mx;
  int cnt = 0;
  long long tot = 0;
#pragma unroll 1
  for (int j = lane; j < r; j += 32) {
    cnt += bf.sig2[j] > cut2 ? 1 : 0;
    const int d = 2 * (emax - ex[j] + bf.piv[j]);
    tot += d < 63 ? nrm[j].n2 >> d : 0;
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  int k = cnt < p.chi ? cnt : p.chi;
  if (k > n) k = n;  // at most n orthogonal columns of length n
  if (k < 1) k = 1;
  long long kept = 0;
#pragma unroll 1
  for (int j = lane; j < r; j += 32) {
    const long long vj = __double_as_longlong(bf.sig2[j]);
    int rk = 0;
#pragma unroll 1
    for (int i = 0; i < r; ++i) {
      const long long vi = __double_as_longlong(bf.sig2[i]);
      rk += (vi > vj || (vi == vj && i < j)) ? 1 : 0;
    }
    if (rk <= k) bf.perm[rk] = j;
    const int d = 2 * (emax - ex[j] + bf.piv[j]);
    if (rk < k) kept += d < 63 ? nrm[j].n2 >> d : 0;
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    tot += __shfl_xor_sync(0xffffffffu, tot, o);
    kept += __shfl_xor_sync(0xffffffffu, kept, o);
  }
  __syncwarp();
  const double kept2 = fx_scale((double)kept, 56 + 2 * emax);
  if (lane == 0) {
    if (sw < 0) atomicOr(p.status, kStatusNoConverge);
    if (!(kept2 > 0.0)) atomicOr(p.status, kStatusNaN);
  }
  // the relative distance between the last kept and the first dropped value,
  // when the cap chi decided the cut
  const bool capped = cnt > k && k < r;
  if (k > Y.dcap[b + 1]) {  // cannot happen (k <= min(m, n, chi)); keeps memory in bounds regardless
    k = Y.dcap[b + 1];
    if (lane == 0) atomicOr(p.status, kStatusBadDims);
  }
  w.sweeps += (sw < 0) ? -sw : sw;
  w.updates += 1;
  if (record) {
    w.disc += tot > kept ? (double)(tot - kept) / (double)tot : 0.0;
    if (k > w.maxk) w.maxk = k;
    if (lane == 0) atomicAdd(&p.counters[kCtrHist + k], 1ull);
  }
  if (count) {
    w.alg += update_flops(m, n, D[b + 1], k);
    if (capped) {
      w.capcuts += 1;
      const double gap = (sqrt(bf.sig2[bf.perm[k - 1]]) - sqrt(bf.sig2[bf.perm[k]])) / sqrt(mx);
      if (lane == 0) atomicMin(&p.counters[kCtrGap], (unsigned long long)__double_as_longlong(gap));
    }
  }
  inv_kn = rsqrt(kept2);
  double* lamw = slot_lam(slot, Y.L) + (size_t)b * Y.L.chi;
#pragma unroll 1
  for (int i = lane; i < k; i += 32) {
    const int j = bf.perm[i];
    const long long s = fx_mul(fx_split(nrm[j].n2), fx_split(nrm[j].y));   // |X_j| 2^shift
    lamw[i] = fx_scale((double)s, ex[j] - bf.piv[j]) * inv_kn;
  }
  __syncwarp();
  return k;
}

// Row i of Y_k^dagger, y_i = X_j / |X_j| with j = perm[i], into T (FP64), by
// thread ti of nt.
__device__ __forceinline__ void right_vectors(const int4* X, int ldx, const ColNorm* nrm, const SvdBufs& bf, int n, int k,
                                              double2* T, int ti, int nt) {
#pragma unroll 1
  for (int it = ti; it < k * n; it += nt) {
    const int i = it / n, c = it - i * n, j = bf.perm[i];
    const int4 z = fx_shift(X[j * ldx + c], bf.piv[j]);
    const Fx y = fx_split(nrm[j].y);
    T[it] = make_double2(fx_scale((double)fx_mul(fx_re(z), y), -56), fx_scale((double)fx_mul(fx_im(z), y), -56));
  }
}

// Phase 4, by thread ti of nt: B_{b+1} <- Y_k^dag, B_b <- Phi Y_k / |S_k|, with
// column i of Y_k = T[i n + .].
template <int kD>
__device__ __noinline__ void theta_split(const Lay& Y, unsigned char* slot, int b, const double2* T, const double2* Phi,
                                         int k, double inv_kn, int ti, int nt) {
  const int* D = slot_dims(slot);
  const int m = kD * D[b], n = kD * D[b + 2];
  double2* sites = slot_sites(slot, Y.L);
  double2* A = sites + Y.site_off[b];
  double2* Bt = sites + Y.site_off[b + 1];
#pragma unroll 1
  for (int it = ti; it < k * n; it += nt) Bt[it] = cconj(T[it]);
#pragma unroll 1
  for (int it = ti; it < m * k; it += nt) {
    const int row = it / k, i = it - row * k;
    const double2* ph = Phi + (size_t)row * n;
    const double2* z = T + (size_t)i * n;
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int c = 0; c < n; ++c) cfma(acc, ph[c], z[c]);
    A[it] = cscale(acc, inv_kn);
  }
}

// Phases 3 and 4 by one warp.
template <int kD>
__device__ __noinline__ void theta_finish(const TrajParams& p, const Lay& Y, unsigned char* slot, int b, const int4* X,
                                          int ldx, const int* ex, ColNorm* nrm, double2* T, const double2* Phi, int r,
                                          int sw, bool record, bool count, WarpCtx& w, SvdBufs bf) {
  TNRC_TIC(t_r);
  double inv_kn;
  const int k = theta_rank<kD>(p, Y, slot, b, X, ldx, ex, nrm, r, sw, record, count, w, bf, inv_kn);
  TNRC_TOC(w, 2, t_r);
  TNRC_TIC(t_w);
  right_vectors(X, ldx, nrm, bf, kD * slot_dims(slot)[b + 2], k, T, w.lane, 32);
  __syncwarp();
  theta_split<kD>(Y, slot, b, T, Phi, k, inv_kn, w.lane, 32);
  __syncwarp();
  if (w.lane == 0) slot_dims(slot)[b + 1] = k;
  __syncwarp();
  TNRC_TOC(w, 3, t_w);
}

// A NaN or infinity in theta does not survive the integers: report it here.
__device__ __forceinline__ void flag_not_finite(const TrajParams& p, double fro, int lane) {
  if (lane == 0 && !(fro < 1e300)) atomicOr(p.status, kStatusNaN);
}

// Slab elements of one update: theta, R^dagger and a pivot column, which the SVD
// works on, and Phi, which is written and read once.
__device__ __forceinline__ int svd_elems(int m, int n) { return m * n + (m < n ? m : n) * (n | 1) + m; }
__device__ __forceinline__ int upd_elems(int m, int n) { return m * n + svd_elems(m, n); }

// The update of bond b by one warp: theta and R^dagger in its shared slab, Phi
// too when it fits, else in the warp's global scratch.
template <int kD>
__device__ __noinline__ void two_site_update(const TrajParams& p, const Lay& Y, unsigned char* slot, int b,
                                             const double2* G, bool adjoint, bool record, bool count, WarpCtx& w,
                                             bool have_pre = false) {
  const int lane = w.lane;
  const int* D = slot_dims(slot);
  const int m = kD * D[b], n = kD * D[b + 2];
  double2* T = w.slab;
  double2* Phi = upd_elems(m, n) <= p.slab_elems ? w.slab + svd_elems(m, n) : w.scratch;
  int4* X = reinterpret_cast<int4*>(w.slab + m * n);
  TNRC_TIC(t_c);
  const double fro = warp_sum(theta_build<kD>(p, Y, slot, b, G, adjoint, T, Phi, have_pre, w.small, false));
  __syncwarp();
  TNRC_TOC(w, 0, t_c);
  TNRC_TIC(t_j);
  flag_not_finite(p, fro, lane);
  const int ldx = n | 1;
  int* ex = reinterpret_cast<int*>(w.qn);
  int r = fx_qr(T, X + (m < n ? m : n) * ldx, m, n, fro, X, ldx, w.perm, w.piv, reinterpret_cast<float*>(w.qn),
                reinterpret_cast<int*>(w.sig2), lane, 32);
  if (r < 1) {  // theta == 0 (or not finite): keep one column; the NaN check reports it
    r = 1;
#pragma unroll 1
    for (int e = lane; e < n; e += 32) X[e] = make_int4(0, 0, 0, 0);
    if (lane == 0) w.perm[0] = 0;
    __syncwarp();
  }
  TNRC_TOC(w, 1, t_j);
  TNRC_TIC(t_s);
  const int sw = fx_jacobi(X, ldx, n, r, w.perm, ex, lane, 32);
  TNRC_TOC(w, 8, t_s);
  theta_finish<kD>(p, Y, slot, b, X, ldx, ex, reinterpret_cast<ColNorm*>(X + (m < n ? m : n) * ldx), T, Phi, r, sw,
                   record, count, w, SvdBufs{w.sig2, w.qn, w.perm, w.piv});
}

// Where a wide update keeps theta, Phi and R^dagger: side by side in the
// CTA's whole shared slab when they fit there, else in the first warp's
// global scratch.
struct WideHome {
  double2 *T, *Phi, *X;
  bool shared;
};
template <int kD>
__device__ __forceinline__ WideHome wide_home(const TrajParams& p, int m, int n, const WarpCtx& w) {
  WideHome h;
  const int mn = m * n;
  h.shared = svd_elems(m, n) <= p.cta_slab_elems;
  const size_t room = (size_t)kD * kD * p.chi * p.chi;
  h.T = h.shared ? w.cta_slab : w.cta_scratch + room;
  h.Phi = upd_elems(m, n) <= p.cta_slab_elems ? w.cta_slab + svd_elems(m, n) : w.cta_scratch;
  h.X = h.shared ? w.cta_slab + mn : w.cta_scratch + 2 * room;
  return h;
}

// The update of a wide bond by the whole CTA (every thread calls it).
template <int kD>
__device__ __noinline__ void wide_update_cta(const TrajParams& p, const Lay& Y, unsigned char* slot, int b,
                                             const double2* G, bool adjoint, bool record, bool count, WarpCtx& w,
                                             bool have_pre = false) {
  const int ti = threadIdx.x, nt = blockDim.x, warp = ti >> 5;
  const int* D = slot_dims(slot);
  const int m = kD * D[b], n = kD * D[b + 2];
  const WideHome h = wide_home<kD>(p, m, n, w);
  int4* X = reinterpret_cast<int4*>(h.X);
  WideShared* ws = w.wide;
  TNRC_TIC(t_c);
  const double part = warp_sum(theta_build<kD>(p, Y, slot, b, G, adjoint, h.T, h.Phi, have_pre, w.cta_small, true));
  if (w.lane == 0) ws->part[warp] = part;
  __syncthreads();
  double fro = 0.0;
#pragma unroll 1
  for (int i = 0; i < (nt >> 5); ++i) fro += ws->part[i];
  TNRC_TOC(w, 0, t_c);
  TNRC_TIC(t_j);
  flag_not_finite(p, fro, ti);
  const int ldx = n | 1;
  int4* Pw = X + (m < n ? m : n) * ldx;
  float* cn = reinterpret_cast<float*>(w.cta_qn);
  int* er = reinterpret_cast<int*>(w.cta_sig2);
  int r = h.shared ? fx_qr_cta<true>(h.T, Pw, m, n, fro, X, ldx, w.cta_perm, w.cta_piv, cn, er, &ws->qr)
                   : fx_qr_cta<false>(h.T, Pw, m, n, fro, X, ldx, w.cta_perm, w.cta_piv, cn, er, &ws->qr);
  if (r < 1) {
    r = 1;
#pragma unroll 1
    for (int e = ti; e < n; e += nt) X[e] = make_int4(0, 0, 0, 0);
    if (ti == 0) w.cta_perm[0] = 0;
    __syncthreads();
  }
  TNRC_TOC(w, 1, t_j);
  TNRC_TIC(t_s);
  int* ex = reinterpret_cast<int*>(w.cta_qn);
  const int sw = h.shared ? fx_jacobi_cta<true>(X, ldx, n, r, w.cta_perm, ex)
                          : fx_jacobi_cta<false>(X, ldx, n, r, w.cta_perm, ex);
  TNRC_TOC(w, 8, t_s);
  TNRC_TIC(t_r);
  ColNorm* nrm = reinterpret_cast<ColNorm*>(Pw);
  const SvdBufs bf{w.cta_sig2, w.cta_qn, w.cta_perm, w.cta_piv};
  if (warp == 0) {
    double inv_kn;
    const int k = theta_rank<kD>(p, Y, slot, b, X, ldx, ex, nrm, r, sw, record, count, w, bf, inv_kn);
    if (w.lane == 0) {
      ws->k = k;
      ws->part[0] = inv_kn;
    }
  }
  __syncthreads();
  TNRC_TOC(w, 2, t_r);
  TNRC_TIC(t_w);
  const int k = ws->k;
  right_vectors(X, ldx, nrm, bf, n, k, h.T, ti, nt);
  __syncthreads();
  theta_split<kD>(Y, slot, b, h.T, h.Phi, k, ws->part[0], ti, nt);
  __syncthreads();
  if (ti == 0) slot_dims(slot)[b + 1] = k;
  __syncthreads();
  TNRC_TOC(w, 3, t_w);
}

constexpr int kPairSide = 64;

// Bonds a warp takes at a time.  Two, with small ones as a pair, on chains of 33
// sites or more; one below that, where pairs leave warps without a bond (8 qubits,
// 4 bonds a layer: 5.9 ms two at a time, 4.7 one).  By the layer's bonds only, so
// that results do not depend on the launch.  ms one / two at a time, gradient, 16
// slices, 152 trajectories as 8 x 1 and 304 as 4 x 2:
//            near a solution (bonds to 9)       random controls (bonds to 19)
//   sites    8 x 1          4 x 2               8 x 1          4 x 2
//   20        7.6 /  8.7    13.1 / 11.2         13.8 / 17.5    21.0 / 21.9
//   26       11.0 / 10.0    16.8 / 15.6         15.1 / 15.6    22.4 / 23.7
//   33       12.9 / 11.4    22.4 / 18.5         17.6 / 18.4    29.9 / 27.9
//   38       15.8 / 14.5    25.9 / 22.0         21.1 / 20.7    34.4 / 32.8
//   50       19.2 / 18.5    33.9 / 27.0         27.1 / 28.9    46.7 / 43.5
__device__ __forceinline__ int group_size(const TrajParams& p) { return p.N - 1 >= 32 ? 2 : 1; }

// Whether bonds b1 and b2 of one layer are updated as a pair: pairing is on
// for the context (the matrix shape the autotuner picks), both thetas and
// both Phis fit the warp's shared slab side by side, and every side is at
// most 64 (the per-warp SVD arrays are split in halves).
template <int kD>
__device__ __forceinline__ bool pair_fits(const TrajParams& p, const int* D, int b1, int b2) {
  const int m1 = kD * D[b1], n1 = kD * D[b1 + 2], m2 = kD * D[b2], n2 = kD * D[b2 + 2];
  return p.pair_svd && upd_elems(m1, n1) + upd_elems(m2, n2) <= p.slab_elems && m1 <= kPairSide && n1 <= kPairSide &&
         m2 <= kPairSide && n2 <= kPairSide;
}

// Where a pair update keeps its two thetas in the slab: theta, Phi, R^dagger and
// the pivot column of the first, then the same of the second.
template <int kD>
__device__ __forceinline__ double2* pair_theta(const TrajParams& p, const int* D, int b1, int which, WarpCtx& w) {
  return which == 0 ? w.slab : w.slab + upd_elems(kD * D[b1], kD * D[b1 + 2]);
}

// Two two-site updates (bonds b1, b2 of one layer, disjoint sites) by one
// warp: thetas built one after the other, then the QR and the Jacobi of both at
// once on the two half-warps, then ranks and splits one after the other.  The
// same arithmetic per bond as two_site_update, in another lane arrangement (so
// the same results up to the order of sums).
template <int kD>
__device__ __noinline__ void two_site_update_pair(const TrajParams& p, const Lay& Y, unsigned char* slot, int b1,
                                     const double2* G1, int b2, const double2* G2, bool adjoint, bool record,
                                     bool count, WarpCtx& w, bool have_pre = false) {
  const int lane = w.lane;
  const int* D = slot_dims(slot);
  const int m1 = kD * D[b1], n1 = kD * D[b1 + 2], m2 = kD * D[b2], n2 = kD * D[b2 + 2];
  double2* T1 = w.slab;
  double2* Phi1 = w.slab + m1 * n1;
  double2* T2 = w.slab + upd_elems(m1, n1);
  double2* Phi2 = T2 + m2 * n2;
  TNRC_TIC(t_c);
  const double fro1 = warp_sum(theta_build<kD>(p, Y, slot, b1, G1, adjoint, T1, Phi1, have_pre, w.small, false));
  const double fro2 = warp_sum(theta_build<kD>(p, Y, slot, b2, G2, adjoint, T2, Phi2, have_pre, w.small + 16, false));
  __syncwarp();
  TNRC_TOC(w, 0, t_c);
  const SvdBufs bf1{w.sig2, w.qn, w.perm, w.piv};
  const SvdBufs bf2{w.sig2 + 64, w.qn + 64, w.perm + 64, w.piv + 64};
  const bool hi = lane >= 16;
  TNRC_TIC(t_j);
  flag_not_finite(p, fro1 + fro2, lane);
  const int ld1 = n1 | 1, ld2 = n2 | 1;
  int4* X1 = reinterpret_cast<int4*>(Phi1 + m1 * n1);
  int4* X2 = reinterpret_cast<int4*>(Phi2 + m2 * n2);
  const SvdBufs bf{hi ? bf2.sig2 : bf1.sig2, hi ? bf2.qn : bf1.qn, hi ? bf2.perm : bf1.perm, hi ? bf2.piv : bf1.piv};
  const int mh = hi ? m2 : m1, nh = hi ? n2 : n1, ldh = hi ? ld2 : ld1;
  int4* Xh = hi ? X2 : X1;
  const int rh = fx_qr(hi ? T2 : T1, Xh + (mh < nh ? mh : nh) * ldh, mh, nh, hi ? fro2 : fro1, Xh, ldh, bf.perm,
                       bf.piv, reinterpret_cast<float*>(bf.qn), reinterpret_cast<int*>(bf.sig2), lane, 16);
  int r1 = __shfl_sync(0xffffffffu, rh, 0), r2 = __shfl_sync(0xffffffffu, rh, 16);
  if (r1 < 1) {
    r1 = 1;
#pragma unroll 1
    for (int e = lane; e < n1; e += 32) X1[e] = make_int4(0, 0, 0, 0);
    if (lane == 0) bf1.perm[0] = 0;
  }
  if (r2 < 1) {
    r2 = 1;
#pragma unroll 1
    for (int e = lane; e < n2; e += 32) X2[e] = make_int4(0, 0, 0, 0);
    if (lane == 0) bf2.perm[0] = 0;
  }
  __syncwarp();
  TNRC_TOC(w, 1, t_j);
  TNRC_TIC(t_s);
  int* ex1 = reinterpret_cast<int*>(bf1.qn);
  int* ex2 = reinterpret_cast<int*>(bf2.qn);
  const int swh = fx_jacobi(Xh, ldh, nh, hi ? r2 : r1, bf.perm, hi ? ex2 : ex1, lane, 16);
  const int sw1 = __shfl_sync(0xffffffffu, swh, 0), sw2 = __shfl_sync(0xffffffffu, swh, 16);
  TNRC_TOC(w, 8, t_s);
  theta_finish<kD>(p, Y, slot, b1, X1, ld1, ex1, reinterpret_cast<ColNorm*>(X1 + (m1 < n1 ? m1 : n1) * ld1), T1, Phi1, r1,
                   sw1, record, count, w, bf1);
  theta_finish<kD>(p, Y, slot, b2, X2, ld2, ex2, reinterpret_cast<ColNorm*>(X2 + (m2 < n2 ? m2 : n2) * ld2), T2, Phi2, r2,
                   sw2, record, count, w, bf2);
}

// ---------------------------------------------------------------------------
// Read-only view of a stored state: a slot of a layout, or a packed record.
// A packed record holds D[N+1], the site offsets off[N] (complex elements) and
// the site tensors at their actual dimensions -- the layer history of the
// costate sweep is kept in this form.
// ---------------------------------------------------------------------------
struct StateView {
  const int* D;
  const int* off;
  const double2* sites;
};

__device__ __forceinline__ StateView slot_view(const unsigned char* slot, const Lay& Y) {
  return StateView{slot_dims(slot), Y.site_off, slot_sites(slot, Y.L)};
}

__device__ __forceinline__ size_t packed_header(int N) { return ((size_t)(2 * N + 1) * 4 + 15) / 16 * 16; }

__device__ __forceinline__ StateView packed_view(const unsigned char* rec, int N) {
  const int* D = reinterpret_cast<const int*>(rec);
  return StateView{D, D + N + 1, reinterpret_cast<const double2*>(rec + packed_header(N))};
}

// CTA-wide: write the packed record of `slot` to `rec`, unless it takes more than
// `room` bytes; returns its size (the same in every thread).  Every warp scans
// the site sizes, then copies every warps-th site: site after site by the whole
// CTA, with each size read from memory in turn, was a tenth of a small
// evaluation.
template <int kD>
__device__ __noinline__ size_t pack_state(const TrajParams& p, const Lay& Y, const unsigned char* slot,
                                          unsigned char* rec, size_t room) {
  const int N = p.N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int* D = slot_dims(slot);
  int* hd = reinterpret_cast<int*>(rec);
  double2* out = reinterpret_cast<double2*>(rec + packed_header(N));
  const double2* src = slot_sites(slot, Y.L);
  int total = 0;
#pragma unroll 1
  for (int i = lane; i < N; i += 32) total += D[i] * kD * D[i + 1];
  total = __reduce_add_sync(0xffffffffu, total);
  const size_t need = packed_header(N) + (size_t)total * 16;
  if (need > room) return need;
  int o = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < N; i0 += 32) {
    const int i = i0 + lane;
    const int cnt = i < N ? D[i] * kD * D[i + 1] : 0, from = i < N ? Y.site_off[i] : 0;
    int sum = cnt;
#pragma unroll 1
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, sum, d);
      if (lane >= d) sum += v;
    }
    const int at = o + sum - cnt;
    if (warp == 0 && i < N) {
      hd[i] = D[i];
      hd[N + 1 + i] = at;
    }
#pragma unroll 1
    for (int u = warp; u < 32 && i0 + u < N; u += nw) {
      const int c = __shfl_sync(0xffffffffu, cnt, u), f = __shfl_sync(0xffffffffu, from, u),
                t = __shfl_sync(0xffffffffu, at, u);
#pragma unroll 1
      for (int e = lane; e < c; e += 32) out[t + e] = src[f + e];
    }
    o += __shfl_sync(0xffffffffu, sum, 31);
  }
  if (threadIdx.x == 0) hd[N] = D[N];
  __syncthreads();
  return need;
}

// ---------------------------------------------------------------------------
// Transfer-matrix steps of <c| . |a>, in FP64.  (In 56-bit integers with one scale
// per tensor the gradient cases were 2 to 7 % faster, but sums of dense operators
// left the range and overlaps of weak controls lost their digits: an environment
// spans as many decades as the overlap does.)
// Left:  Eout[b'][a'] = sum_{b,s,a} conj(c[b][s][b']) Ein[b][a] a[a][s][a']
// Right: Eout[b][a]   = sum_{s,b',a'} conj(c[b][s][b']) Ein[b'][a'] a[a][s][a']
// ---------------------------------------------------------------------------

// Environments of a region: chi^2 elements per bond, L_0 .. L_N and R_0 .. R_N.
__device__ __forceinline__ double2* env_left(const TrajParams& p, int region) {
  return p.env_scratch + (size_t)region * 2 * (p.N + 1) * p.chi * p.chi;
}
__device__ __forceinline__ double2* env_right(const TrajParams& p, int region) {
  return env_left(p, region) + (size_t)(p.N + 1) * p.chi * p.chi;
}

// The team of one sweep meets at its named barrier; a single warp (team < 0)
// needs none.  Literal barrier numbers: with one in a register the kernel is given
// all 16.
__device__ __forceinline__ void team_sync(int team, int nt) {
  if (team < 0)
    __syncwarp();
  else if (team == 0)
    asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
  else
    asm volatile("bar.sync 2, %0;" ::"r"(nt) : "memory");
}

// One step by thread ti of nt, in FP64.  Left (team 0, or one warp with team -1):
// k runs over the left bonds.  Every element is summed by one thread in a fixed
// order, so results do not depend on the team.
template <int kD>
__device__ __noinline__ void env_step(int team, const double2* Ein, int D1, int K1, const double2* c, int cs1, int cs2,
                                      const double2* a, int as1, int as2, int D2, int Da2, double2* tmp, double2* Eout,
                                      int ti, int nt) {
  // tmp[i][s][y] = sum_k Ein[i][k] a(k, s, y), i < D1, k < K1, y < Da2; a(k, s, y) at
  // k as1 + s Da' + y as2 (s stride: Da2 on the left, K1 on the right)
  const bool left = team != 1;
  const int as_s = left ? Da2 : K1, w2 = kD * Da2;
#pragma unroll 1
  for (int it = ti; it < D1 * w2; it += nt) {
    const int i = it / w2, rest = it - i * w2, s = rest / Da2, y = rest - s * Da2;
    const double2* ap = a + s * as_s + y * as2;
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 2
    for (int k = 0; k < K1; ++k) cfma(acc, Ein[i * K1 + k], ap[k * as1]);
    tmp[it] = acc;
  }
  team_sync(team, nt);
  // Eout[x][y] = sum_{i,s} conj(c(i, s, x)) tmp[i][s][y], c(i, s, x) at i cs1 + s cs' + x cs2
  const int cs_s = left ? D2 : D1;
#pragma unroll 1
  for (int it = ti; it < D2 * Da2; it += nt) {
    const int x = it / Da2, y = it - x * Da2;
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int i = 0; i < D1; ++i)
#pragma unroll
      for (int s = 0; s < kD; ++s) cfmac(acc, c[i * cs1 + s * cs_s + x * cs2], tmp[i * w2 + s * Da2 + y]);
    Eout[it] = acc;
  }
  team_sync(team, nt);
}

// <t|a> by one warp.
template <int kD>
__device__ __noinline__ double2 warp_overlap(const TrajParams& p, const Lay& Yt, const unsigned char* tslot, const Lay& Ya,
                                const unsigned char* aslot, WarpCtx& w) {
  const int* Dt = slot_dims(tslot);
  const int* Da = slot_dims(aslot);
  const double2* ts = slot_sites(tslot, Yt.L);
  const double2* as = slot_sites(aslot, Ya.L);
  const size_t cc = (size_t)p.chi * p.chi;
  double2* E0 = w.scratch;
  double2* E1 = w.scratch + cc;
  double2* tmp = w.scratch + 2 * cc;
  if (w.lane == 0) E0[0] = make_double2(1.0, 0.0);
  __syncwarp();
#pragma unroll 1
  for (int i = 0; i < p.N; ++i) {
    env_step<kD>(-1, E0, Dt[i], Da[i], ts + Yt.site_off[i], kD * Dt[i + 1], 1, as + Ya.site_off[i], kD * Da[i + 1], 1,
                 Dt[i + 1], Da[i + 1], tmp, E1, w.lane, 32);
    double2* x = E0;
    E0 = E1;
    E1 = x;
  }
  return E0[0];
}

// Cost of a two-site update with theta of (2 Dl) x (2 Dr): the Jacobi work
// grows as m n min(m, n).
__device__ __forceinline__ long long update_cost(int Dl, int Dr) {
  const long long m = 2 * Dl, n = 2 * Dr;
  return m * n * (m < n ? m : n);
}

// Whether the update of bond b is shared by every warp of the CTA: its SVD does
// not fit the warp's shared slab, or it is a good part of the layer's work
// (more than a sixth; one warp would then still be at it when the others are
// done with the rest) and large enough for its rounds to occupy several warps
// (12 qubits at the cap, theta up to 64 x 64, 5 or 6 bonds a layer: 661 ms with one
// warp per bond, 130 ms shared).  The rule looks at sizes and at the slab, and the
// work is cut into the same lane groups whatever the number of warps, so for one slab
// size results depend neither on that nor on what else runs.  Another launch shape or
// the allocation-free entry point, with another slab, may take a bond on another path:
// the same up to the order of sums.
constexpr int kWideSide = 16;
template <int kD>
__device__ __forceinline__ bool wide_update(const TrajParams& p, const int* D, int b, long long total) {
  const int m = kD * D[b], n = kD * D[b + 2];
  return svd_elems(m, n) > p.slab_elems ||
         ((m < n ? m : n) >= kWideSide && 6 * update_cost(D[b], D[b + 2]) > total);
}

// One warp: the bonds of parity `parity` in decreasing order of update cost
// into w.order, their total cost, and the shared counter reset.
static __device__ __noinline__ void order_layer(const TrajParams& p, const int* D, int parity, WarpCtx& w) {
  const int nb = (p.N - 1 - parity + 1) / 2;
  const int lane = w.lane;
  long long total = 0;
#pragma unroll 1
  for (int j = lane; j < nb; j += 32) {
    const long long cj = update_cost(D[parity + 2 * j], D[parity + 2 * j + 2]);
    int rk = 0;
#pragma unroll 1
    for (int i = 0; i < nb; ++i) {
      const long long ci = update_cost(D[parity + 2 * i], D[parity + 2 * i + 2]);
      rk += (ci > cj || (ci == cj && i < j)) ? 1 : 0;
    }
    w.order[rk] = parity + 2 * j;
    total += cj;
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
  if (lane == 0) {
    *w.next = 0;
    w.wide->total = total;
  }
}

// ---------------------------------------------------------------------------
// Gradient of one layer (App. A), split so that each bond's gradient and its
// costate update run back to back on one warp:
//   layer_envs    left/right environments of <c|.|a> for the layer, by the even
//                 and the odd warps;
//   bond_gradient the mixed two-site density rho of bond b and dO/du =
//                 tr(Q_u rho) for every control u of its gate, added to the
//                 trajectory's gradient row as 2 Re(conj(O) dO/du); it leaves
//                 the costate's two-site product c_b c_{b+1} where the costate
//                 update of the bond takes theta, which then skips its own
//                 contraction.
// ---------------------------------------------------------------------------
template <int kD>
__device__ __noinline__ void layer_envs(const TrajParams& p, const Lay& Y, const unsigned char* cslot, const StateView av,
                                        WarpCtx& w, int warp) {
  const int N = p.N;
  const size_t cc = (size_t)p.chi * p.chi;
  const int* Dc = slot_dims(cslot);
  const int* Da = av.D;
  const double2* cs = slot_sites(cslot, Y.L);
  double2* L = env_left(p, w.region);
  double2* R = env_right(p, w.region);

  // left environments L_i (sites < i) for i <= N-2 by the even warps, right
  // R_i (sites >= i) for i >= 2 by the odd warps: each sweep is sequential
  // over the sites, so each step is shared by its team of warps; the step's
  // intermediate (at most Dc x kD Da) sits in the team's first warp's shared
  // slab when it fits, else in its scratch.
  TNRC_TIC(t_e);
  const int team = warp & 1;                               // 0: left, 1: right
  const int nt = 32 * (team == 0 ? (p.warps + 1) / 2 : p.warps / 2);
  const int ti = (warp >> 1) * 32 + w.lane;
  double2* lead_slab = w.slab - (size_t)(warp - team) * p.slab_elems;
  double2* lead_scratch = w.scratch - (size_t)(warp - team) * p.scratch_elems;
#pragma unroll 1
  for (int t = 0; t < N - 2; ++t) {
    const int i = team == 0 ? t : N - 1 - t;               // the site taken in
    const int cl = Dc[i], cr = Dc[i + 1], al = Da[i], ar = Da[i + 1];
    const int n1 = kD * (team == 0 ? cl * ar : cr * al);
    double2* tmp = n1 <= p.slab_elems ? lead_slab : lead_scratch;
    const double2 *c = cs + Y.site_off[i], *a = av.sites + av.off[i];
    if (team == 0)
      env_step<kD>(0, L + i * cc, cl, al, c, kD * cr, 1, a, kD * ar, 1, cr, ar, tmp, L + (i + 1) * cc, ti, nt);
    else
      env_step<kD>(1, R + (i + 1) * cc, cr, ar, c, 1, kD * cr, a, 1, kD * ar, cl, al, tmp, R + i * cc, ti, nt);
    if (ti == 0) w.alg += 8ull * n1 * (unsigned long long)(team == 0 ? al : ar) + 8ull * kD * cl * cr * (team == 0 ? ar : al);
  }
  TNRC_TOC(w, 4, t_e);
}

// out[i][j] = sum_k A[i K + k] B(k, j), M x J outputs, B(k, j) at k bk + j bj.
static __device__ __noinline__ void small_gemm(const double2* A, const double2* B, int M, int K, int J, int bk, int bj,
                                               double2* out, int ti, int nt) {
#pragma unroll 1
  for (int it = ti; it < M * J; it += nt) {
    const int i = it / J, j = it - i * J;
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 2
    for (int k = 0; k < K; ++k) cfma(acc, A[i * K + k], B[k * bk + j * bj]);
    out[it] = acc;
  }
}

template <int kD>
__device__ __noinline__ void bond_gradient(const TrajParams& p, const Lay& Y, const unsigned char* cslot, const StateView av,
                              int s, int l, int b, double2 wO, double* gsp_row, WarpCtx& w, double2* Wc, bool cta) {
  constexpr int kDD = kD * kD, kI = kD / 2;
  const int chi = p.chi;
  const size_t cc = (size_t)chi * chi;
  const int* Dc = slot_dims(cslot);
  const int* Da = av.D;
  const double2* cs = slot_sites(cslot, Y.L);
  const int* so = Y.site_off;
  const double2* L = env_left(p, w.region) + (size_t)b * cc;
  const double2* R = env_right(p, w.region) + (size_t)(b + 2) * cc;
  const double2* a0 = av.sites + av.off[b];
  const double2* a1 = av.sites + av.off[b + 1];
  const int lane = w.lane;
  const int ti = cta ? (int)threadIdx.x : lane, nt = cta ? (int)blockDim.x : 32;
  auto sync = [&]() {
    if (cta)
      __syncthreads();
    else
      __syncwarp();
  };
  TNRC_TIC(t_g);
  const int dcl = Dc[b], dcm = Dc[b + 1], dcr = Dc[b + 2];
  const int dal = Da[b], dam = Da[b + 1], dar = Da[b + 2];
  const double2* c0 = cs + so[b];
  const double2* c1 = cs + so[b + 1];
  // the costate product c_b c_{b+1} is shared with the bond's costate update
  // (counted there)
  if (ti < 32)
    w.alg += 8ull * dcl * (kD * dam * dal + kDD * dar * dam + kDD * dcr * dar +
                           (unsigned long long)kDD * kDD * dcr) + 2048ull;
  // Wc = c_b c_{b+1} [dcl][kD^2][dcr] at Wc (theta's home); the other three
  // intermediates packed at their actual sizes right after it in the shared
  // slab when they fit there, else in global scratch past theta's room
  const int n1 = dcl * kD * dam, n2 = dcl * kDD * dar, n3 = dcl * kDD * dcr;
  double2* slab = cta ? w.cta_slab : w.slab;
  const int slab_elems = cta ? p.cta_slab_elems : p.slab_elems;
  const bool wc_in_slab = Wc >= slab && Wc < slab + slab_elems;
  double2* U1 = (wc_in_slab && (Wc - slab) + n3 + n1 + n2 + n3 <= slab_elems)
                    ? Wc + n3
                    : (cta ? w.cta_scratch : w.scratch) + (size_t)2 * kDD * chi * chi;
  double2* U2 = U1 + n1;   // U1 [dcl][kD][dam], U2 [dcl][kD^2][dar]
  double2* U3 = U2 + n2;   // [dcl][kD^2][dcr]
  small_gemm(L, a0, dcl, dal, kD * dam, kD * dam, 1, U1, ti, nt);
#pragma unroll 1
  for (int it = ti; it < dcl * kDD * dcr; it += nt) {
    const int be = it / (kDD * dcr), rest = it - be * kDD * dcr;
    const int ss = rest / dcr, b2 = rest - ss * dcr;
    const int s1 = ss / kD, s2 = ss % kD;
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int b1 = 0; b1 < dcm; ++b1)
      cfma(acc, c0[(size_t)be * kD * dcm + s1 * dcm + b1], c1[(size_t)b1 * kD * dcr + s2 * dcr + b2]);
    Wc[it] = acc;
  }
  sync();
  small_gemm(U1, a1, dcl * kD, dam, kD * dar, kD * dar, 1, U2, ti, nt);
  sync();
  small_gemm(U2, R, dcl * kDD, dar, dcr, 1, dar, U3, ti, nt);
  sync();
  // rho[o'][o] = sum_{i1,i2} sum_{be,b2} U3[be][s'][b2] conj(Wc[be][s][b2]) over the
  // two-site out indices o (the in indices, if any, traced out: the gate acts
  // as Q (x) I); one (o', o) pair and a stride of be per thread: 2 parts for
  // one warp, 8 for a wide bond, added in fixed order
  double2* rho = cta ? w.cta_small : w.small;
  {
    const int parts = cta ? 8 : 2;
    double2* sums = cta ? w.cta_small : w.small;   // at least two warps' 64 elements
#pragma unroll 1
    for (int it = ti; it < 16 * parts; it += nt) {
      const int o = it & 15, part = it >> 4;
      const int op = o >> 2, oq = o & 3;
      double2 acc = make_double2(0.0, 0.0);
#pragma unroll 1
      for (int ii = 0; ii < kI * kI; ++ii) {
        const int i1 = ii / kI, i2 = ii % kI;
        const int sp = ((op >> 1) * kI + i1) * kD + (op & 1) * kI + i2;
        const int sq = ((oq >> 1) * kI + i1) * kD + (oq & 1) * kI + i2;
#pragma unroll 1
        for (int be = part; be < dcl; be += parts) {
          const double2* u = U3 + (size_t)be * kDD * dcr + sp * dcr;
          const double2* wv = Wc + (size_t)be * kDD * dcr + sq * dcr;
#pragma unroll 1
          for (int b2 = 0; b2 < dcr; ++b2) cfmac(acc, wv[b2], u[b2]);
        }
      }
      sums[it] = acc;
    }
    sync();
    if (ti < 16) {
      double2 acc = sums[ti];
#pragma unroll 1
      for (int q = 1; q < parts; ++q) {
        acc.x += sums[q * 16 + ti].x;
        acc.y += sums[q * 16 + ti].y;
      }
      rho[ti] = acc;
    }
    __syncwarp();
  }
  // dO/du_q = tr(Q_q rho) = sum_ij Q_q[i][j] rho[j][i]: control q by four lanes,
  // one row i each
  if (ti < 32) {
    const LayerGate& lg = layer_rec(p, s, l, b);
    const int nq = lg.nq;
#pragma unroll 1
    for (int q0 = 0; q0 < nq; q0 += 8) {
      const int q = q0 + (lane >> 2), i = lane & 3;
      double2 v = make_double2(0.0, 0.0);
      if (q < nq) {
        const double2* Q = lg.Q[q] + i * 4;
#pragma unroll
        for (int j = 0; j < 4; ++j) cfma(v, Q[j], rho[j * 4 + i]);
      }
      double t = fma(wO.x, v.x, wO.y * v.y);
      t += __shfl_xor_sync(0xffffffffu, t, 1);
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      if (q < nq && i == 0) gsp_row[lg.slot[q]] += 2.0 * t;
    }
  }
  sync();
  TNRC_TOC(w, 5, t_g);
}

// ---------------------------------------------------------------------------
// Copy the used part of a state slot; src and dst may use different layouts.
// Returns 1 (and copies nothing) when a dimension exceeds dst's capacity.
template <int kD>
__device__ __noinline__ int copy_slot(const TrajParams& p, const Lay& Ys, const unsigned char* src, const Lay& Yd,
                         unsigned char* dst) {
  __syncthreads();
  const int* Ds = slot_dims(src);
  int* Dd = slot_dims(dst);
  const int tid = threadIdx.x, nt = blockDim.x;
  int bad = 0;
#pragma unroll 1
  for (int i = tid; i <= p.N; i += nt) bad |= (Ds[i] > Yd.dcap[i]) ? 1 : 0;
  if (__syncthreads_or(bad)) return 1;
#pragma unroll 1
  for (int i = tid; i <= p.N; i += nt) Dd[i] = Ds[i];
  const double* ls = slot_lam(src, Ys.L);
  double* ld = slot_lam(dst, Yd.L);
#pragma unroll 1
  for (int b = 0; b < p.N - 1; ++b) {
    const int d = Ds[b + 1];
#pragma unroll 1
    for (int j = tid; j < d; j += nt) ld[(size_t)b * Yd.L.chi + j] = ls[(size_t)b * Ys.L.chi + j];
  }
  const double2* ss = slot_sites(src, Ys.L);
  double2* sd = slot_sites(dst, Yd.L);
#pragma unroll 1
  for (int i = 0; i < p.N; ++i) {
    const int cnt = Ds[i] * kD * Ds[i + 1];
    const double2* a = ss + Ys.site_off[i];
    double2* b = sd + Yd.site_off[i];
#pragma unroll 1
    for (int e = tid; e < cnt; e += nt) b[e] = a[e];
  }
  __syncthreads();
  return 0;
}

// Entries e and e+1 of the layer's bond order (w.order, nb entries): one
// warp updates both, as a pair when both are small (two_site_update_pair),
// else one after the other.  The grouping depends only on the order, the bond
// dimensions and the slab, not on which warp or CTA takes it, so every launch form
// of one shape computes the same thing.
template <int kD>
__device__ __noinline__ void forward_group(const TrajParams& p, const Lay& Y, unsigned char* slot, int s, int l, int e, int nb,
                              bool adjoint, bool record, bool count, WarpCtx& w) {
  const int b1 = w.order[e];
  const int b2 = (group_size(p) == 2 && e + 1 < nb) ? w.order[e + 1] : -1;
  if (b2 >= 0 && pair_fits<kD>(p, slot_dims(slot), b1, b2)) {
    two_site_update_pair<kD>(p, Y, slot, b1, layer_rec(p, s, l, b1).G, b2, layer_rec(p, s, l, b2).G, adjoint,
                             record, count, w);
    return;
  }
  two_site_update<kD>(p, Y, slot, b1, layer_rec(p, s, l, b1).G, adjoint, record, count, w);
  if (b2 >= 0) two_site_update<kD>(p, Y, slot, b2, layer_rec(p, s, l, b2).G, adjoint, record, count, w);
}

// Wide bonds at the head of the layer's order (the cost order puts them first;
// a long thin theta further down is picked out too), by the whole CTA one
// after the other; they are taken out of the order.  Returns the number of
// bonds left.
template <int kD, class F>
__device__ int wide_bonds(const TrajParams& p, const int* D, int nb, WarpCtx& w, F update) {
  int left = 0;
#pragma unroll 1
  for (int e = 0; e < nb; ++e) {
    const int b = w.order[e];
    if (wide_update<kD>(p, D, b, w.wide->total)) {
      update(b);
    } else {
      __syncthreads();   // every thread has read order[left] before it is overwritten
      if (threadIdx.x == 0) w.order[left] = b;
      ++left;
    }
  }
  __syncthreads();
  return left;
}
template <int kD>
__device__ bool any_wide(const TrajParams& p, const int* D, int nb, const WarpCtx& w) {
  bool any = false;
#pragma unroll 1
  for (int e = 0; e < nb; ++e) any = any || wide_update<kD>(p, D, w.order[e], w.wide->total);
  return any;
}

// All bonds of truncated layer l.  The warps take bonds from a shared counter
// in decreasing order of cost (largest SVD first), so that they reach the
// layer barrier together; a bond's result does not depend on which warp
// computes it.
template <int kD>
__device__ void apply_layer(const TrajParams& p, const Lay& Y, unsigned char* slot, int s, int l, bool adjoint,
                            bool record, bool count, WarpCtx& w, int warp) {
  const int parity = layer_parity(p, l);
  int nb = (p.N - 1 - parity + 1) / 2;
  const int lane = w.lane;
  if (warp == 0) order_layer(p, slot_dims(slot), parity, w);
  __syncthreads();
  if (any_wide<kD>(p, slot_dims(slot), nb, w))
    nb = wide_bonds<kD>(p, slot_dims(slot), nb, w, [&](int b) {
      wide_update_cta<kD>(p, Y, slot, b, layer_rec(p, s, l, b).G, adjoint, record, count, w);
    });
  for (;;) {
    int e = 0;
    if (lane == 0) e = atomicAdd(w.next, group_size(p));
    e = __shfl_sync(0xffffffffu, e, 0);
    if (e >= nb) break;
    forward_group<kD>(p, Y, slot, s, l, e, nb, adjoint, record, count, w);
  }
  TNRC_TIC(t_b);
  __syncthreads();
  TNRC_TOC(w, 7, t_b);
}

// Entries e and e+1 of the layer's bond order: each bond's gradient and its
// costate update, the two updates as a pair when both bonds are small (the
// grouping rule of forward_group).
template <int kD>
__device__ __noinline__ void costate_group(const TrajParams& p, const Lay& Y, unsigned char* cslot, const StateView av, int s,
                              int l, int e, int nb, double2 wO, double* gsp_row, WarpCtx& w) {
  const int* Dc = slot_dims(cslot);
  const int b1 = w.order[e];
  const int b2 = (group_size(p) == 2 && e + 1 < nb) ? w.order[e + 1] : -1;
  if (b2 >= 0 && pair_fits<kD>(p, Dc, b1, b2)) {
    double2* th1 = pair_theta<kD>(p, Dc, b1, 0, w);
    double2* th2 = pair_theta<kD>(p, Dc, b1, 1, w);
    bond_gradient<kD>(p, Y, cslot, av, s, l, b1, wO, gsp_row, w, th1, false);
    bond_gradient<kD>(p, Y, cslot, av, s, l, b2, wO, gsp_row, w, th2, false);
    two_site_update_pair<kD>(p, Y, cslot, b1, layer_rec(p, s, l, b1).G, b2, layer_rec(p, s, l, b2).G, true, false,
                             true, w, true);
    return;
  }
#pragma unroll 1
  for (int q = 0; q < 2; ++q) {
    const int b = q == 0 ? b1 : b2;
    if (b < 0) break;
    bond_gradient<kD>(p, Y, cslot, av, s, l, b, wO, gsp_row, w, w.slab, false);
    two_site_update<kD>(p, Y, cslot, b, layer_rec(p, s, l, b).G, true, false, true, w, true);
  }
}

// One layer of the costate sweep (App. A): the environments of <c_l|.|a_l>,
// then every bond of layer l -- largest first from the shared counter -- its
// gradient and at once its costate update
// c_{l-1} = G^dag c_l, which reuses the product c_b c_{b+1} the gradient
// formed.  A bond's gradient reads only its own two costate sites and the
// environments; its update rewrites those two sites, which no other bond of
// the layer touches.
template <int kD>
__device__ void costate_layer(const TrajParams& p, const Lay& Y, unsigned char* cslot, const StateView av, int s,
                              int l, double2 wO, double* gsp_row, WarpCtx& w, int warp) {
  const int parity = layer_parity(p, l);
  int nb = (p.N - 1 - parity + 1) / 2;
  const int lane = w.lane;
  const int* Dc = slot_dims(cslot);
  if (warp == p.warps - 1) order_layer(p, Dc, parity, w);
  if (threadIdx.x == 0) {
    env_left(p, w.region)[0] = make_double2(1.0, 0.0);
    env_right(p, w.region)[(size_t)p.N * p.chi * p.chi] = make_double2(1.0, 0.0);
  }
  __syncthreads();
  layer_envs<kD>(p, Y, cslot, av, w, warp);
  __syncthreads();
  if (any_wide<kD>(p, Dc, nb, w))
    nb = wide_bonds<kD>(p, Dc, nb, w, [&](int b) {
      double2* th = wide_home<kD>(p, kD * Dc[b], kD * Dc[b + 2], w).T;
      bond_gradient<kD>(p, Y, cslot, av, s, l, b, wO, gsp_row, w, th, true);
      __syncthreads();
      wide_update_cta<kD>(p, Y, cslot, b, layer_rec(p, s, l, b).G, true, false, true, w, true);
    });
  for (;;) {
    int e = 0;
    if (lane == 0) e = atomicAdd(w.next, group_size(p));
    e = __shfl_sync(0xffffffffu, e, 0);
    if (e >= nb) break;
    costate_group<kD>(p, Y, cslot, av, s, l, e, nb, wO, gsp_row, w);
  }
  TNRC_TIC(t_b);
  __syncthreads();
  TNRC_TOC(w, 7, t_b);
}

// One trajectory (sample s, input pi) with the CTA's work region `base`.
//   packed = true : every layer state of the forward pass is kept as a packed
//                   record in the region (no recomputation in the costate
//                   sweep); returns 1 if the history outgrows the region.
//   packed = false: checkpoints every Y.seg layers and recomputation of each
//                   segment (fits by construction).
template <int kD>
__device__ __noinline__ int run_trajectory(const TrajParams& p, bool packed, unsigned char* base, int t, int s, int pi,
                              WarpCtx& w, int warp, double* s_disc, int* s_maxk, double2* s_O) {
  const Lay& Y = p.full;
  const int lane = w.lane;
  const size_t sb = (size_t)Y.L.bytes;
  const int L = p.n_layers;  // truncated layers
  unsigned char* a_slot = base;
  unsigned char* c_slot = base + sb;
  unsigned char* ckpt = base + 2 * sb;
  unsigned char* segs = ckpt + (size_t)Y.nseg * sb;
  long long* hpos = reinterpret_cast<long long*>(base + 2 * sb);  // packed mode: record offsets
  unsigned char* harena = base + 2 * sb + (((size_t)L * 8 + 255) / 256) * 256;
  const size_t hbytes = min((size_t)p.work_stride - (size_t)(harena - base), (size_t)p.history_cap);
  const int KCN = p.K * p.C * p.N;
  w.disc = 0.0;
  w.maxk = 0;
  copy_slot<kD>(p, Y, p.in_slots + (size_t)pi * sb, Y, a_slot);
  // ---- forward ----
  size_t pos = 0;
#pragma unroll 1
  for (int l = 0; l < L; ++l) {
    const int q = l / Y.seg;
    if (p.want_grad && !packed && (l % Y.seg) == 0 && q < Y.nseg - 1) copy_slot<kD>(p, Y, a_slot, Y, ckpt + (size_t)q * sb);
    apply_layer<kD>(p, Y, a_slot, s, l, false, true, true, w, warp);
    if (p.want_grad) {
      if (packed) {
        TNRC_TIC(t_h);
        const size_t room = pos < hbytes ? hbytes - pos : 0, need = pack_state<kD>(p, Y, a_slot, harena + pos, room);
        TNRC_TOC(w, 6, t_h);
        if (need > room) return 1;
        if (threadIdx.x == 0) hpos[l] = (long long)pos;
        pos += (need + 255) / 256 * 256;
      } else if (q == Y.nseg - 1) {
        copy_slot<kD>(p, Y, a_slot, Y, segs + (size_t)(l - q * Y.seg) * sb);
      }
    }
  }
  const unsigned char* tg = p.tg_slots + (size_t)pi * sb;
  if (warp == 0) {
    const double2 O = warp_overlap<kD>(p, Y, tg, Y, a_slot, w);
    if (lane == 0) *s_O = O;
    const int* Dt = slot_dims(tg);
    const int* Da = slot_dims(a_slot);
#pragma unroll 1
    for (int i = 0; i < p.N; ++i)
      w.alg += 8ull * kD * Da[i + 1] * (unsigned long long)(Dt[i] * Da[i] + Dt[i + 1] * Dt[i]);
  }
  if (lane == 0) {
    s_disc[warp] = w.disc;
    s_maxk[warp] = w.maxk;
  }
  __syncthreads();
  const double2 O = *s_O;
  if (threadIdx.x == 0) {
    p.O[t] = O;
    double d = 0.0;
    int mk = 0;
#pragma unroll 1
    for (int i = 0; i < p.warps; ++i) {
      d += s_disc[i];
      mk = max(mk, s_maxk[i]);
    }
    p.disc[t] = d;
    atomicMax(&p.counters[2], (unsigned long long)mk);
  }
  if (!p.want_grad) return 0;
  // ---- costate sweep ----
  double* grow = p.gsp + (size_t)t * KCN;
#pragma unroll 1
  for (int i = threadIdx.x; i < KCN; i += blockDim.x) grow[i] = 0.0;
  copy_slot<kD>(p, Y, tg, Y, c_slot);
  if (packed) {
#pragma unroll 1
    for (int l = L - 1; l >= 0; --l)
      costate_layer<kD>(p, Y, c_slot, packed_view(harena + hpos[l], p.N), s, l, O, grow, w, warp);
    return 0;
  }
#pragma unroll 1
  for (int q = Y.nseg - 1; q >= 0; --q) {
    const int l0 = q * Y.seg;
    const int l1 = min(L, l0 + Y.seg);
    if (q != Y.nseg - 1) {
      unsigned char* ck = ckpt + (size_t)q * sb;
#pragma unroll 1
      for (int l = l0; l < l1; ++l) {
        apply_layer<kD>(p, Y, ck, s, l, false, false, false, w, warp);
        copy_slot<kD>(p, Y, ck, Y, segs + (size_t)(l - l0) * sb);
      }
    }
#pragma unroll 1
    for (int l = l1 - 1; l >= l0; --l)
      costate_layer<kD>(p, Y, c_slot, slot_view(segs + (size_t)(l - l0) * sb, Y), s, l, O, grow, w, warp);
  }
  return 0;
}

// Compiled twice: kMinBlocks = 1 without a limit on registers (210 a thread, 208 for
// operators: nine warps would fit an SM, launches use up to eight); kMinBlocks = 2
// with at most 128 so that 16 warps fit, trading a few spilled values for twice the
// warps to hide latency.
template <int kMinBlocks, int kD>
__global__ void __launch_bounds__(kWarps * 32, kMinBlocks) traj_kernel(TrajParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_item;
  __shared__ double s_disc[kWarps];
  __shared__ int s_maxk[kWarps];
  __shared__ double2 s_O;
  __shared__ int s_order[128];
  __shared__ int s_next;
  __shared__ int s_region;
  __shared__ WideShared s_wide;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  double2* slabs = reinterpret_cast<double2*>(smem_raw);
  double* sig = reinterpret_cast<double*>(slabs + (size_t)p.warps * p.slab_elems);
  double* qns = sig + (size_t)p.warps * kMaxDim;
  int* perms = reinterpret_cast<int*>(qns + (size_t)p.warps * kMaxDim);
  int* pivs = perms + (size_t)p.warps * kMaxDim;
  double2* smalls = reinterpret_cast<double2*>(pivs + (size_t)p.warps * kMaxDim);

  // pooled launch: take a free work region (bounded scan; a full pool cannot
  // happen while n_regions covers the CTAs that can be resident at once)
  int region = blockIdx.x;
  if (p.pooled) {
    if (blockIdx.x >= p.T) return;
    if (threadIdx.x == 0) {
      int got = -1;
#pragma unroll 1
      for (int attempt = 0; attempt < kRegionTries && got < 0; ++attempt) {
#pragma unroll 1
        for (int i = 0; i < p.n_regions; ++i) {
          const int r = (int)((blockIdx.x + (unsigned)i) % (unsigned)p.n_regions);
          if (atomicCAS(&p.region_owner[r], 0, 1) == 0) {
            got = r;
            break;
          }
        }
        if (got < 0) __nanosleep(16000);
      }
      s_region = got;
    }
    __syncthreads();
    region = s_region;
    if (region < 0) {
      if (threadIdx.x == 0) atomicOr(p.status, kStatusTimeout);
      return;
    }
  }
  WarpCtx w;
  w.region = region;
  w.slab = slabs + (size_t)warp * p.slab_elems;
  w.scratch = p.warp_scratch + ((size_t)region * p.warps + warp) * p.scratch_elems;
  w.sig2 = sig + (size_t)warp * kMaxDim;
  w.perm = perms + (size_t)warp * kMaxDim;
  w.qn = qns + (size_t)warp * kMaxDim;
  w.piv = pivs + (size_t)warp * kMaxDim;
  w.small = smalls + (size_t)warp * 64;
  w.lane = lane;
  w.cta_slab = slabs;
  w.cta_scratch = p.warp_scratch + (size_t)region * p.warps * p.scratch_elems;
  w.cta_small = smalls;
  w.cta_sig2 = sig;
  w.cta_qn = qns;
  w.cta_perm = perms;
  w.cta_piv = pivs;
  w.wide = &s_wide;
  w.sweeps = 0;
  w.updates = 0;
  w.alg = 0;
  w.capcuts = 0;
#pragma unroll 1
  for (int i = 0; i < kNumPhases; ++i) w.ph[i] = 0;
  w.order = s_order;
  w.next = &s_next;
  unsigned char* base = p.work + (size_t)region * p.work_stride;

#pragma unroll 1
  for (int iter = 0;; ++iter) {
    if (threadIdx.x == 0) s_item = p.pooled ? (iter == 0 ? (int)blockIdx.x : p.T) : atomicAdd(p.work_counter, 1);
    __syncthreads();
    const int t = s_item;
    __syncthreads();
    if (t >= p.T) break;
    const int s = t / p.P, pi = t - s * p.P;
    bool redo = true;
    if (p.want_grad && p.packed_history) {
      const long long sw0 = w.sweeps, up0 = w.updates, cc0 = w.capcuts;
      const unsigned long long al0 = w.alg;
      redo = run_trajectory<kD>(p, true, base, t, s, pi, w, warp, s_disc, s_maxk, &s_O) != 0;
      if (redo) {  // history outgrew the region: discard the attempt's counts, count the fallback
        w.sweeps = sw0;
        w.updates = up0;
        w.alg = al0;
        w.capcuts = cc0;
        if (threadIdx.x == 0) atomicAdd(&p.counters[4], 1ull);
      }
    }
    if (redo) run_trajectory<kD>(p, false, base, t, s, pi, w, warp, s_disc, s_maxk, &s_O);
  }
  if (lane == 0) {
    atomicAdd(&p.counters[0], (unsigned long long)w.updates);
    atomicAdd(&p.counters[1], (unsigned long long)w.sweeps);
    atomicAdd(&p.counters[3], w.alg);
    atomicAdd(&p.counters[kCtrCapTrunc], (unsigned long long)w.capcuts);
#ifdef TNRC_PHASE_TIMERS
#pragma unroll 1
    for (int i = 0; i < kNumPhases; ++i) atomicAdd(&p.counters[kCtrPhase + i], (unsigned long long)w.ph[i]);
#endif
  }
  if (p.pooled) {   // hand the region back once every thread is done with it
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicExch(&p.region_owner[region], 0);
    }
  }
}

}  // namespace tnrc
