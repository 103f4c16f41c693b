// Warp-level one-sided (Hestenes) Jacobi SVD in FP64, which brings inputs and
// targets to canonical form (canon.cu), and the rank and truncation decision of
// the TEBD compression step (Sec. II: "compressed after each time step ...
// using truncated singular-value decomposition"), whose SVD is svd_fx.cuh.
//
// The matrix is held column-major (column j at T + j*n, n rows).  Its m
// columns are orthogonalised by plane rotations in the round-robin (circle)
// ordering, m/2 disjoint pairs per round, so that a whole round runs in
// parallel: each pair gets g lanes (g * pairs <= 32), each lane owns rows
// lig, lig+g, ...; the three inner products of a pair are reduced over its g
// lanes by shuffles (bitwise identical in every lane, so every lane takes the
// same decision).  After convergence column j equals
// sigma_j y_j with y_j orthonormal: for T = M^dagger, y_j are the right
// singular vectors of M and sigma_j its singular values.
#pragma once
#include "tnrc_device.cuh"

namespace tnrc {

__device__ __forceinline__ void rr_pair(int mp, int r, int q, int& i, int& j) {
  if (q == 0) {
    i = r;
    j = mp - 1;
  } else {
    const int m1 = mp - 1;
    i = (r + q) % m1;
    j = (r - q + m1) % m1;
  }
}

// Sum of v over the g lanes gb .. gb+g-1 of this lane's group (lig = lane -
// gb, gmask = those lanes); every lane of the group receives the same value.
// A power-of-two g uses an xor butterfly; any other g a shift-down tree into
// lane gb and a broadcast from it (a source lane outside the group is never
// added).
template <class T>
__device__ __forceinline__ T group_sum(T v, int g, int lig, int gb, unsigned gmask) {
  if ((g & (g - 1)) == 0) {
    for (int o = g >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(gmask, v, o);
    return v;
  }
  int o = 1;
  while (2 * o < g) o <<= 1;
  for (; o > 0; o >>= 1) {
    const T x = __shfl_down_sync(gmask, v, o);
    if (lig + o < g) v += x;
  }
  return __shfl_sync(gmask, v, gb);
}

__device__ __forceinline__ unsigned group_mask(int g, int gb) {
  return (g >= 32) ? 0xffffffffu : (((1u << g) - 1u) << gb);
}

// out[c] = |column c|^2 for the m columns of length n of T (column-major),
// with g = 32 / m lanes per column (any g), so that short columns keep most
// lanes busy.
__device__ inline void warp_col_norms(const double2* T, int n, int m, double* out, int lane) {
  const int g = (m >= 32 || m < 1) ? 1 : 32 / m;
  const int gi = lane / g, lig = lane - gi * g, gb = gi * g;
  const int groups = 32 / g;
  const unsigned gmask = group_mask(g, gb);
  for (int c = gi; c < m && gi < groups; c += groups) {
    const double2* col = T + (size_t)c * n;
    double s = 0.0;
    for (int row = lig; row < n; row += g) s = fma(col[row].x, col[row].x, fma(col[row].y, col[row].y, s));
    if (g > 1) s = group_sum(s, g, lig, gb, gmask);
    if (lig == 0) out[c] = s;
  }
  __syncwarp();
}

// Returns the number of sweeps (the last one made no rotation, or only
// rotations with |cos| <= 1e-10 between the pair's columns), or -kMaxSweeps
// when the sweep limit was reached.  fro2 = squared Frobenius norm of T;
// cn: shared scratch of m doubles holding the column norms squared.
//
// Lanes per pair: an odd m is padded with a zero column, which the circle
// ordering pairs with a different real column in every round (pair q = 0);
// that pair needs no work, so the Pe = floor(m / 2) real pairs of a round
// share the 32 lanes, g = floor(32 / Pe) each (not necessarily a power of two).
// Each lane then owns ceil(n / g) rows of its pair.
//
// The norms are computed exactly before the first sweep and in the first
// round of every sweep (where the pair's lanes form all three inner
// products); in the other rounds only <a, b> is formed and the norms are
// carried through each rotation by |a'|^2 = |a|^2 - t |<a,b>|,
// |b'|^2 = |b|^2 + t |<a,b>| (t = tan theta), recomputed from the rotated
// column should a norm fall below 1/16 of its old value (cancellation).
__device__ inline int warp_jacobi(double2* T, int n, int m, double fro2, double* cn, int lane) {
  const int mp = m + (m & 1);
  if (mp < 2 || n < 1) return 0;
  const int P = mp >> 1;
  const int q0 = m & 1;          // pair 0 holds the padding column of an odd m
  const int Pe = P - q0;         // real pairs per round
  if (Pe < 1) return 1;          // a single column is already orthogonal
  const int g = Pe >= 32 ? 1 : 32 / Pe;
  const int groups = 32 / g;
  const int gi = lane / g, lig = lane - gi * g, gb = gi * g;
  const unsigned gmask = group_mask(g, gb);
  const double thr = kJacobiZero * kJacobiZero * fro2;
  const double tol = 2.0 * (double)(m > n ? m : n) * 2.220446049250313e-16;
  const double tol2 = tol * tol;
  warp_col_norms(T, n, m, cn, lane);
  for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
    int rotated = 0, large = 0;
    for (int r = 0; r < mp - 1; ++r) {
      for (int q = q0 + gi; q < P && gi < groups; q += groups) {
        int i, j;
        rr_pair(mp, r, q, i, j);
        double2* a = T + (size_t)i * n;
        double2* b = T + (size_t)j * n;
        double aa, bb;
        double2 ab = make_double2(0.0, 0.0);
        if (r == 0) {
          aa = 0.0;
          bb = 0.0;
          for (int row = lig; row < n; row += g) {
            const double2 x = a[row], y = b[row];
            aa = fma(x.x, x.x, fma(x.y, x.y, aa));
            bb = fma(y.x, y.x, fma(y.y, y.y, bb));
            cfmac(ab, x, y);
          }
          if (g > 1) {
            aa = group_sum(aa, g, lig, gb, gmask);
            bb = group_sum(bb, g, lig, gb, gmask);
            ab.x = group_sum(ab.x, g, lig, gb, gmask);
            ab.y = group_sum(ab.y, g, lig, gb, gmask);
          }
        } else {
          aa = cn[i];
          bb = cn[j];
          for (int row = lig; row < n; row += g) cfmac(ab, a[row], b[row]);
          if (g > 1) {
            ab.x = group_sum(ab.x, g, lig, gb, gmask);
            ab.y = group_sum(ab.y, g, lig, gb, gmask);
          }
        }
        double na = aa, nb = bb;
        const double ab2 = cabs2(ab);
        const double pab = aa * bb;
        if (aa > thr && bb > thr && ab2 > tol2 * pab) {
          rotated = 1;
          large |= (ab2 > kJacobiQuad * pab) ? 1 : 0;
          // Real rotation of the pair after the phase of <a,b> is divided out,
          // cot(2 theta) = (|b|^2 - |a|^2) / (2 |<a,b>|).  With d = |b|^2 - |a|^2
          // and w = 1 / sqrt(d^2 + 4 |<a,b>|^2): cos 2theta = |d| w,
          // sin 2theta = 2 |<a,b>| w, c = sqrt((1 + cos 2theta) / 2) and
          // s e^{i phi} = sign(d) w / sqrt((1 + cos 2theta) / 2) <a,b> -- two
          // reciprocal square roots, no division, no cancellation.
          const double d = bb - aa;
          const double w = rsqrt(fma(d, d, 4.0 * ab2));
          const double hq = fma(0.5, fabs(d) * w, 0.5);   // c^2
          const double rc = rsqrt(hq);
          const double c = hq * rc;
          const double f = copysign(w * rc, d);
          const double2 sp = make_double2(f * ab.x, f * ab.y);  // s e^{i phi}
          // a <- c a - conj(sp) b ;  b <- c b + sp a
          for (int row = lig; row < n; row += g) {
            const double2 x = a[row], y = b[row];
            double2 na_ = cscale(x, c);
            na_.x = fma(-sp.x, y.x, na_.x);
            na_.x = fma(-sp.y, y.y, na_.x);
            na_.y = fma(-sp.x, y.y, na_.y);
            na_.y = fma(sp.y, y.x, na_.y);
            double2 nb_ = cscale(y, c);
            cfma(nb_, sp, x);
            a[row] = na_;
            b[row] = nb_;
          }
          // t |<a,b>| = sign(d) 2 |<a,b>|^2 w; c^2 = hq, s^2 = 1 - hq
          const double dl = copysign(2.0 * ab2 * w, d);
          na = fma(hq, aa, fma(1.0 - hq, bb, -dl));
          nb = fma(hq, bb, fma(1.0 - hq, aa, dl));
          if (na < 0.0625 * aa) {
            na = 0.0;
            for (int row = lig; row < n; row += g) na = fma(a[row].x, a[row].x, fma(a[row].y, a[row].y, na));
            if (g > 1) na = group_sum(na, g, lig, gb, gmask);
          }
          if (nb < 0.0625 * bb) {
            nb = 0.0;
            for (int row = lig; row < n; row += g) nb = fma(b[row].x, b[row].x, fma(b[row].y, b[row].y, nb));
            if (g > 1) nb = group_sum(nb, g, lig, gb, gmask);
          }
        }
        if (lig == 0) {
          cn[i] = na;
          cn[j] = nb;
        }
      }
      __syncwarp();
    }
    // converged: a sweep without rotations -- or one whose rotations all had
    // |cos| <= 1e-10 between the pair's columns, after which (the cyclic
    // method converging quadratically) the next sweep would find every
    // |cos| near 1e-20, far below tol, and rotate nothing
    if (!__any_sync(0xffffffffu, rotated) || !__any_sync(0xffffffffu, large)) return sweep + 1;
  }
  return -kMaxSweeps;
}

// Column norms, ranking and the truncation decision after warp_jacobi.
// sig2[j] = |column j|^2 (j < m); perm[i] = column of rank i (i <= k, i < m),
// ranks by decreasing sigma with ties broken by the smaller index.  Returns
// k = max(1, min(kcap, #{sigma_j > eps sigma_max})); kept2 / tot2 receive the
// squared norms of the kept values and of all values.  When the cap decided
// the cut (more than kcap values above the cutoff), gap = (sigma_(k) -
// sigma_(k+1)) / sigma_max, the relative distance between the last kept and
// the first dropped value; otherwise gap = -1.
__device__ inline int warp_rank_truncate(const double2* T, int n, int m, int kcap, double eps, double* sig2,
                                  int* perm, int lane, double& kept2, double& tot2, double& gap) {
  warp_col_norms(T, n, m, sig2, lane);
  double mx = 0.0, tot = 0.0;
#pragma unroll 1
  for (int j = lane; j < m; j += 32) {
    mx = fmax(mx, sig2[j]);
    tot += sig2[j];
  }
  mx = warp_max(mx);
  tot = warp_sum(tot);
  const double cut2 = eps * eps * mx;
  int cnt = 0;
#pragma unroll 1
  for (int j = lane; j < m; j += 32) cnt += (sig2[j] > cut2) ? 1 : 0;
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  int k = cnt < kcap ? cnt : kcap;
  if (k > n) k = n;  // at most n orthogonal columns of length n
  if (k < 1) k = 1;
#pragma unroll 1
  for (int j = lane; j < m; j += 32) {
    const long long vj = __double_as_longlong(sig2[j]);
    int rk = 0;
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
      const long long vi = __double_as_longlong(sig2[i]);
      rk += (vi > vj || (vi == vj && i < j)) ? 1 : 0;
    }
    if (rk <= k) perm[rk] = j;
  }
  __syncwarp();
  double kn = 0.0;
#pragma unroll 1
  for (int i = lane; i < k; i += 32) kn += sig2[perm[i]];
  kept2 = warp_sum(kn);
  tot2 = tot;
  gap = (cnt > k && k < m) ? (sqrt(sig2[perm[k - 1]]) - sqrt(sig2[perm[k]])) / sqrt(mx) : -1.0;
  return k;
}

}  // namespace tnrc
