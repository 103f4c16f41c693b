// The truncated SVD of the TEBD compression step in fixed point (fx.cuh), by
// one warp or, for two small matrices at once, by its two half-warps.
//
//   fx_qr      theta = Q R by modified Gram-Schmidt with column pivoting (Q not
//              kept), stopping at the numerical rank r: R is as accurate as
//              Householder's (Bjorck and Paige, SIAM J. Matrix Anal. Appl. 13,
//              1992), needs one reciprocal square root a step and no phases.
//   fx_jacobi  one-sided (Hestenes) Jacobi on the r columns of R^dagger in the
//              round-robin (circle) ordering: column j becomes sigma_j y_j with
//              y_j the right singular vectors of theta.  QR first, then Jacobi
//              on R^dagger is the method of Drmac and Veselic (SIAM J. Matrix
//              Anal. Appl. 29, 2008).
//
// lw lanes work on one matrix (32, or 16 with two matrices per warp: lane
// hb + ll, hb = 0 or 16; every loop with a warp-wide barrier runs to the
// larger of the two trip counts, the half that is done idling).  A column of a
// QR step or a pair of a Jacobi round gets the largest power of two up to lw / units lanes, which
// split its rows.
#pragma once
#include "fx.cuh"
#include "svd_warp.cuh"

namespace tnrc {

__device__ __forceinline__ Fx fx_re(int4 a) { return Fx{a.x, a.y}; }
__device__ __forceinline__ Fx fx_im(int4 a) { return Fx{a.z, a.w}; }
__device__ __forceinline__ int4 fx_pack(long long re, long long im) {
  const Fx r = fx_split(re), i = fx_split(im);
  return make_int4(r.hi, r.lo, i.hi, i.lo);
}

// re += a b, im += a b (complex), and with conj(a)
__device__ __forceinline__ void fx_cmac(FxAcc& re, FxAcc& im, int4 a, int4 b) {
  const Fx ar = fx_re(a), ai = fx_im(a), br = fx_re(b), bi = fx_im(b);
  fx_mac(re, ar, br);
  fx_mac(re, fx_neg(ai), bi);
  fx_mac(im, ar, bi);
  fx_mac(im, ai, br);
}
__device__ __forceinline__ void fx_cmacc(FxAcc& re, FxAcc& im, int4 a, int4 b) {
  const Fx ar = fx_re(a), ai = fx_im(a), br = fx_re(b), bi = fx_im(b);
  fx_mac(re, ar, br);
  fx_mac(re, ai, bi);
  fx_mac(im, ar, bi);
  fx_mac(im, fx_neg(ai), br);
}
// |a|^2: h 2^56 + 2 x 2^28
__device__ __forceinline__ void fx_cabs2(FxAcc& s, int4 a) {
  s.h += (long long)a.x * a.x;
  s.h += (long long)a.z * a.z;
  s.x += (long long)a.x * a.y;
  s.x += (long long)a.z * a.w;
}
__device__ __forceinline__ long long fx_sum2(FxAcc s) { return s.h + ((s.x + (1ll << 26)) >> 27); }

// |a|^2 in FP32, for scales and pivots
__device__ __forceinline__ float fx_cabs2f(int4 a) {
  const float r = fmaf((float)a.x, 268435456.0f, (float)a.y);
  const float i = fmaf((float)a.z, 268435456.0f, (float)a.w);
  return fmaf(r, r, i * i);
}

__device__ __forceinline__ int4 fx_shift(int4 a, int k) {   // a 2^k
  if (k >= 0) return fx_pack(fx_val(fx_re(a)) << k, fx_val(fx_im(a)) << k);
  const long long h = 1ll << (-k - 1);
  return fx_pack((fx_val(fx_re(a)) + h) >> -k, (fx_val(fx_im(a)) + h) >> -k);
}

// a 2^k for any k (what leaves the 64 bits on the right is zero)
__device__ __forceinline__ int4 fx_shift_any(int4 a, int k) { return fx_shift(a, k < -62 ? -62 : k); }

// x 2^k, and FP64 to fixed point
__device__ __forceinline__ double fx_scale(double x, int k) {
  const int h = __double2hiint(x), e = (h >> 20) & 2047;
  return (e == 0 || e + k <= 0) ? 0.0 : __hiloint2double(h + (k << 20), __double2loint(x));
}
__device__ __forceinline__ int4 fx_from_double2(double2 a, int k) {
  return fx_pack(__double2ll_rn(fx_scale(a.x, k)), __double2ll_rn(fx_scale(a.y, k)));
}

// Element access: the matrices of a warp are in shared memory (SH, 32-bit
// addresses) unless they are too wide for its slab.
template <bool SH>
struct FxMem {
  int4* g;
  unsigned s;
  __device__ __forceinline__ explicit FxMem(int4* p) : g(p), s(SH ? (unsigned)__cvta_generic_to_shared(p) : 0u) {}
  __device__ __forceinline__ int4 ld(int i) const {
    if (SH) {
      int4 v;
      asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                   : "r"(s + 16u * (unsigned)i)
                   : "memory");
      return v;
    }
    return g[i];
  }
  __device__ __forceinline__ void st(int i, int4 v) const {
    if (SH)
      asm volatile("st.shared.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(s + 16u * (unsigned)i), "r"(v.x), "r"(v.y),
                   "r"(v.z), "r"(v.w)
                   : "memory");
    else
      g[i] = v;
  }
};

// 2^k brings a vector of squared norm pn to a norm in [2^55, 2^56)
__device__ __forceinline__ int fx_pivot_shift(float pn) { return (111 - fx_ilog2f(pn)) >> 1; }
// squared norm at which columns count as zero, in units of 2^(2 E0)
__device__ __forceinline__ float fx_zero_norm2(double fro, int E0) {
  return (float)(kJacobiZero * kJacobiZero) * (float)fx_scale(fro, -2 * E0);
}

// log2 of the lanes per unit: the largest power of two <= LW / units (0 when
// there are more units than half the lanes)
__device__ __forceinline__ int fx_lanes(int units, int lw) {
  return units >= lw ? 0 : 31 - __clz(lw / (units < 1 ? 1 : units));
}
// the larger value of the warp's two halves
__device__ __forceinline__ int fx_umax(int v) { return (int)__reduce_max_sync(0xffffffffu, (unsigned)v); }

// ---------------------------------------------------------------------------
// Pivoted Gram-Schmidt of theta (m x n, row-major, FP64 in; W the same memory).
//
// theta's rows are graded (row (al, s) carries the Schmidt value lam_al, down
// to 1e-12 of the largest), and the small singular vectors live in the small
// rows, so every row has a scale of its own: theta = W 2^(er[row] + E0), the
// largest entry of a row near 2^54 and kept below 2^55 (fx_rescale_rows).  (One
// scale for the whole matrix loses the digits of components of weight 1e-6, which
// an overlap of 1e-7 still depends on.)  Inner products over rows use a weighted
// copy of the pivot column, Pw = p 2^(2 er + kw); the update of a column needs no
// weights.
//
// thr: squared norm (in units of 2^(2 E0)) at which the remaining columns count
// as zero.  Column j of R^dagger goes to X + j ldx (n entries) with exponent
// xe[j], at full scale; ord (n ints), cn (n floats), er (m ints) and Pw (m
// elements) are scratch.  Returns the rank.
//
// Step j takes the remaining column p of largest norm (FP32 norms, refreshed
// while the columns are updated; near-ties to the smaller position) and y =
// 1 / |p| (fx_rsqrt); for every remaining c: r = <p, c> y, X[j][c] = conj(r),
// c -= p (r y).
//
// Control flow is uniform over the warp and every shuffle takes all 32 lanes:
// shuffles under a partial mask cost a warp barrier each, and a step is bound
// by its chain of latencies, not by issue.
// ---------------------------------------------------------------------------

// Sum over the 2^lg lanes of an aligned group; lgm >= lg uniform over the warp.
template <class T>
__device__ __forceinline__ T fx_group_sum(T v, int lg, int lgm) {
#pragma unroll 1
  for (int o = lgm - 1; o >= 0; --o) {
    const T x = __shfl_xor_sync(0xffffffffu, v, 1 << o);
    if (o < lg) v += x;
  }
  return v;
}

// squared norm of a column of X (n entries at off) by the group's lanes
// (nothing read unless on)
template <bool SH>
__device__ __forceinline__ float fx_norm2f(const FxMem<SH>& X, bool on, int off, int len, int lig, int lg, int lgm) {
  float q = 0.0f;
  if (on)
#pragma unroll 1
    for (int i = lig; i < len; i += 1 << lg) q += fx_cabs2f(X.ld(off + i));
  return fx_group_sum(q, lg, lgm);
}

// The exponent of row i (|entries| < 2^x) and then the row as integers.
__device__ __forceinline__ int fx_row_exponent(const double2* T, int n, int i, bool on, int lig, int lg, int lgm) {
  int mx = 0;
  if (on)
#pragma unroll 1
    for (int c = lig; c < n; c += 1 << lg) {
      const double2 v = T[i * n + c];
      mx = max(mx, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
    }
#pragma unroll 1
  for (int o = lgm - 1; o >= 0; --o) {
    const int x = __shfl_xor_sync(0xffffffffu, mx, 1 << o);
    if (o < lg) mx = max(mx, x);
  }
  return (mx >> 20) - 1022;
}

// Weighted squared norm of column c of W.
template <bool SH>
__device__ __forceinline__ float fx_column_norm(const FxMem<SH>& W, int m, int n, int c, const int* er, bool on,
                                                int lig, int lg, int lgm) {
  float q = 0.0f;
  if (on)
#pragma unroll 1
    for (int i = lig; i < m; i += 1 << lg) q = fmaf(fx_cabs2f(W.ld(i * n + c)), fx_pow2f(2 * er[i]), q);
  return fx_group_sum(q, lg, lgm);
}

// The pivot of step j by lw lanes of a warp: the position of the largest
// remaining column (keyed by its norm, the low 7 bits of which give way to
// the position).
__device__ __forceinline__ unsigned fx_pivot_key(const float* cn, const int* ord, int j, int n, bool on, int ll,
                                                 int lw) {
  unsigned key = 0;
  if (on)
#pragma unroll 1
    for (int u = j + ll; u < n; u += lw) {
      const unsigned v = ((unsigned)__float_as_int(cn[ord[u]]) & ~127u) | (unsigned)(127 - u);
      key = v > key ? v : key;
    }
#pragma unroll 1
  for (int o = lw >> 1; o > 0; o >>= 1) {
    const unsigned v = __shfl_xor_sync(0xffffffffu, key, o);
    key = v > key ? v : key;
  }
  return key;
}

// Pivot column p by lw lanes: its squared norm 2^-56 at full scale (entries
// p 2^(er + k)), and the weighted copy Pw = p 2^(2 er + kw).  pn: the squared norm
// in FP32.
template <bool SH>
__device__ __forceinline__ long long fx_pivot(const FxMem<SH>& W, int4* Pw, int m, int n, int p, float pn, int k,
                                              const int* er, bool on, int ll, int lw, int& kw) {
  FxSquares nn{0, 0, 0};
  int top = -1000;
  if (on)
#pragma unroll 1
    for (int i = ll; i < m; i += lw) {
      const int4 a = W.ld(i * n + p);
      const int e = er[i];
      const int4 f = fx_shift_any(a, e + k);
      fx_square(nn, fx_re(f));
      fx_square(nn, fx_im(f));
      const float q = fx_cabs2f(a);
      if (q > 0.0f) top = max(top, fx_ilog2f(q) + 4 * e);
    }
  long long N = fx_sum(nn);
#pragma unroll 1
  for (int o = lw >> 1; o > 0; o >>= 1) {
    N += __shfl_xor_sync(0xffffffffu, N, o);
    top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  }
  kw = fx_pivot_weight(top, pn);
  if (on)
#pragma unroll 1
    for (int i = ll; i < m; i += lw) Pw[i] = fx_shift_any(W.ld(i * n + p), 2 * er[i] + kw);
  return N;
}

// Column c of step j (pivot p, y = 1 / |p|, inner products shifted by sh, kx = 2 k -
// kw - sh) by its group of lanes;
// the high limbs that it leaves are ORed into high.
template <bool SH>
__device__ __forceinline__ void fx_qr_column(const FxMem<SH>& W, const FxMem<SH>& X, const int4* Pw, int m, int n,
                                             int p, int c, int xoff, Fx y, int sh, int kx, const int* er, bool mine, int lig,
                                             int lg, int lgm, float* cn, int& high) {
  FxAcc re{0, 0}, im{0, 0};
  if (mine)
#pragma unroll 1
    for (int i = lig; i < m; i += 1 << lg) fx_cmacc(re, im, Pw[i], W.ld(i * n + c));
  const long long dr = fx_group_sum(fx_sum_shifted(re, sh), lg, lgm);
  const long long di = fx_group_sum(fx_sum_shifted(im, sh), lg, lgm);
  const int4 r = fx_shift_any(fx_pack(fx_mul(fx_split(dr), y), fx_mul(fx_split(di), y)), kx);
  if (mine && lig == 0) X.st(xoff + c, make_int4(r.x, r.y, -r.z, -r.w));
  const int4 s = fx_pack(-fx_mul(fx_re(r), y), -fx_mul(fx_im(r), y));
  float q = 0.0f;
  if (mine)
#pragma unroll 1
    for (int i = lig; i < m; i += 1 << lg) {
      const int4 a = W.ld(i * n + c);
      FxAcc ur{0, 0}, ui{0, 0};
      fx_cmac(ur, ui, s, W.ld(i * n + p));
      const int4 b = fx_pack(fx_val(fx_re(a)) + fx_sum(ur), fx_val(fx_im(a)) + fx_sum(ui));
      W.st(i * n + c, b);
      high |= fx_high_bits(b.x) | fx_high_bits(b.z);
      q = fmaf(fx_cabs2f(b), fx_pow2f(2 * er[i]), q);
    }
  q = fx_group_sum(q, lg, lgm);
  if (mine && lig == 0) cn[c] = q;
}

// Rows whose entries have passed 2^55 in the columns from position u0 on are taken
// down, with their exponents, by lw lanes.  Rows of small weight grow when the
// pivots, chosen by the large rows, are nearly parallel in the small ones: by up
// to 50 in 64 x 64 thetas of states whose Schmidt values spread over decades, by 128
// in a Hadamard matrix with one small row; two limbs hold 32.
template <bool SH>
__device__ __noinline__ void fx_rescale_rows(FxMem<SH> W, int m, int n, int u0, const int* ord, int* er, bool on, int ll,
                                             int lw) {
  if (on)
#pragma unroll 1
    for (int i = ll; i < m; i += lw) {
      int high = 0;
#pragma unroll 1
      for (int u = u0; u < n; ++u) {
        const int4 a = W.ld(i * n + ord[u]);
        high |= fx_high_bits(a.x) | fx_high_bits(a.z);
      }
      const int k = fx_row_shift(high);
      if (k > 0) {
#pragma unroll 1
        for (int u = u0; u < n; ++u) W.st(i * n + ord[u], fx_shift(W.ld(i * n + ord[u]), -k));
        er[i] += k;
      }
    }
}

static __device__ __noinline__ int fx_qr(double2* T, int4* Pw, int m, int n, double fro, int4* Xp, int ldx, int* xe,
                                         int* ord, float* cn, int* er, int lane, int lw) {
  const FxMem<true> W(reinterpret_cast<int4*>(T)), X(Xp);
  const int ll = lane & (lw - 1);
  const unsigned hmask = lw == 32 ? 0xffffffffu : (0xffffu << (lane & 16));
  int xmax = -2000;
  {
    const int lg = fx_lanes(m, lw), gi = ll >> lg, lig = ll & ((1 << lg) - 1), groups = lw >> lg;
    const int iters = fx_umax((m + groups - 1) / groups), lgm = fx_umax(lg);
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
      const int i = gi + it * groups;
      const int x = fx_row_exponent(T, n, i, i < m, lig, lg, lgm);
      if (i < m) {
        xmax = max(xmax, x);
#pragma unroll 1
        for (int c = lig; c < n; c += 1 << lg) W.st(i * n + c, fx_from_double2(T[i * n + c], 54 - x));
        if (lig == 0) er[i] = x;
      }
    }
  }
#pragma unroll 1
  for (int o = lw >> 1; o > 0; o >>= 1) xmax = max(xmax, __shfl_xor_sync(0xffffffffu, xmax, o));
  __syncwarp();
#pragma unroll 1
  for (int i = ll; i < m; i += lw) er[i] = max(er[i] - xmax, -200);
  __syncwarp();
  const int E0 = xmax - 54;
  const float thr = fx_zero_norm2(fro, E0);
  {
    const int lg = fx_lanes(n, lw), gi = ll >> lg, lig = ll & ((1 << lg) - 1), groups = lw >> lg;
    const int iters = fx_umax((n + groups - 1) / groups), lgm = fx_umax(lg);
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
      const int c = gi + it * groups;
      const float q = fx_column_norm(W, m, n, c, er, c < n, lig, lg, lgm);
      if (lig == 0 && c < n) {
        cn[c] = q;
        ord[c] = c;
      }
    }
  }
  __syncwarp();
  const int own = m < n ? m : n;
  const int steps = fx_umax(own);
  int rank = own;
  bool on = true;
#pragma unroll 1
  for (int j = 0; j < steps; ++j) {
    on = on && j < own;
    const unsigned key = fx_pivot_key(cn, ord, j, n, on, ll, lw);
    const float pn = __int_as_float((int)(key & ~127u));
    if (on && !(pn > thr)) {
      rank = j;
      on = false;
    }
    if (!__any_sync(0xffffffffu, on)) break;
    const int up = on ? 127 - (int)(key & 127u) : 0;
    const int p = on ? ord[up] : 0, k = on ? fx_pivot_shift(pn) : 0;
    int kw;
    const long long N = fx_pivot(W, Pw, m, n, p, pn, k, er, on, ll, lw, kw);
    if (on && ll == 0) {   // every lane has read ord[up] (the shuffles above)
      ord[up] = ord[j];
      ord[j] = p;
      xe[j] = E0 - k;
    }
    __syncwarp();
    const Fx y = fx_split(fx_rsqrt(on ? N : 1ll << 55));
    if (on) {
      if (ll == 0) X.st(j * ldx + p, fx_pack(fx_mul(fx_split(N), y), 0));
#pragma unroll 1
      for (int u = ll; u < j; u += lw) X.st(j * ldx + ord[u], make_int4(0, 0, 0, 0));
    }
    const int sh = on ? fx_dot_shift(kw, pn) : 0, kx = 2 * k - kw - sh;
    const int na = on ? n - j - 1 : 0;
    const int lg = fx_lanes(na, lw), gi = ll >> lg, lig = ll & ((1 << lg) - 1), groups = lw >> lg;
    const int iters = fx_umax((na + groups - 1) / groups), lgm = fx_umax(lg);
    int high = 0;
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
      const int u = j + 1 + gi + it * groups;
      const bool mine = on && u < n;
      fx_qr_column(W, X, Pw, m, n, p, mine ? ord[u] : 0, j * ldx, y, sh, kx, er, mine, lig, lg, lgm, cn, high);
    }
    __syncwarp();
    const unsigned grown = __ballot_sync(0xffffffffu, high >= (1 << 27));
    if (grown != 0u) {
      fx_rescale_rows(W, m, n, j + 1, ord, er, on && (grown & hmask) != 0u, ll, lw);
      __syncwarp();
    }
  }
  return rank;
}

// The same by every thread of a CTA.  The first warp finds and scales the
// pivot; a column gets 2^lg lanes by its step's count, as for 256 threads
// whatever the CTA's size, so that results do not depend on it.
constexpr int kCtaLanes = 256;
__device__ __forceinline__ int fx_cta_lanes(int units) {
  const int lg = 31 - __clz(kCtaLanes / (units < 1 ? 1 : units > kCtaLanes ? kCtaLanes : units));
  return lg > 5 ? 5 : lg;
}
struct FxQrShared {
  int p, sh, kx, xmax;
  long long y, N;
};

template <bool SH>
__device__ __noinline__ int fx_qr_cta(double2* T, int4* Pw, int m, int n, double fro, int4* Xp, int ldx, int* xe,
                                      int* ord, float* cn, int* er, FxQrShared* sh) {
  const FxMem<SH> W(reinterpret_cast<int4*>(T)), X(Xp);
  const int ti = threadIdx.x, nt = blockDim.x;
  {
    const int lg = fx_cta_lanes(m), gi = ti >> lg, lig = ti & ((1 << lg) - 1), groups = nt >> lg;
#pragma unroll 1
    for (int i0 = 0; i0 < m; i0 += groups) {
      const int i = i0 + gi;
      const int x = fx_row_exponent(T, n, i, i < m, lig, lg, lg);
      if (i < m) {
#pragma unroll 1
        for (int c = lig; c < n; c += 1 << lg) W.st(i * n + c, fx_from_double2(T[i * n + c], 54 - x));
        if (lig == 0) er[i] = x;
      }
    }
  }
  __syncthreads();
  if (ti < 32) {
    int xmax = -2000;
#pragma unroll 1
    for (int i = ti; i < m; i += 32) xmax = max(xmax, er[i]);
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) xmax = max(xmax, __shfl_xor_sync(0xffffffffu, xmax, o));
#pragma unroll 1
    for (int i = ti; i < m; i += 32) er[i] = max(er[i] - xmax, -200);
    if (ti == 0) sh->xmax = xmax;
  }
  __syncthreads();
  const int E0 = sh->xmax - 54;
  const float thr = fx_zero_norm2(fro, E0);
  {
    const int lg = fx_cta_lanes(n), gi = ti >> lg, lig = ti & ((1 << lg) - 1), groups = nt >> lg;
#pragma unroll 1
    for (int c0 = 0; c0 < n; c0 += groups) {
      const int c = c0 + gi;
      const float q = fx_column_norm(W, m, n, c, er, c < n, lig, lg, lg);
      if (lig == 0 && c < n) {
        cn[c] = q;
        ord[c] = c;
      }
    }
  }
  __syncthreads();
  const int own = m < n ? m : n;
#pragma unroll 1
  for (int j = 0; j < own; ++j) {
    if (ti < 32) {
      const unsigned key = fx_pivot_key(cn, ord, j, n, true, ti, 32);
      const float pn = __int_as_float((int)(key & ~127u));
      const bool on = pn > thr;
      const int up = 127 - (int)(key & 127u);
      const int p = on ? ord[up] : -1, k = on ? fx_pivot_shift(pn) : 0;
      int kw;
      const long long N = fx_pivot(W, Pw, m, n, p, pn, k, er, on, ti, 32, kw);
      if (ti == 0) {
        if (on) {
          ord[up] = ord[j];
          ord[j] = p;
          xe[j] = E0 - k;
          sh->sh = fx_dot_shift(kw, pn);
          sh->kx = 2 * k - kw - sh->sh;
          sh->N = N;
          sh->y = fx_rsqrt(N);
        }
        sh->p = p;
      }
    }
    __syncthreads();
    const int p = sh->p;
    if (p < 0) {
      __syncthreads();   // sh is read before the caller (or a later call) writes it again
      return j;
    }
    const Fx y = fx_split(sh->y);
    const int ds = sh->sh, kx = sh->kx;
    if (ti == 0) X.st(j * ldx + p, fx_pack(fx_mul(fx_split(sh->N), y), 0));
#pragma unroll 1
    for (int u = ti; u < j; u += nt) X.st(j * ldx + ord[u], make_int4(0, 0, 0, 0));
    const int na = n - j - 1;
    const int lg = fx_cta_lanes(na), gi = ti >> lg, lig = ti & ((1 << lg) - 1), groups = nt >> lg;
    int high = 0;
#pragma unroll 1
    for (int u0 = j + 1; u0 < n; u0 += groups) {
      const int u = u0 + gi;
      const bool mine = u < n;
      fx_qr_column(W, X, Pw, m, n, p, mine ? ord[u] : 0, j * ldx, y, ds, kx, er, mine, lig, lg, lg, cn, high);
    }
    if (__syncthreads_or(high >= (1 << 27))) {
      fx_rescale_rows(W, m, n, j + 1, ord, er, true, ti, nt);
      __syncthreads();
    }
  }
  return own;
}

// ---------------------------------------------------------------------------
// One-sided Jacobi on the m columns (n rows each, column j at X + j ldx, real
// values X 2^xe[j]) in place; ex[j] receives the exponent of column j.  Returns
// the number of sweeps, or -kMaxSweeps.
//
// A round-robin (circle) ordering rotates floor(m / 2) disjoint pairs a round
// (an odd m is padded with a zero column, whose pair is skipped).  The inner
// products and both norms of a pair are formed in every round (the integer
// products are cheap, carried norms would need FP64), the angle in FP32
// (fx_rotation).  The last sweep is one whose rotations all had |cos| max(|cos|,
// sin) <= 1e-16, with |cos| between the pair's columns and sin of the angle:
// what a rotation puts back into the pairs before it in the sweep is that
// product, and what the FP32 angle leaves of its own pair is 1e-7 |cos|.
// ---------------------------------------------------------------------------

// Column c to full scale (norm in [2^55, 2^56)).
template <bool SH>
__device__ __forceinline__ void fx_scale_column(const FxMem<SH>& X, int ldx, int n, int c, bool on, const int* xe, int* ex,
                                                int lig, int lg, int lgm) {
  const float q = fx_norm2f(X, on, c * ldx, n, lig, lg, lgm);
  const int k = q > 0.0f ? (111 - fx_ilog2f(q)) >> 1 : 0;
  if (on) {
    if (k != 0)
#pragma unroll 1
      for (int i = lig; i < n; i += 1 << lg) X.st(c * ldx + i, fx_shift(X.ld(c * ldx + i), k));
    if (lig == 0) ex[c] = xe[c] - k;
  }
}

// Columns of pair q in round r of the circle ordering of mp (even) columns.
__device__ __forceinline__ void fx_circle(int m1, int r, int q, int& i, int& j) {
  i = r + q;
  j = r - q;
  if (i >= m1) i -= m1;
  if (j < 0) j += m1;
  if (q == 0) {
    i = r;
    j = m1;
  }
}

// |cos|^2 between two columns below which they count as orthogonal: 4 units of
// FP64 rounding (the integer inner products resolve a quarter of one)
constexpr float kFxTol2 = 1e-30f;

// Pair (i, j) by its group of lanes; called by whole warps.
template <bool SH>
__device__ __forceinline__ void fx_pair(const FxMem<SH>& X, int ldx, int n, int i, int j, bool on, int* ex,
                                        int lig, int lg, int lgm, int& rotated, int& large) {
  const int oa = i * ldx, ob = j * ldx, nr = on ? n : 0;
  FxAcc sa{0, 0}, sb{0, 0}, re{0, 0}, im{0, 0};
#pragma unroll 1
  for (int row = lig; row < nr; row += 1 << lg) {
    const int4 x = X.ld(oa + row), y = X.ld(ob + row);
    fx_cabs2(sa, x);
    fx_cabs2(sb, y);
    fx_cmacc(re, im, x, y);
  }
  const int ei = ex[i], ej = ex[j];
  long long aa = fx_sum2(sa), bb = fx_sum2(sb), abr = fx_sum(re), abi = fx_sum(im);
#pragma unroll 1
  for (int o = lgm - 1; o >= 0; --o) {
    const long long x0 = __shfl_xor_sync(0xffffffffu, aa, 1 << o), x1 = __shfl_xor_sync(0xffffffffu, bb, 1 << o);
    const long long x2 = __shfl_xor_sync(0xffffffffu, abr, 1 << o), x3 = __shfl_xor_sync(0xffffffffu, abi, 1 << o);
    if (o < lg) {
      aa += x0;
      bb += x1;
      abr += x2;
      abi += x3;
    }
  }
  constexpr float k40 = 9.094947017729282e-13f;   // 2^-40
  const float af = fx_to_float(aa) * k40, bf = fx_to_float(bb) * k40;
  const float xr = fx_to_float(abr) * k40, xi = fx_to_float(abi) * k40;
  const float ab2 = fmaf(xr, xr, xi * xi), pab = af * bf;
  if (on && ab2 > kFxTol2 * pab) {
    FxRot R;
    fx_rotation(aa, bb, abr, abi, ej - ei, af, bf, xr, xi, ab2, R);
    rotated = 1;
    large |= (ab2 * fmaxf(ab2, R.s2 * pab) > 1e-32f * pab * pab) ? 1 : 0;
    const Fx n2x = fx_neg(R.s2x), n2y = fx_neg(R.s2y), n3y = fx_neg(R.s3y);
#pragma unroll 1
    for (int row = lig; row < n; row += 1 << lg) {
      const int4 x = X.ld(oa + row), y = X.ld(ob + row);
      const Fx ar = fx_re(x), ai = fx_im(x), br = fx_re(y), bi = fx_im(y);
      FxAcc t0{0, 0}, t1{0, 0}, t2{0, 0}, t3{0, 0};
      fx_mac(t0, R.c, ar);
      fx_mac(t1, R.c, ai);
      fx_mac(t2, R.c, br);
      fx_mac(t3, R.c, bi);
      fx_mac(t0, n2x, br);
      fx_mac(t1, n2x, bi);
      fx_mac(t2, R.s3x, ar);
      fx_mac(t3, R.s3x, ai);
      fx_mac(t0, n2y, bi);
      fx_mac(t1, R.s2y, br);
      fx_mac(t2, n3y, ai);
      fx_mac(t3, R.s3y, ar);
      X.st(oa + row, fx_pack(fx_sum(t0), fx_sum(t1)));
      X.st(ob + row, fx_pack(fx_sum(t2), fx_sum(t3)));
    }
    if ((R.ka | R.kb) != 0) {   // rare
#pragma unroll 1
      for (int row = lig; row < n; row += 1 << lg) {
        X.st(oa + row, fx_shift(X.ld(oa + row), R.ka));
        X.st(ob + row, fx_shift(X.ld(ob + row), R.kb));
      }
      if (lig == 0) {   // every lane of the group has read the exponents (the shuffles above)
        ex[i] = ei - R.ka;
        ex[j] = ej - R.kb;
      }
    }
  }
}


static __device__ __noinline__ int fx_jacobi(int4* Xp, int ldx, int n, int m, const int* xe, int* ex, int lane, int lw) {
  const FxMem<true> X(Xp);
  const int hb = lane & ~(lw - 1), ll = lane & (lw - 1);
  const unsigned hmask = lw == 32 ? 0xffffffffu : (0xffffu << hb);
  {
    const int lg = fx_lanes(m, lw), gi = ll >> lg, lig = ll & ((1 << lg) - 1), groups = lw >> lg;
    const int iters = fx_umax((m + groups - 1) / groups), lgm = fx_umax(lg);
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
      const int c = gi + it * groups;
      fx_scale_column(X, ldx, n, c, c < m, xe, ex, lig, lg, lgm);
    }
  }
  __syncwarp();
  const int m1 = m + (m & 1) - 1, P = (m1 + 1) >> 1, q0 = m & 1, Pe = P - q0;
  const bool trivial = (m < 1 || n < 1 || Pe < 1);
  const int lg = fx_lanes(trivial ? lw : Pe, lw), gi = ll >> lg, lig = ll & ((1 << lg) - 1), groups = lw >> lg;
  const int iters = fx_umax(trivial ? 0 : (Pe + groups - 1) / groups), lgm = fx_umax(lg);
  const int rounds = fx_umax(trivial ? 0 : m1);
  bool active = !trivial;
  int result = trivial ? ((m < 1 || n < 1) ? 0 : 1) : -kMaxSweeps;
  for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
    if (!__any_sync(0xffffffffu, active)) break;
    int rotated = 0, large = 0;
#pragma unroll 1
    for (int r = 0; r < rounds; ++r) {
#pragma unroll 1
      for (int it = 0; it < iters; ++it) {
        const int q = q0 + gi + it * groups;
        const bool on = active && r < m1 && q < P;
        int i = 0, j = 0;
        if (on) fx_circle(m1, r, q, i, j);
        fx_pair(X, ldx, n, i, j, on, ex, lig, lg, lgm, rotated, large);
      }
      __syncwarp();
    }
    const unsigned rt = __ballot_sync(0xffffffffu, rotated) & hmask;
    const unsigned big = __ballot_sync(0xffffffffu, large) & hmask;
    if (active && (rt == 0u || big == 0u)) {
      active = false;
      result = sweep + 1;
    }
  }
  return result;
}

// The same by every thread of a CTA (lane groups as in fx_qr_cta).
template <bool SH>
__device__ __noinline__ int fx_jacobi_cta(int4* Xp, int ldx, int n, int m, const int* xe, int* ex) {
  const FxMem<SH> X(Xp);
  const int ti = threadIdx.x, nt = blockDim.x;
  {
    const int lg = fx_cta_lanes(m), gi = ti >> lg, lig = ti & ((1 << lg) - 1), groups = nt >> lg;
#pragma unroll 1
    for (int c0 = 0; c0 < m; c0 += groups) fx_scale_column(X, ldx, n, c0 + gi, c0 + gi < m, xe, ex, lig, lg, lg);
  }
  __syncthreads();
  const int m1 = m + (m & 1) - 1, P = (m1 + 1) >> 1, q0 = m & 1, Pe = P - q0;
  if (m < 1 || n < 1) return 0;
  if (Pe < 1) return 1;
  const int lg = fx_cta_lanes(Pe), gi = ti >> lg, lig = ti & ((1 << lg) - 1), groups = nt >> lg;
  for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
    int rotated = 0, large = 0;
#pragma unroll 1
    for (int r = 0; r < m1; ++r) {
#pragma unroll 1
      for (int q1 = q0; q1 < P; q1 += groups) {
        const int q = q1 + gi;
        const bool on = q < P;
        int i = 0, j = 0;
        if (on) fx_circle(m1, r, q, i, j);
        fx_pair(X, ldx, n, i, j, on, ex, lig, lg, lg, rotated, large);
      }
      __syncthreads();
    }
    const int rt = __syncthreads_or(rotated), big = __syncthreads_or(large);
    if (!rt || !big) return sweep + 1;
  }
  return -kMaxSweeps;
}

}  // namespace tnrc
