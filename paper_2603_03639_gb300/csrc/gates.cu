// Layer gate table of the truncated TEBD layers, and the noise realisations.
//
// layer_gate_kernel: eight lanes per (sample s, truncated layer l, bond b of
// that layer).  The layer's gate on bond b is a product of factors
// exp(-i tau h_f) (time order f = 1..F), each h_f Hermitian and linear in the
// controls it contains:
//   second order  (A(dts/2) B(dts) A(dts/2) per Trotter step, dts = dt/n_sub):
//     one factor h_b = c ZZ + J^x XX + J^y YY + wL (x_b X + y_b Y) (x) I
//                      + wR I (x) (x_{b+1} X + y_{b+1} Y)          (Eq. sysH, Eq. Hp)
//     with tau = dts (odd bonds) or dts/2 (even bonds), or two such half-step
//     factors where a step boundary merges them;
//   first order   (Eq. circuit): the interaction c ZZ + J^x XX + J^y YY with
//     tau = dts, followed on the bond that carries them by the single-site
//     rotations y Y then x X of its sites;
// c = g_b (if a control) + gfix_{k,b} + J^z(s)_b.  Each factor is diagonalised
// by cyclic complex Jacobi rotations (FP64); the gate is the product and, for
// every control u, Q_u = sum_f L_f (dG_f/du) G_f^dag L_f^dag (L_f the factors
// after f) with dG_f/du by the Daleckii-Krein formula
//   dG = V (Gam o (V^dag P V)) V^dag,  Gam_jk = -i tau e^{-i tau (l_j + l_k)/2} sinc(tau (l_j - l_k)/2),
// P = dh_f/du.  The trajectory kernel then needs only tr(Q_u rho) per control.
//
// noise_kernel: J^(s)_b from the counter-based SplitMix64 generator (Steele,
// Lea, Flood 2014): out(i) = mix(seed + (i+1) * 0x9E3779B97F4A7C15).
#include "tnrc_device.cuh"

namespace tnrc {

// Eight lanes work on one record: two factors (later: two controls) at a time,
// each by four lanes, lane r holding row r of its 4 x 4 matrices.  One thread
// per record was a chain of FP64 instructions of 0.9 ms (64 cycles each, square
// roots and divisions 600) whatever the number of records, half of a small
// evaluation: the smallest call went from 1.63 to 1.05 ms.  The FP64
// instructions per record stay about the same (the lanes share them).
constexpr int kRecLanes = 8;
constexpr int kGateThreads = 64;
constexpr int kMaxFactors = 5;

__device__ __forceinline__ double2 shfl4(double2 v, int src) {   // from lane src of the group of four
  return make_double2(__shfl_sync(0xffffffffu, v.x, src, 4), __shfl_sync(0xffffffffu, v.y, src, 4));
}

// 1 / sqrt(x) for x of normal FP32 size: the FP32 estimate (2e-7) and one
// third-order step, seven FP64 instructions in the place of thirty.
__device__ __forceinline__ double rsqrt_of(double x) {
  const double y = (double)rsqrtf((float)x);
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}

// Cyclic Jacobi of the Hermitian 4 x 4 matrix whose row r is h: on return the
// diagonal holds the eigenvalues and v is row r of V, h = V diag V^dagger.  A
// round rotates two disjoint pairs (p, q), U = [[c, s], [-conj(s), c]].  (Angles
// from FP32, as in svd_fx.cuh, take a sweep more here: one fidelity of six
// qubits 636 us against 619, 8 qubits with gradient 3.93 ms against 3.84, and
// errors the same or a little larger.)  Returns false if it did not converge.
__device__ bool herm_eig4_rows(double2 (&h)[4], double2 (&v)[4], int r) {
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] = make_double2(c == r ? 1.0 : 0.0, 0.0);
  double sc = 0.0;
#pragma unroll
  for (int c = 0; c < 4; ++c) sc += cabs2(h[c]);
  sc += __shfl_xor_sync(0xffffffffu, sc, 1, 4);
  sc += __shfl_xor_sync(0xffffffffu, sc, 2, 4);
  // 2^-e with 2^(2e) about sc: angles from entries of order one
  const int e2 = (__double2hiint(sc) >> 20) & 2047;
  const double inv = __hiloint2double((1023 - ((e2 - 1023) >> 1)) << 20, 0);
  bool ok = false;
#pragma unroll 1
  for (int sweep = 0; sweep < 30; ++sweep) {
    double off = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c != r) off += cabs2(h[c]);
    off += __shfl_xor_sync(0xffffffffu, off, 1, 4);
    off += __shfl_xor_sync(0xffffffffu, off, 2, 4);
    ok = off <= 2e-32 * sc;
    if (__all_sync(0xffffffffu, ok)) break;
#pragma unroll
    for (int rd = 0; rd < 3; ++rd) {
      // partner of index i in round rd: i ^ 1, i ^ 2, i ^ 3
      const int mate = r ^ (rd + 1);
      const bool low = r < mate;
      // z = h[p][q] (p < q), d = h[q][q] - h[p][p], the same in both lanes of a pair
      double2 hm = h[0], hd = h[0];
#pragma unroll
      for (int c = 1; c < 4; ++c) {
        if (c == mate) hm = h[c];
        if (c == r) hd = h[c];
      }
      if (r == 0) hd = h[0];
      const double other = __shfl_sync(0xffffffffu, hd.x, mate, 4);
      const double2 z = shfl4(hm, low ? r : mate);
      const double zx = z.x * inv, zy = z.y * inv, d = (low ? other - hd.x : hd.x - other) * inv;
      const double z2 = fma(zx, zx, zy * zy);
      // with w = 1 / sqrt(d^2 + 4 |z|^2): cos 2theta = |d| w, c = sqrt((1 + cos
      // 2theta) / 2), s = sign(d) w / c z
      double c = 1.0;
      double2 s = make_double2(0.0, 0.0);
      if (z2 > 1e-35) {
        const double w = rsqrt_of(fma(d, d, 4.0 * z2));
        const double hq = fma(0.5, fabs(d) * w, 0.5);
        const double rc = rsqrt_of(hq);
        c = hq * rc;
        const double f = copysign(w * rc, d);
        s = make_double2(f * zx, f * zy);
      }
      // columns of both pairs: (p, q) <- (c p - conj(s) q, s p + c q)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int p0 = rd == 0 ? 2 * k : k, q0 = p0 ^ (rd + 1);
        const int a = p0 < q0 ? p0 : q0, b2 = p0 < q0 ? q0 : p0;
        const double ck = __shfl_sync(0xffffffffu, c, a, 4);
        const double2 sk = shfl4(s, a);
        const double2 hp = h[a], hq = h[b2], vp = v[a], vq = v[b2];
        double2 np = cscale(hp, ck), nq = cscale(hq, ck), wp = cscale(vp, ck), wq = cscale(vq, ck);
        cfmac(np, make_double2(-sk.x, -sk.y), hq);
        cfma(nq, sk, hp);
        cfmac(wp, make_double2(-sk.x, -sk.y), vq);
        cfma(wq, sk, vp);
        h[a] = np;
        h[b2] = nq;
        v[a] = wp;
        v[b2] = wq;
      }
      // rows: p <- c p - s q, q <- conj(s) p + c q
      const double2 sr = low ? make_double2(-s.x, -s.y) : cconj(s);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const double2 o = shfl4(h[k], mate);
        double2 nh = cscale(h[k], c);
        cfma(nh, sr, o);
        h[k] = nh;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k == mate) h[k] = make_double2(0.0, 0.0);
    }
  }
  return ok;
}

// sin(x) / x, with sn = sin x known to about 1e-16
__device__ __forceinline__ double sinc_of(double x, double sn) {
  const double x2 = x * x;
  if (x2 < 0.25) {   // Taylor series to x^14: the next term is below 1e-18
    double p = -1.0 / 1307674368000.0;
    p = fma(p, x2, 1.0 / 6227020800.0);
    p = fma(p, x2, -1.0 / 39916800.0);
    p = fma(p, x2, 1.0 / 362880.0);
    p = fma(p, x2, -1.0 / 5040.0);
    p = fma(p, x2, 1.0 / 120.0);
    p = fma(p, x2, -1.0 / 6.0);
    return fma(p, x2, 1.0);
  }
  return sn / x;
}

// Row i of a generator in the bond basis |s_b s_{b+1}> (index 2 s_b + s_{b+1}),
// scaled by w: one entry, `val` in column `col`.  0: X (x) I, 1: Y (x) I,
// 2: I (x) X, 3: I (x) Y, 4: Z (x) Z.
__device__ __forceinline__ void generator_row(int code, double w, int i, int& col, double2& val) {
  const int bit = code < 2 ? 2 : 1;
  if (code == 4) {
    col = i;
    val = make_double2((i == 0 || i == 3) ? w : -w, 0.0);
  } else {
    col = i ^ bit;
    val = (code & 1) ? make_double2(0.0, (i & bit) ? w : -w) : make_double2(w, 0.0);
  }
}

struct LayerGateArgs {
  int N, K, C, M, terms, order, nsub, L, R, first_parity;
  double dt;
  const double* u;            // [K][C][N]
  const unsigned char* mask;  // [C][N]
  const double* gfix;         // [K][N-1] or null
  const double* J;            // [M][N-1][terms]: (J^z) or (J^x, J^y, J^z)
  const int* layer_off;       // [L + 1]
  LayerGate* out;             // [M][R]
  int* status;
};

// factor kinds
constexpr int kFBond = 0, kFInter = 1, kFXl = 2, kFYl = 3, kFXr = 4, kFYr = 5;

struct GateShared {                     // one record
  double2 V[kMaxFactors][16], G[kMaxFactors][16], GE[kMaxFactors][16];
  double2 T[2][16], Lt[16];
};

__global__ void __launch_bounds__(kGateThreads) layer_gate_kernel(LayerGateArgs a) {
  __shared__ GateShared sh[kGateThreads / kRecLanes];
  const int lane8 = threadIdx.x & (kRecLanes - 1), half = lane8 >> 2, r = lane8 & 3;
  GateShared& S = sh[threadIdx.x / kRecLanes];
  const long long total = (long long)a.M * a.R;
  const long long idx0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kRecLanes;
  const bool live = idx0 < total;
  const long long idx = live ? idx0 : total - 1;   // idle groups repeat the last record and write nothing
  const int s = (int)(idx / a.R);
  const int rec = (int)(idx - (long long)s * a.R);
  int lo = 0, hi = a.L;  // largest l with layer_off[l] <= rec
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (a.layer_off[mid] <= rec) lo = mid; else hi = mid;
  }
  const int l = lo;
  const int parity = (l + a.first_parity) & 1;
  const int b = parity + 2 * (rec - a.layer_off[l]);
  const int N = a.N, nb = N - 1;
  const int St = a.K * a.nsub;
  const double dts = a.dt / a.nsub;

  // the layer's factors on bond b, first in time first: kind, bin and duration of factor f
  int nf, kind0 = kFBond, k0, k1;
  double tau;
  if (a.order == 2) {
    nf = 1;
    if (l & 1) {
      k0 = k1 = ((l - 1) >> 1) / a.nsub;
      tau = dts;
    } else {
      const int st = (l >> 1) - 1;   // the half steps of steps st and st + 1, merged
      tau = 0.5 * dts;
      k0 = (l == 0 ? 0 : st) / a.nsub;
      k1 = (l == 2 * St ? St - 1 : st + 1) / a.nsub;
      if (l != 0 && l != 2 * St) nf = 2;
    }
  } else {
    k0 = k1 = (l >> 1) / a.nsub;
    tau = dts;
    kind0 = kFInter;
    // even bonds: both sites' rotations, Y before X; else the last site of an odd chain
    nf = (l & 1) ? 5 : ((N & 1) && b == N - 2) ? 3 : 1;
  }
  auto fkind = [&](int f) {
    if (a.order == 2 || f == 0) return kind0;
    if (nf == 3) return f == 1 ? kFYr : kFXr;
    return f == 1 ? kFYl : f == 2 ? kFYr : f == 3 ? kFXl : kFXr;
  };
  auto fbin = [&](int f) { return f == 0 ? k0 : k1; };

  const double* Jb = a.J + ((size_t)s * nb + b) * a.terms;
  const double jz = Jb[a.terms - 1];
  const double jx = (a.terms == 3) ? Jb[0] : 0.0;
  const double jy = (a.terms == 3) ? Jb[1] : 0.0;
  const double wl = (b == 0) ? 1.0 : 0.5;
  const double wr = (b + 1 == N - 1) ? 1.0 : 0.5;
  const unsigned char* mk = a.mask;

  // eigendecomposition, exponential and divided differences, two factors at a time
  const int nfw = (int)__reduce_max_sync(0xffffffffu, (unsigned)nf);
#pragma unroll 1
  for (int f0 = 0; f0 < nfw; f0 += 2) {
    const bool mine = f0 + half < nf;
    const int f = mine ? f0 + half : 0;
    const int kind = fkind(f), k = fbin(f);
    const double* uk = a.u + (size_t)k * a.C * N;
    const double xl = uk[b] * mk[b], yl = uk[N + b] * mk[N + b];
    const double xr = uk[b + 1] * mk[b + 1], yr = uk[N + b + 1] * mk[N + b + 1];
    double c = jz;
    if (a.C == 3) c += uk[2 * N + b] * mk[2 * N + b];
    if (a.gfix) c += a.gfix[(size_t)k * nb + b];
    double2 h[4], v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = make_double2(0.0, 0.0);
    if (kind == kFBond || kind == kFInter) {
      // J^x XX + J^y YY: <00|.|11> = jx - jy, <01|.|10> = jx + jy; (x X + y Y) on
      // a site couples |0> <-> |1> with <0|.|1> = x - i y
      const bool bond = kind == kFBond;
      const double2 lz = make_double2(bond ? wl * xl : 0.0, bond ? ((r & 2) ? wl * yl : -wl * yl) : 0.0);
      const double2 rz = make_double2(bond ? wr * xr : 0.0, bond ? ((r & 1) ? wr * yr : -wr * yr) : 0.0);
      const double dg = (r == 0 || r == 3) ? c : -c, cr = (r == 0 || r == 3) ? jx - jy : jx + jy;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j == r) h[j] = make_double2(dg, 0.0);
        if (j == (r ^ 3)) h[j] = make_double2(cr, 0.0);
        if (j == (r ^ 2)) h[j] = lz;
        if (j == (r ^ 1)) h[j] = rz;
      }
    } else {
      const int code = kind - kFXl;  // 0 X(x)I, 1 Y(x)I, 2 I(x)X, 3 I(x)Y
      int col;
      double2 val;
      generator_row(code, (code == 0) ? xl : (code == 1) ? yl : (code == 2) ? xr : yr, r, col, val);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j == col) h[j] = val;
    }
    const bool ok = herm_eig4_rows(h, v, r);
    if (live && mine && r == 0 && !ok) atomicOr(a.status, kStatusNoConverge);
    double lam = h[0].x;
#pragma unroll
    for (int j = 1; j < 4; ++j)
      if (j == r) lam = h[j].x;
    double sn, cs;
    sincos(0.5 * tau * lam, &sn, &cs);
    const double2 E = make_double2(-2.0 * sn * sn, -2.0 * sn * cs);   // e^{-i tau lam_r} - 1
    double2 ge[4], vE[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // Gam_rj e^{i tau lam_j} = -i tau e^{-i x} sinc(x), x = tau (lam_r - lam_j) / 2
      const double x = 0.5 * tau * (lam - __shfl_sync(0xffffffffu, lam, j, 4));
      sincos(x, &sn, &cs);
      const double sc = tau * sinc_of(x, sn);
      ge[j] = make_double2(-sc * sn, -sc * cs);
      vE[j] = cmul(v[j], shfl4(E, j));
    }
    if (mine) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        S.V[f][r * 4 + j] = v[j];
        S.GE[f][r * 4 + j] = ge[j];
      }
    }
    __syncwarp();
    if (mine) {
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        // G = 1 + V (E - 1) V^dagger: what V lacks in orthogonality (some 1e-16, the
        // roundings of its rotations) then enters times the angle and not times one
        double2 g = make_double2(0.0, 0.0);
#pragma unroll
        for (int j = 0; j < 4; ++j) cfmac(g, S.V[f][cc * 4 + j], vE[j]);
        if (cc == r) g.x += 1.0;
        S.G[f][r * 4 + cc] = g;
      }
    }
    __syncwarp();
  }

  // walk the factors backwards: Lt = product of the factors after f, row r in lt
  LayerGate& out = a.out[idx];
  double2 lt[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    lt[j] = make_double2(j == r ? 1.0 : 0.0, 0.0);
    if (half == 0) S.Lt[r * 4 + j] = lt[j];
  }
  __syncwarp();
  int nq = 0;
#pragma unroll 1
  for (int f1 = nfw - 1; f1 >= 0; --f1) {
    const bool on = f1 < nf;
    const int f = on ? f1 : 0;
    const int kind = fkind(f), k = fbin(f);
    const bool last = f == nf - 1;   // Lt = 1
    // the controls of this factor, as bits of their generator codes
    unsigned ctl = 0;
    if (on) {
      if (kind == kFBond)
        ctl = (mk[b] ? 1u : 0u) | (mk[N + b] ? 2u : 0u) | (mk[b + 1] ? 4u : 0u) | (mk[N + b + 1] ? 8u : 0u);
      if ((kind == kFBond || kind == kFInter) && a.C == 3 && mk[2 * N + b]) ctl |= 16u;
      if (kind >= kFXl) {
        const int code = kind - kFXl;
        if (mk[(code & 1) * N + b + (code >> 1)]) ctl |= 1u << code;
      }
    }
    const int np = __popc(ctl);
    // both half steps of one bin: their matrices add up in the same records
    const bool again = on && !last && a.order == 2 && k0 == k1;
    const int base = again ? 0 : nq;
    const int npw = (int)__reduce_max_sync(0xffffffffu, (unsigned)np);
    const bool any_lt = __any_sync(0xffffffffu, on && !last);
#pragma unroll 1
    for (int q0 = 0; q0 < npw; q0 += 2) {
      const int q = q0 + half;
      const bool mine = q < np;
      unsigned rest = ctl;
#pragma unroll 1
      for (int i = 0; i < q && mine; ++i) rest &= rest - 1;
      const int code = mine ? __ffs(rest) - 1 : 0;
      const double w = kind != kFBond || code == 4 ? 1.0 : code < 2 ? wl : wr;
      // row r of T = (Gam o (V^dag P V)) e^{i tau Lam}, then of T V^dag
      double2 t[4], u[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) t[j] = make_double2(0.0, 0.0);
#pragma unroll
      for (int m = 0; m < 4; ++m) {   // (V^dag P V)[r][j] = sum_m conj(V[m][r]) P[m][col] V[col][j]
        int col;
        double2 val;
        generator_row(code, w, m, col, val);
        const double2 x = cmulc(val, S.V[f][m * 4 + r]);
#pragma unroll
        for (int j = 0; j < 4; ++j) cfma(t[j], x, S.V[f][col * 4 + j]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) t[j] = cmul(S.GE[f][r * 4 + j], t[j]);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        u[j] = make_double2(0.0, 0.0);
#pragma unroll
        for (int m = 0; m < 4; ++m) cfmac(u[j], S.V[f][j * 4 + m], t[m]);
        S.T[half][r * 4 + j] = u[j];
      }
      __syncwarp();
      // Q_f = V (T V^dag)  (= dG_f G_f^dag)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        t[j] = make_double2(0.0, 0.0);
#pragma unroll
        for (int m = 0; m < 4; ++m) cfma(t[j], S.V[f][r * 4 + m], S.T[half][m * 4 + j]);
      }
      __syncwarp();
      if (any_lt) {   // L Q_f L^dag
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          u[j] = make_double2(0.0, 0.0);
#pragma unroll
          for (int m = 0; m < 4; ++m) cfmac(u[j], S.Lt[j * 4 + m], t[m]);
          S.T[half][r * 4 + j] = u[j];
        }
        __syncwarp();
        if (!last) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            t[j] = make_double2(0.0, 0.0);
#pragma unroll
            for (int m = 0; m < 4; ++m) cfma(t[j], lt[m], S.T[half][m * 4 + j]);
          }
        }
        __syncwarp();
      }
      if (live && mine) {
        const int at = base + q;   // at most 10 distinct controls: kMaxLayerParams
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (again) {
            const double2 o = out.Q[at][r * 4 + j];
            t[j].x += o.x;
            t[j].y += o.y;
          }
          out.Q[at][r * 4 + j] = t[j];
        }
        if (r == 0) {
          const int cidx = code == 4 ? 2 : (code & 1), site = (code == 2 || code == 3) ? b + 1 : b;
          out.slot[at] = (k * a.C + cidx) * N + site;
        }
      }
    }
    if (on && !again) nq += np;
    // Lt <- Lt G_f
    double2 x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[j] = make_double2(0.0, 0.0);
#pragma unroll
      for (int m = 0; m < 4; ++m) cfma(x[j], lt[m], S.G[f][m * 4 + j]);
    }
    __syncwarp();
    if (on) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        lt[j] = x[j];
        if (half == 0) S.Lt[r * 4 + j] = x[j];
      }
    }
    __syncwarp();
  }
  if (live && half == 0) {
#pragma unroll
    for (int j = 0; j < 4; ++j) out.G[r * 4 + j] = lt[j];
    if (r == 0) out.nq = nq;
  }
}

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long seed, unsigned long long i) {
  unsigned long long z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void noise_kernel(unsigned long long seed, int dist, double scale, int M, int nb, double* J) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)M * nb) return;
  const double two53 = 1.0 / 9007199254740992.0;
  if (dist == 0) {
    const double u = (double)(splitmix64(seed, idx) >> 11) * two53;
    J[idx] = scale * (2.0 * u - 1.0);
  } else {
    const double u1 = (double)((splitmix64(seed, 2 * idx) >> 11) + 1ull) * two53;
    const double u2 = (double)(splitmix64(seed, 2 * idx + 1) >> 11) * two53;
    J[idx] = scale * sqrt(-2.0 * log(u1)) * cos(2.0 * 3.141592653589793 * u2);
  }
}

// F = (1/T) sum_t |O_t|^2 ; per_traj[t] = |O_t|^2 ; grad[x] = (1/T) sum_t gsp[t][x]
// (fixed summation order: independent of launch configuration and timing).
__global__ void reduce_fidelity_kernel(const double2* O, int T, double* F, double* per_traj) {
  __shared__ double part[256];
  double s = 0.0;
  for (int t = threadIdx.x; t < T; t += blockDim.x) {
    const double v = cabs2(O[t]);
    if (per_traj) per_traj[t] = v;
    s += v;
  }
  part[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *F = part[0] / (double)T;
}

__global__ void reduce_grad_kernel(const double* gsp, int T, int X, double* grad) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= X) return;
  double s = 0.0;
  for (int t = 0; t < T; ++t) s += gsp[(size_t)t * X + x];
  grad[x] = s / (double)T;
}

}  // namespace tnrc

extern "C" cudaError_t tnrc_launch_layer_gates(int N, int K, int C, int M, int terms, int order, int nsub,
                                               int L, int R, int first_parity, double dt, const double* u,
                                               const unsigned char* mask, const double* gfix, const double* J,
                                               const int* layer_off, tnrc::LayerGate* out, int* status,
                                               cudaStream_t st) {
  tnrc::LayerGateArgs a{N, K, C, M, terms, order, nsub, L, R, first_parity, dt, u, mask, gfix, J, layer_off, out,
                        status};
  const long long total = (long long)M * R * tnrc::kRecLanes;
  const int threads = tnrc::kGateThreads;
  const long long blocks = (total + threads - 1) / threads;
  (void)cudaGetLastError();  // report only this launch below
  tnrc::layer_gate_kernel<<<(unsigned)blocks, threads, 0, st>>>(a);
  return cudaGetLastError();
}

extern "C" cudaError_t tnrc_launch_noise(unsigned long long seed, int dist, double scale, int M, int nb, double* J,
                                         cudaStream_t st) {
  const long long total = (long long)M * nb;
  const int threads = 256;
  (void)cudaGetLastError();  // report only this launch below
  tnrc::noise_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, st>>>(seed, dist, scale, M, nb, J);
  return cudaGetLastError();
}

extern "C" cudaError_t tnrc_launch_reduce(const double2* O, int T, double* F, double* per_traj, const double* gsp,
                                          int X, double* grad, cudaStream_t st) {
  (void)cudaGetLastError();  // report only this launch below
  tnrc::reduce_fidelity_kernel<<<1, 256, 0, st>>>(O, T, F, per_traj);
  if (gsp && grad) tnrc::reduce_grad_kernel<<<(X + 127) / 128, 128, 0, st>>>(gsp, T, X, grad);
  return cudaGetLastError();
}
