// Fixed-point arithmetic of the trajectory kernel: 64-bit integers with a
// common power-of-two scale in the place of FP64 values.
//
// GB300 issues one warp-wide FP64 FMA per sub-partition every 64 cycles and a
// 32 x 32 + 64 bit integer multiply-add (IMAD.WIDE) about every 5 (both measured),
// so a product of two 56-bit numbers as three integer multiply-adds costs a quarter
// of one DFMA.
// A value v (|v| < 2^59) is held as two limbs, v = hi 2^28 + lo with lo in
// [-2^27, 2^27); a complex value is an int4 (re.hi, re.lo, im.hi, im.lo), the
// 16 bytes of a double2.  Products keep hi hi and the two cross terms and drop
// lo lo (up to a quarter of the last place after the shift by 56 bits); what is
// kept is summed exactly in two 64-bit accumulators and rounded once, at its end.
// Vectors are scaled so that their norm is near 2^56: a rounding is 2^-57 of
// the norm, against 2^-53 of each element in FP64.
#pragma once
#ifdef __CUDACC__
#define TNRC_HD __host__ __device__ __forceinline__
#else
#define TNRC_HD inline
#endif

namespace tnrc {

struct Fx {       // one fixed-point number
  int hi, lo;
};

struct FxAcc {    // a sum of products: h 2^56 + x 2^28 in units of the product
  long long h, x;
};

TNRC_HD long long fx_val(Fx a) { return ((long long)a.hi << 28) + a.lo; }

TNRC_HD Fx fx_split(long long v) {
  Fx a;
  a.lo = (int)((unsigned)v << 4) >> 4;
  a.hi = (int)((v + (1ll << 27)) >> 28);
  return a;
}

TNRC_HD Fx fx_neg(Fx a) { return Fx{-a.hi, -a.lo}; }

TNRC_HD void fx_mac(FxAcc& s, Fx a, Fx b) {
  s.h += (long long)a.hi * b.hi;
  s.x += (long long)a.hi * b.lo;
  s.x += (long long)a.lo * b.hi;
}

// the sum / 2^56, rounded
TNRC_HD long long fx_sum(FxAcc s) { return s.h + ((s.x + (1ll << 27)) >> 28); }

// the sum / 2^(56 - sh), rounded, 0 <= sh < 28
TNRC_HD long long fx_sum_shifted(FxAcc s, int sh) { return (s.h << sh) + ((s.x + (1ll << (27 - sh))) >> (28 - sh)); }

// A sum of squares h 2^56 + 2 x 2^28 + l, and itself / 2^56, rounded.  The low parts
// are all positive here: dropped, they would bias a norm by a sixth of a unit of
// 2^-56 an entry.
struct FxSquares {
  long long h, x, l;
};
TNRC_HD void fx_square(FxSquares& s, Fx a) {
  s.h += (long long)a.hi * a.hi;
  s.x += (long long)a.hi * a.lo;
  s.l += (long long)a.lo * a.lo;
}
TNRC_HD long long fx_sum(FxSquares s) { return s.h + ((s.x + (s.l >> 29) + (1ll << 26)) >> 27); }

TNRC_HD long long fx_mul(Fx a, Fx b) {
  FxAcc s{0, 0};
  fx_mac(s, a, b);
  return fx_sum(s);
}

TNRC_HD float fx_bits_float(int b) {
#ifdef __CUDA_ARCH__
  return __int_as_float(b);
#else
  union { int i; float f; } u;
  u.i = b;
  return u.f;
#endif
}
TNRC_HD int fx_float_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_int(f);
#else
  union { int i; float f; } u;
  u.f = f;
  return u.i;
#endif
}

// 2^e as a float, e clamped to the normal range
TNRC_HD float fx_pow2f(int e) {
  e = e < -126 ? -126 : e > 127 ? 127 : e;
  return fx_bits_float((e + 127) << 23);
}

// floor(log2 f) of a positive normal float
TNRC_HD int fx_ilog2f(float f) { return ((fx_float_bits(f) >> 23) & 255) - 127; }

TNRC_HD int fx_rint(float f) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(f);
#else
  return (int)rintf(f);
#endif
}

TNRC_HD float fx_rsqrtf(float f) {
#ifdef __CUDA_ARCH__
  return rsqrtf(f);
#else
  return 1.0f / sqrtf(f);
#endif
}

TNRC_HD float fx_rcpf(float f) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.0f, f);
#else
  return 1.0f / f;
#endif
}

// y (|y| < 8) in units of 2^-56: exact, a float has 24 bits
TNRC_HD Fx fx_from_float(float y) {
  Fx a;
  const float z = y * 268435456.0f;
  a.hi = fx_rint(z);
  a.lo = fx_rint((z - (float)a.hi) * 268435456.0f);
  return a;
}

// A 64-bit integer as a float, from its 32-bit halves: the conversion of a
// 64-bit integer runs on the FP64 pipe (64 cycles a warp).
TNRC_HD float fx_to_float(long long v) {
  const int lo = (int)v, hi = (int)((v + (1ll << 31)) >> 32);
  return (float)hi * 4294967296.0f + (float)lo;
}

// Entries of a Gram-Schmidt row, by the bits of their high limbs: a row is taken
// down by 2^fx_row_shift (to below 2^54) once an entry has passed 2^55.  An update
// c -= p (r y), |r y| <= 1, at most doubles an entry (2.5 times by components), so
// entries stay below 2^57, a quarter of what two limbs hold.
TNRC_HD int fx_high_bits(int hi) { return hi ^ (hi >> 31); }
TNRC_HD int fx_row_shift(int high_bits) {
  int k = 0;
  if (high_bits >= (1 << 27))
    while ((high_bits >> k) >= (1 << 26)) ++k;
  return k;
}

// The exponent kw of a pivot column's weighted copy, p_i 2^(2 er_i + kw): entries
// below 2^56 (top: the largest log2 |p_i 2^(2 er_i)|^2), and inner products with the
// remaining columns, which |p|^2 2^kw bounds (pn = |p|^2, the largest left), below
// 2^(56 + 57).  They are kept as multiples of 2^(56 - sh), sh = fx_dot_shift, so that
// an inner product near the bound has 57 bits whatever the columns' shape.  As large
// as both allow: the low x low products that fx_mac drops are up to 2^54 each, and
// beside |p|^2 2^kw they are what is lost.
TNRC_HD int fx_pivot_weight(int top, float pn) {
  const int a = (111 - top) >> 1, b = 112 - fx_ilog2f(pn);
  return a < b ? a : b;
}
TNRC_HD int fx_dot_shift(int kw, float pn) {
  const int sh = 112 - fx_ilog2f(pn) - kw;
  return sh < 27 ? sh : 27;
}

// 1 / sqrt(N 2^-56) in units of 2^-56, for N in about [2^54, 2^56]: the float
// estimate y0 and one third-order step, y = y0 (1 + e/2 + 3 e^2 / 8) with e =
// 1 - a y0^2 formed in integers.
TNRC_HD long long fx_rsqrt(long long N) {
  const float y0f = fx_rsqrtf(fx_to_float(N) * 1.3877787807814457e-17f);   // 2^-56
  const int Y0 = fx_rint(y0f * 268435456.0f);
  const long long one = 1ll << 56;
  const long long e = one - fx_mul(fx_split(N), fx_split((long long)Y0 * Y0));
  const float ef = fx_to_float(e);
  const long long g = (e >> 1) + (long long)fx_rint(ef * ef * (0.375f * 1.3877787807814457e-17f));
  const Fx gs = fx_split(g);
  return ((long long)Y0 << 28) + (long long)Y0 * gs.hi + (((long long)Y0 * gs.lo + (1ll << 27)) >> 28);
}

// The plane rotation that orthogonalises two columns a and b held as integers
// A 2^ea and B 2^eb, from their inner products in integers (aa = |A|^2 2^-56,
// bb = |B|^2 2^-56, ab = <A, B> 2^-56) and de = eb - ea:
//   A' = c A - conj(s2) B,  B' = c B + s3 A,
// s2 = s 2^de, s3 = s 2^-de.  The angle is computed in FP32 (which only slows
// the quadratic convergence below |cos| = 1e-7, where it no longer matters),
// from the difference |b|^2 - |a|^2 taken in integers, so that equal norms
// are seen as equal; s is that float, exactly, and c = sqrt(1 - |s|^2) is
// completed to 2^-55 in integers (two Newton steps), so the rotation is
// unitary to better than FP64 rounding.  ka, kb: left shifts (negative: right)
// that bring the norms of A', B' back towards 2^56 when they have left
// [2^54, 2^57).
struct FxRot {
  Fx c, s2x, s2y, s3x, s3y;
  int ka, kb;
  float s2;   // sin^2 of the angle
};

TNRC_HD void fx_rotation(long long aa, long long bb, long long abr, long long abi, int de, float af, float bf,
                         float xr, float xi, float ab2, FxRot& R) {
  const float dn1 = 9.094947017729282e-13f;   // 2^-40: the scale of af, bf, xr, xi
  // mixed-unit difference D = bb 2^de - aa 2^-de
  float D;
  const int ad = de < 0 ? -de : de;
  if (ad <= 2 && aa < (1ll << 58) && bb < (1ll << 58)) {
    const long long d = de >= 0 ? (bb << (2 * ad)) - aa : bb - (aa << (2 * ad));
    D = fx_to_float(d) * dn1 * fx_pow2f(-ad);
  } else {
    D = bf * fx_pow2f(de) - af * fx_pow2f(-de);
  }
  // cos 2theta = |D| w, w = 1 / sqrt(D^2 + 4 |ab|^2), c = sqrt((1 + cos 2theta) /
  // 2), s e^{i phi} = sign(D) w / c ab, scaled by inv against overflow: three
  // dependent reciprocals and roots
  const float inv = fx_rcpf(fmaxf(fabsf(D), 2.0f * (fabsf(xr) + fabsf(xi))));
  const float dn = fabsf(D) * inv, an2 = 4.0f * ab2 * inv * inv;
  const float w = fx_rsqrtf(fmaf(dn, dn, an2));
  const float hq = fmaf(0.5f, dn * w, 0.5f);   // c^2
  const float rc = fx_rsqrtf(hq);
  const float c0 = hq * rc;
  const float f = copysignf(inv * w * rc, D);
  float sx = f * xr, sy = f * xi;
  R.s2 = sx * sx + sy * sy;
  const float p = fx_pow2f(de), q = fx_pow2f(-de);
  float dt = ab2 * f * rc;   // tan theta |ab|, with the sign of D
  if (!(fmaxf(fabsf(sx), fabsf(sy)) * fmaxf(p, q) < 7.5f)) {
    // scales out of date by more than the limbs hold (cannot happen while the
    // shifts below keep up): refresh them, rotate in a later round
    sx = sy = dt = 0.0f;
  }
  R.s2x = fx_from_float(sx * p);
  R.s2y = fx_from_float(sy * p);
  R.s3x = fx_from_float(sx * q);
  R.s3y = fx_from_float(sy * q);
  // c = sqrt(1 - |s|^2), |s|^2 = s2 s3
  FxAcc pp{0, 0};
  fx_mac(pp, R.s2x, R.s3x);
  fx_mac(pp, R.s2y, R.s3y);
  const long long P = fx_sum(pp);
  const float cf = (sx == 0.0f && sy == 0.0f) ? 1.0f : c0;
  const float hc = 0.5f * fx_rcpf(cf);
  const int C0 = fx_rint(cf * 268435456.0f);
  const long long rest = (1ll << 56) - P;
  const long long r0 = rest - (long long)C0 * C0;   // below 2^34
  const long long C1 = ((long long)C0 << 28) + ((long long)fx_rint(fx_to_float(r0) * hc * 0.0625f) << 4);
  const Fx c1 = fx_split(C1);
  const long long r1 = rest - (long long)c1.hi * c1.hi - (((long long)c1.hi * c1.lo + (1ll << 26)) >> 27);
  R.c = fx_split(C1 + fx_rint(fx_to_float(r1) * hc));
  // norms after the rotation (in 2^-40 of the units of aa): ilog2 16 is 2^56
  const float na = fmaxf(af - dt * p, af * 5.9604645e-8f), nb = fmaxf(bf + dt * q, bf * 5.9604645e-8f);
  const int la = fx_ilog2f(na) + 40, lb = fx_ilog2f(nb) + 40;
  R.ka = (la >= 52 && la < 58) ? 0 : (55 - la) >> 1;
  R.kb = (lb >= 52 && lb < 58) ? 0 : (55 - lb) >> 1;
}

}  // namespace tnrc
