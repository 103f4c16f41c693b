"""The integer arithmetic of the trajectory kernel's SVD (csrc/fx.cuh) on the
CPU: its scalars compiled with the host compiler against long double."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
FX = os.path.join(HERE, "..", "paper_2603_03639_gb300", "csrc", "fx.cuh")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "%s"
using namespace tnrc;
static double uni(std::mt19937_64& g) { return std::generate_canonical<double, 53>(g); }
int main() {
  std::mt19937_64 g(7);
  const long double one = powl(2, 56);
  double e_split = 0, e_rsqrt = 0, e_unit = 0, e_angle = 0, e_float = 0;
  for (int t = 0; t < 100000; ++t) {
    const long long v = (long long)(g() >> 5) - (1ll << 58);
    const Fx s = fx_split(v);
    if (fx_val(s) != v || s.lo < -(1 << 27) || s.lo >= (1 << 27)) e_split = 1;
    const long long small = v >> (g() %% 59);
    if (small) e_float = fmax(e_float, fabs((double)fx_to_float(small) / (double)small - 1));
    const long long N = (1ll << 54) + (long long)(g() %% (3ull << 54));
    e_rsqrt = fmax(e_rsqrt, (double)fabsl(fx_rsqrt(N) / one * sqrtl(N / one) - 1));
    // two columns: norms over the range that is kept, any angle, equal norms among them
    long long aa = (long long)exp2(52 + 6 * uni(g)), bb = (long long)exp2(52 + 6 * uni(g));
    int de = (int)(g() %% 9) - 4;
    if (t %% 3 == 0) { bb = aa + (long long)(g() %% 64); de = 0; }
    const double mag = sqrt((double)aa * bb) * exp2(-50 * uni(g)) * 0.99, ph = 6.283185307 * uni(g);
    const long long xr = (long long)(mag * cos(ph)), xi = (long long)(mag * sin(ph));
    const float k = 9.094947017729282e-13f, af = fx_to_float(aa) * k, bf = fx_to_float(bb) * k;
    const float fr = fx_to_float(xr) * k, fi = fx_to_float(xi) * k, ab2 = fr * fr + fi * fi;
    if (!(ab2 > 0)) continue;
    FxRot R;
    fx_rotation(aa, bb, xr, xi, de, af, bf, fr, fi, ab2, R);
    const long double c = fx_val(R.c) / one, px = fx_val(R.s2x) / one, py = fx_val(R.s2y) / one;
    const long double qx = fx_val(R.s3x) / one, qy = fx_val(R.s3y) / one;
    e_unit = fmax(e_unit, (double)fabsl(c * c + px * qx + py * qy - 1));
    // <a', b'> 2^-de relative to the norms: what the rotation leaves of the pair's cosine
    if (px == 0 && py == 0) continue;
    const long double d = powl(2, de), A = aa, B = bb * d * d, X = xr * d, Y = xi * d;   // in units of |a|^2
    const long double sx = px / d, sy = py / d;                                          // s, a' = c a - conj(s) b, b' = c b + s a
    const long double re = c * c * X - (sx * sx - sy * sy) * X - 2 * sx * sy * Y + c * sx * (A - B);
    const long double im = c * c * Y + (sx * sx - sy * sy) * Y - 2 * sx * sy * X + c * sy * (A - B);
    const long double was = sqrtl((X * X + Y * Y) / (A * B));
    if (was > 1e-9L) e_angle = fmax(e_angle, (double)(sqrtl((re * re + im * im) / (A * B)) / was));
  }
  printf("%%.3e %%.3e %%.3e %%.3e %%.3e\n", e_split, e_float, e_rsqrt, e_unit, e_angle);
}
"""


def test_fixed_point_scalars(tmp_path):
    """Splitting is exact; the float of a 64-bit integer has float accuracy; the
    reciprocal square root and the rotation's unitarity hold to 2^-54 (four units
    of 2^-56: two roundings and the dropped low products); the FP32 angle leaves
    at most 1e-5 of a pair's cosine (FP32 rounding, 6e-8, amplified by the
    cancellation in |b|^2 - |a|^2 outside the exact range)."""
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "fx.cpp", tmp_path / "fx"
    src.write_text(PROGRAM % os.path.abspath(FX))
    subprocess.run([gxx, "-O2", "-std=c++17", "-o", str(exe), str(src)], check=True)
    split, flt, rsq, unit, angle = (float(x) for x in subprocess.run([str(exe)], capture_output=True, text=True,
                                                                   check=True).stdout.split())
    assert split == 0.0
    assert flt <= 2.0 ** -23
    assert rsq <= 2.0 ** -54
    assert unit <= 2.0 ** -54
    assert angle <= 1e-5
