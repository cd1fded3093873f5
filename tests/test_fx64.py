"""The fixed-point arithmetic of the FP64 path (csrc/fx64.cuh), whose functions are host and device
code, against extended precision on the CPU.  Every bound is the one its comment states, in units of
the last place of the integers."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_01178_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "fx64.cuh"
typedef long double L;
static std::mt19937_64 g(1812);
static L two(int e) { return ldexpl(1.0L, e); }
static fx_t val(int bits) {  // signed, below 2^bits, of any size
  fx_t x = (fx_t)(g() >> (64 - bits)) >> (g() % bits);
  return (g() & 1) ? -x : x;
}
static double dbl(int lo, int hi) {
  const double m = 1.0 + (double)(g() >> 12) * 0x1p-52;
  return std::ldexp((g() & 1) ? -m : m, lo + (int)(g() % (unsigned)(hi - lo)));
}
static L coef(FxCoef c) { return ((L)c.h * 4294967296.0L + (L)c.l) * two(-62); }
#define CHECK(c, ...) do { if (!(c)) { printf(__VA_ARGS__); printf("\n"); return 1; } } while (0)
int main() {
  for (int n = 0; n < 400000; ++n) {
    // FP64 to integer: nearest (fx_from), cut towards zero (fx_cut)
    const int e = 300 + (int)(g() % 1400), t = 1 + (int)(g() % 8);
    const double d = std::ldexp(dbl(-70, 1), e - 1023);
    const L x = (L)d * two(62 - (e + t - 1023));
    CHECK(fabsl((L)fx_from(d, e + t) - x) <= 0.5L, "from %a %d", d, t);
    const L c = (L)fx_cut(d, e + 2), y = (L)d * two(62 - (e + 2 - 1023));
    CHECK(fabsl(c) <= fabsl(y) && fabsl(c - y) < 1.0L, "cut %a", d);
    // and back, nearest: half of a unit of 2^-53 of the value
    const fx_t v = val(62);
    const L w = (L)v * two(e - 1023 - 62);
    CHECK(fabsl((L)fx_to(v, e) - w) <= two(-53) * fabsl(w), "to %lld", v);
    CHECK(fabsl((L)(fx_double(v) * fx_unit(e)) - w) <= two(-53) * fabsl(w), "double %lld", v);
    // products: a unit and a half (rounding, and the dropped product of the low limbs)
    const fx_t a = val(62), b = val(62);
    CHECK(fabsl((L)fx_mulhi(a, b) - (L)a * (L)b * two(-64)) <= 1.5L, "mulhi");
    CHECK(fabsl((L)fx_sqrhi(a) - (L)a * (L)a * two(-64)) <= 1.5L, "sqrhi");
    // complex product with a twiddle: sum of two products a component, 2^-sh
    const int sh = (int)(g() % 3);
    const double th = 6.28318530717958648 * (double)(g() >> 11) * 0x1p-53;
    FxTw tw{fx_limbs((fx_t)llroundl(cosl(th) * two(62))), fx_limbs((fx_t)llroundl(sinl(th) * two(62)))};
    const Fx2 z{val(59 + sh), val(59 + sh)};
    const L cc = coef(tw.c), ss = coef(tw.s), sc = two(-sh);
    const Fx2 p = fx_cmul<-1>(z, tw, sh), q = fx_cmul<1>(z, tw, sh);
    CHECK(fabsl((L)p.x - ((L)z.x * cc + (L)z.y * ss) * sc) <= 2.5L && fabsl((L)p.y - ((L)z.y * cc - (L)z.x * ss) * sc) <= 2.5L, "cmul-");
    CHECK(fabsl((L)q.x - ((L)z.x * cc - (L)z.y * ss) * sc) <= 2.5L && fabsl((L)q.y - ((L)z.y * cc + (L)z.x * ss) * sc) <= 2.5L, "cmul+");
    CHECK(fabsl((L)fx_shr(a, sh) - (L)a * sc) <= 0.5L, "shr");
    // a sum of five products whose scales lie up to 60 binary orders apart: the weights' sum stays
    // below 1, and the result within a unit a term
    double co[5];
    int et[5], em = FX_NONE;
    fx_t X[5];
    for (int k = 0; k < 5; ++k) {
      co[k] = g() % 8 ? dbl(-30, 30) : 0.0;
      et[k] = 900 + (int)(g() % 60);
      X[k] = val(k < 2 ? 62 : 61);
      em = std::max(em, fx_wexp(co[k], et[k]));
    }
    unsigned parts = 0;
    for (int k = 0; k < 5; ++k) parts += fx_wpart(co[k], fx_wexp(co[k], et[k]), em);
    const int er = fx_wscale(em, parts);
    FxAcc s = fx_wacc(0);
    L ref = 0, weights = 0;
    for (int k = 0; k < 5; ++k) {
      if (fx_wexp(co[k], et[k]) == FX_NONE) continue;
      fx_wmac(s, X[k], fx_wcoef(co[k], et[k], er));
      ref += (L)X[k] * (L)co[k] * two(et[k] - er);
      weights += fabsl((L)co[k]) * two(et[k] + 2 - er);
      if (k == 2) fx_wfold(s);
    }
    CHECK(weights < 1.0L, "weights %Lg", weights);
    CHECK(fabsl((L)fx_wsum(s) - ref) <= 6.0L, "wsum %Lg", (L)fx_wsum(s) - ref);
    const double wl = (double)(g() >> 11) * 0x1p-53 * 0.999 + 0.0005;
    const fx_t i0 = val(61), i1 = val(61);
    const FxCoef c0 = fx_limbs(fx_from(wl, 1023)), c1 = fx_limbs(fx_from(1.0 - wl, 1023));
    CHECK(fabsl((L)fx_interpolate(i0, i1, c0, c1) - 2.0L * ((L)i0 * (L)wl + (L)i1 * (L)(1.0 - wl))) <= 16.0L, "interp");
    CHECK(fabsl((L)fx_mul_s3(a) - (L)a * 0.866025403784438646763723170752936L) <= 4.0L, "s3");
  }
  for (double z : {0.0, -0.0, 5e-324, 2e-308}) CHECK(fx_from(z, 1024) == 0 && fx_cut(z, 1025) == 0, "zero");
  CHECK(fx_to(0, 1023) == 0.0 && fx_double(0) == 0.0, "to zero");
  return 0;
}
"""


def test_fixed_point_arithmetic(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "fx64_check.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "fx64_check")
    subprocess.run([gxx, "-O1", "-std=c++17", "-x", "c++", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
