// 64-bit fixed-point arithmetic on the integer pipes, for FP64 values of one common scale.
//
// The FP64 unit of this part takes a warp instruction every 16 cycles per SM (2 lanes per clock);
// the integer pipes take 24 lanes per clock of 32 x 32 + 64 -> 64 multiply-adds (mad.wide) and 62
// of 64-bit additions (measured).  A product of a 64-bit fixed-point number and a 62-bit coefficient
// is three multiply-adds and a few shifts, so a transform or a stencil whose operands share a scale
// runs several times faster than in FP64, and keeps 60 bits below the largest operand where FP64
// keeps 53 below each result.
//
// A value x is held as the integer X = x 2^(F - e): e is the common exponent (the biased binary64
// exponent of the largest magnitude) and F says where its leading bit stands.  Functions are
// __host__ __device__ so that their arithmetic is checked on the CPU.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

typedef long long fx_t;

FX_HD int fx_hi(fx_t x) { return (int)(x >> 32); }
FX_HD unsigned fx_lo(fx_t x) { return (unsigned)x; }
// One multiply-add of 32 x 32 + 64 bits.  (Written as a C product of operands cut out of 64-bit values
// the compiler forms some of them from three or four multiplications.)
FX_HD fx_t fx_mad(int a, int b, fx_t c) {
#ifdef __CUDA_ARCH__
  fx_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (fx_t)a * b + c;
#endif
}
FX_HD uint64_t fx_bits(double d) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(d);
#else
  uint64_t b;
  __builtin_memcpy(&b, &d, 8);
  return b;
#endif
}
FX_HD double fx_from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}
FX_HD int fx_clz(uint64_t x) {  // 64 for 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// High word of |d|: its maximum over a set, shifted right by 20, is the set's common exponent.
FX_HD unsigned fx_mag(double d) { return (unsigned)(fx_bits(d) >> 32) & 0x7fffffffu; }

// Common exponents the fixed-point path takes: no infinities or NaN, no result near the ends of the
// binary64 range.  A set of zeros counts as exponent 1023.
FX_HD bool fx_exponent_ok(int e) { return e >= 128 && e <= 1920; }
FX_HD int fx_exponent(unsigned maxhi) { return maxhi == 0 ? 1023 : (int)(maxhi >> 20); }

// d as an integer with the leading bit of a value of exponent e at bit 62 - t: pass s = e + t.
// Rounded to the nearest integer.  t >= 1 keeps |X| <= 2^62.
FX_HD fx_t fx_from(double d, int s) {
  const uint64_t b = fx_bits(d);
  const unsigned hi = (unsigned)(b >> 32);
  int sh = s - (int)((hi >> 20) & 0x7ffu);
  sh = sh < 64 ? sh : 64;  // zeros and subnormals end here as well: their implicit bit is shifted out
  const uint64_t m = ((((uint64_t)((hi & 0xfffffu) | 0x100000u)) << 32) | (uint32_t)b) << 10;
  const fx_t v = (fx_t)(((m >> (sh - 1)) + 1) >> 1);
  const fx_t sg = (fx_t)((int)hi >> 31);
  return (v ^ sg) - sg;
}

// The double nearest to x (ties upwards in magnitude) where bit 62 stands for the biased exponent e
FX_HD double fx_to(fx_t x, int e) {
  const fx_t sg = x >> 63;
  const uint64_t m0 = (uint64_t)((x ^ sg) - sg);
  // 32-bit steps: normalise the high word, or the low one where that is zero
  const bool low = (m0 >> 32) == 0;
  unsigned th = low ? (unsigned)m0 : (unsigned)(m0 >> 32), tl = low ? 0u : (unsigned)m0;
#ifdef __CUDA_ARCH__
  const int n = __clz((int)th);
  const bool zero = th == 0;
  th = __funnelshift_l(tl, th, n);
  tl <<= n & 31;
  const unsigned bl = __funnelshift_r(tl, th, 11);
#else
  const bool zero = th == 0;
  const int n = zero ? 0 : __builtin_clz(th);
  const uint64_t m = (((uint64_t)th << 32) | tl) << n;
  th = (unsigned)(m >> 32);
  tl = (unsigned)m;
  const unsigned bl = (unsigned)(m >> 11);
#endif
  // 53 leading bits, rounded; the implicit bit and a carry out of the fraction add to the exponent
  const unsigned bh = (th >> 11) + ((unsigned)(e - n - (low ? 32 : 0)) << 20);
  uint64_t b = (((uint64_t)bh << 32) | bl) + ((tl >> 10) & 1);
  b = zero ? 0 : b;
  return fx_from_bits(b | ((uint64_t)sg & 0x8000000000000000ull));
}

// x as a double, rounded, by two FP64 instructions (the high limb scaled by 2^32 is exact)
FX_HD double fx_double(fx_t x) {
  const double h = fx_from_bits(0x4330000000000000ull | ((uint64_t)(x >> 32) & 0xffffffffull) ^ 0x80000000ull);
  const double l = fx_from_bits(0x4330000000000000ull | (uint64_t)(uint32_t)x);
  // h = 2^52 + 2^31 + hi, l = 2^52 + lo
#ifdef __CUDA_ARCH__
  return fma(h, 0x1p32, -(0x1p84 + 0x1p63 + 0x1p52)) + l;
#else
  return (h * 0x1p32 - (0x1p84 + 0x1p63 + 0x1p52)) + l;
#endif
}
// the unit of a sum at scale e: 2^(e - 1023 - 62)
FX_HD double fx_unit(int e) { return fx_from_bits((uint64_t)(uint32_t)(e - 62) << 52); }

// Two signed limbs: x = h 2^32 + l, |l| <= 2^31.  Products drop l times l only, whose mean is zero: a
// bias, however small, would add up in the lowest modes, which the pressure solve amplifies.
struct FxCoef {
  int h, l;
};
FX_HD FxCoef fx_limbs(fx_t x) {
  const int l = (int)x;
  return FxCoef{fx_hi(x) - (l >> 31), l};
}
// A coefficient |w| <= 1 is held as the limbs of w 2^62
FX_HD FxCoef fx_neg(FxCoef w) { return FxCoef{-w.h, -w.l}; }

struct alignas(16) Fx2 {
  fx_t x, y;
};
FX_HD Fx2 fx_add(Fx2 a, Fx2 b) { return Fx2{a.x + b.x, a.y + b.y}; }
FX_HD Fx2 fx_sub(Fx2 a, Fx2 b) { return Fx2{a.x - b.x, a.y - b.y}; }

// Twiddle exp(-i th): c = cos th, s = sin th (both |.| <= 1)
struct alignas(16) FxTw {
  FxCoef c, s;
};

// a times the twiddle (SIGN < 0: exp(-i th), SIGN > 0: its conjugate), times 2^-sh, sh = 0, 1 or 2.
// |a| <= 2^(59.5 + sh) in modulus keeps every partial sum in range.
template <int SIGN>
FX_HD Fx2 fx_cmul(Fx2 a, FxTw w, int sh) {
  const FxCoef ns = fx_neg(w.s);
  const FxCoef sr = SIGN < 0 ? w.s : ns, si = SIGN < 0 ? ns : w.s;
  const FxCoef x = fx_limbs(a.x), y = fx_limbs(a.y);
  const int x2 = (int)((unsigned)x.h << (2 - sh)), y2 = (int)((unsigned)y.h << (2 - sh));
  // half a unit, less four bits of the last place for half of the values: with w = 1 the sums end in
  // ties, and rounding those one way would add up in mode 0
  const fx_t r0 = (fx_t)1 << (29 + sh);  // 2^31 for sh = 2
  const fx_t mr = fx_mad(x.l, w.c.h, fx_mad(x.h, w.c.l, fx_mad(y.l, sr.h, fx_mad(y.h, sr.l, r0 - (x.l & 4)))));
  const fx_t mi = fx_mad(y.l, w.c.h, fx_mad(y.h, w.c.l, fx_mad(x.l, si.h, fx_mad(x.h, si.l, r0 - (y.l & 4)))));
  const fx_t hr = fx_mad(x2, w.c.h, fx_mad(y2, sr.h, 0));
  const fx_t hi = fx_mad(y2, w.c.h, fx_mad(x2, si.h, 0));
  return Fx2{hr + (mr >> (30 + sh)), hi + (mi >> (30 + sh))};
}
// a 2^-sh, rounded to the nearest (ties to even), sh = 0, 1 or 2
FX_HD fx_t fx_shr(fx_t a, int sh) {
  const int even = (int)(fx_lo(a) >> sh) & (sh > 0 ? 1 : 0);
  return (a + ((sh >> 1) + even)) >> sh;
}
FX_HD Fx2 fx_shr(Fx2 a, int sh) { return Fx2{fx_shr(a.x, sh), fx_shr(a.y, sh)}; }

// Butterflies.  Inputs already scaled and twiddled; outputs at most the sum of the input moduli.
template <int SIGN>
FX_HD void fx_bfly4(Fx2 a, Fx2 b, Fx2 c, Fx2 d, Fx2* y) {
  const Fx2 t0 = fx_add(a, c), t1 = fx_sub(a, c), t2 = fx_add(b, d), t3 = fx_sub(b, d);
  const Fx2 r3 = SIGN < 0 ? Fx2{t3.y, -t3.x} : Fx2{-t3.y, t3.x};
  y[0] = fx_add(t0, t2);
  y[2] = fx_sub(t0, t2);
  y[1] = fx_add(t1, r3);
  y[3] = fx_sub(t1, r3);
}
// x sqrt(3)/2 (|x| < 2^62): 2^62 sqrt(3) / 2 = 0x376cf5d0b09954e7...
FX_HD fx_t fx_mul_s3(fx_t a) {
  const FxCoef w = {0x376cf5d1, (int)0xb09954e7u}, x = fx_limbs(a);
  const fx_t m = fx_mad(x.l, w.h, fx_mad(x.h, w.l, (fx_t)1 << 29));
  return fx_mad(x.h, w.h, 0) * 4 + (m >> 30);
}
template <int SIGN>
FX_HD void fx_bfly3(Fx2 a, Fx2 b, Fx2 c, Fx2* y) {
  const Fx2 S = fx_add(b, c), D = fx_sub(b, c);
  y[0] = fx_add(a, S);
  const Fx2 T = Fx2{a.x - fx_shr(S.x, 1), a.y - fx_shr(S.y, 1)};
  const Fx2 G = SIGN < 0 ? Fx2{fx_mul_s3(D.x), fx_mul_s3(D.y)} : Fx2{-fx_mul_s3(D.x), -fx_mul_s3(D.y)};
  y[1] = Fx2{T.x + G.y, T.y - G.x};
  y[2] = Fx2{T.x - G.y, T.y + G.x};
}
// Bits set above the leading bits of both components: the or over a set gives the set's scale
FX_HD unsigned fx_span(Fx2 a) {
  const int x = fx_hi(a.x), y = fx_hi(a.y);
  return (unsigned)((x ^ (x >> 31)) | (y ^ (y >> 31)));
}

// ---- sums of products with coefficients of any size (the stencils)
//
// A coefficient c meeting values whose bit 62 stands for the exponent et enters a sum whose bit 62
// stands for er as w = c 2^(et + 2 - er), |w| < 1; the sum of X w / 4 over terms |X| <= 2^62 whose
// |w| add up to less than 1 stays below 2^60.
FX_HD FxCoef fx_wcoef(double c, int et, int er) { return fx_limbs(fx_from(c, 1021 - et + er)); }
// h + m / 2^32.  Room in m: the |X| of the terms between two folds add up to at most 2^63.3 (2.5
// times 2^62).
struct FxAcc {
  fx_t h, m;
};
FX_HD FxAcc fx_wacc(fx_t x) { return FxAcc{x, (fx_t)1 << 31}; }
FX_HD void fx_wmac(FxAcc& a, fx_t v, FxCoef w) {  // adds X w / 4
  const FxCoef x = fx_limbs(v);
  a.h = fx_mad(x.h, w.h, a.h);
  a.m = fx_mad(x.l, w.h, fx_mad(x.h, w.l, a.m));
}
FX_HD void fx_wfold(FxAcc& a) {
  a.h += a.m >> 32;
  a.m = (fx_t)(uint32_t)a.m;
}
FX_HD fx_t fx_wsum(const FxAcc& a) { return a.h + (a.m >> 32); }
// x0 c0 + x1 c1 of weights c0 + c1 <= 1 and values up to 2^61, brought up to 2^62
FX_HD fx_t fx_interpolate(fx_t x0, fx_t x1, FxCoef c0, FxCoef c1) {
  FxAcc s = {0, (fx_t)1 << 28};
  fx_wmac(s, x0, c0);
  fx_wmac(s, x1, c1);
  return s.h * 8 + (s.m >> 29);
}
// The part of the sum of |c| 2^(et + 2) one term takes, relative to 2^(emax - 1023 - 20) (emax: the
// largest ee of the terms), rounded up; ee = fx_wexp(c, et)
constexpr int FX_NONE = -100000;
FX_HD int fx_wexp(double c, int et) {
  const int ec = (int)(fx_mag(c) >> 20);
  return ec == 0 ? FX_NONE : ec + et + 2;
}
FX_HD unsigned fx_wpart(double c, int ee, int emax) {
  const int d = emax - ee;
  return ee == FX_NONE ? 0u : d > 24 ? 1u : ((((fx_mag(c) & 0xfffffu) | 0x100000u) + 1) >> d) + 1;
}
FX_HD int fx_wscale(int emax, unsigned parts) {  // er
  return emax == FX_NONE ? 1023 : emax - 1023 - 20 + (64 - fx_clz(parts));
}
// X Y / 2^64 of |X|, |Y| <= 2^62, to about one unit
FX_HD fx_t fx_mulhi(fx_t a, fx_t b) {
  const FxCoef x = fx_limbs(a), y = fx_limbs(b);
  return fx_mad(x.h, y.h, 0) + (fx_mad(x.l, y.h, fx_mad(x.h, y.l, (fx_t)1 << 31)) >> 32);
}
FX_HD fx_t fx_sqrhi(fx_t a) {
  const FxCoef x = fx_limbs(a);
  return fx_mad(x.h, x.h, 0) + (fx_mad(x.l, x.h, (fx_t)1 << 30) >> 31);
}
// fx_from for planes of a common exponent e = s - 2, cut towards zero
FX_HD fx_t fx_cut(double d, int s) {
  const uint64_t b = fx_bits(d);
  const unsigned hi = (unsigned)(b >> 32);
  int sh = s - 2 - (int)((hi >> 20) & 0x7ffu);
  sh = sh < 63 ? sh : 63;
  const fx_t v = (fx_t)((((((uint64_t)((hi & 0xfffffu) | 0x100000u)) << 32) | (uint32_t)b) << 8) >> sh);
  const fx_t sg = (fx_t)((int)hi >> 31);
  return (v ^ sg) - sg;
}
