// 64-bit fixed-point arithmetic for the transforms of the FP64-class precisions.
//
// GB300 issues 2 FP64 operations per clock and SM against 128 32-bit integer ones, so an FP64
// transform of 256 points (20 FP64 instructions per element) keeps that pipe busy for eight
// times as long as its bytes take from HBM.  A transform's error is relative to its line's norm
// whatever the arithmetic, so it may as well run on block fixed point: the elements of a CTA's
// tile as 64-bit integers under one exponent, exact additions (two 32-bit instructions instead
// of an FP64 one), products by 64-bit constants through three 32 x 32 -> 64 multiply-adds.
// With components below 2^58 on entry, a stage's outputs stay below 2^62 up to radix 10, and the
// tile is rescaled by its largest output before the next stage, so the last bit stays at 2^-58 of
// the tile's largest element: below an FP64 rounding of the elements' rms up to 512 points.
// Bound by integer issue (about 200 instructions per complex element and pass).  Measured, us, the
// FP64 transforms -> these: 256^3 K1 430 -> 127, K2 328 -> 74, K3 690 -> 170.  Phi against extended precision
// (rel-L2, clouds and noise, 36 .. 480 points): 3.8e-16 .. 7.1e-16 -> 2.3e-16 .. 4.2e-16.
#pragma once
#include <cstring>

#include "dgpe_stages.cuh"

namespace dgpe {

#define DGPE_HD __host__ __device__ __forceinline__

struct fxc {   // a complex value under the tile's exponent
  long long re, im;
};
DGPE_HD fxc operator+(fxc a, fxc b) { return {a.re + b.re, a.im + b.im}; }
DGPE_HD fxc operator-(fxc a, fxc b) { return {a.re - b.re, a.im - b.im}; }
template <int DIR>
DGPE_HD fxc fx_rot(fxc a) { return DIR < 0 ? fxc{a.im, -a.re} : fxc{-a.im, a.re}; }   // times DIR i

// a = hi 2^32 + lo with a signed lo, so that every product below is a signed one
DGPE_HD int fx_hi(long long a) { return (int)(a >> 32) + (int)((unsigned)a >> 31); }
DGPE_HD int fx_lo(long long a) { return (int)(unsigned)a; }
// a b + c, one instruction (written out: the compiler widens some of these products to 64 x 64 bits)
DGPE_HD long long fx_mad(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (long long)a * b + c;
#endif
}
constexpr long long kFxHalf = 0x80000000LL;

// a w / 2^64 (the product of the low words, less than half a unit, left out).  |a| < 2^63 - 2^31,
// |w| < 2^63 - 2^31 and |a| |w| < 2^125.
DGPE_HD long long fx_mul(long long a, int wh, int wl) {
  const int ah = fx_hi(a), al = fx_lo(a);
  const long long mid = fx_mad(ah, wl, fx_mad(al, wh, kFxHalf));
  return fx_mad(ah, wh, mid >> 32);
}
// a (n + f / 2^64), n = -1, 0, 1 and |f| < 2^63: a real constant to 64 fraction bits
template <int NI, unsigned long long F>
DGPE_HD long long fx_const(long long a) {
  constexpr long long f = (long long)F;
  constexpr int fl = (int)(unsigned)F, fh = (int)((f - fl) / 4294967296LL);
  const long long p = fx_mul(a, fh, fl);
  return NI == 0 ? p : NI > 0 ? p + a : p - a;
}

// A twiddle w 2^60, split into signed words.  The low word of the imaginary part is never -2^31, which
// has no 32-bit negative: fx_words, by which every factor is made, moves such a value by one unit.
struct __align__(16) fxw {
  int rh, rl, ih, il;
};
DGPE_HD fxw fx_words(long long re, long long im) {
  if (fx_lo(im) == (int)0x80000000) ++im;
  return {fx_hi(re), fx_lo(re), fx_hi(im), fx_lo(im)};
}
// a w / 2^64 = a w / 16 (DIR < 0) or a conj(w) / 16, for components of a below 2^62 (|a| below
// 2^62.5): the middle sums stay below 2^62 + 2^60.  (The negatives in 32 bits cost nothing; with sums
// subtracted in 64 bits K3 at 256^3 took 191 us instead of 171.)
template <int DIR>
DGPE_HD fxc fx_twiddle(fxc a, fxw w) {
  const int rh = fx_hi(a.re), rl = fx_lo(a.re), ih = fx_hi(a.im), il = fx_lo(a.im);
  const int wih = DIR < 0 ? w.ih : -w.ih, wil = DIR < 0 ? w.il : -w.il;
  const long long mr = fx_mad(rh, w.rl, fx_mad(rl, w.rh, fx_mad(ih, -wil, fx_mad(il, -wih, kFxHalf))));
  const long long mi = fx_mad(rh, wil, fx_mad(rl, wih, fx_mad(ih, w.rl, fx_mad(il, w.rh, kFxHalf))));
  return {fx_mad(rh, w.rh, fx_mad(ih, -wih, mr >> 32)), fx_mad(rh, wih, fx_mad(ih, w.rh, mi >> 32))};
}

// ---- block scaling -------------------------------------------------------------------------
// Every stage of a transform starts from components below 2^kFxBits, so that the outputs of its
// radix P <= 10 stay below 10 2^58.5 < 2^62.  The largest output of the tile (the or of the
// magnitudes' high words, exchanged at the barrier that ends the stage) gives the shift to the
// next stage's range: down by the growth that there was, not by the most that there could be.
constexpr int kFxBits = 58;
DGPE_HD int fx_mag(long long a) { return (int)(a >> 32) ^ (int)(a >> 63); }   // bits of the high word's magnitude
DGPE_HD int fx_mag(fxc a) { return fx_mag(a.re) | fx_mag(a.im); }
// the shift down that takes magnitudes mag to kFxBits bits (negative: up); -26 at least:
// a tile whose outputs nearly all cancelled carries on with fewer bits
DGPE_HD int fx_shift(int mag) {
#ifdef __CUDA_ARCH__
  const int d = 64 - __clz(mag) - kFxBits;
#else
  const int d = (mag ? 64 - __builtin_clz(mag) : 32) - kFxBits;
#endif
  return d;
}
// a 2^-d, rounded
DGPE_HD long long fx_scale(long long a, int d) { return d > 0 ? (a + (1LL << (d - 1))) >> d : a << -d; }
// 16 a 2^-d, the input of fx_twiddle (d <= 4: a radix up to 10 makes components grow by at most
// 10 sqrt 2 < 16)
DGPE_HD fxc fx_up(fxc a, int d) {
  return {(long long)((unsigned long long)a.re << (4 - d)), (long long)((unsigned long long)a.im << (4 - d))};
}

// ---- butterflies (the usual radix-2/3/4/5/7/8 forms and their prime-factor products) --------
template <int DIR>
DGPE_HD void fx_bf2(fxc *v) {
  const fxc t = v[0] - v[1];
  v[0] = v[0] + v[1];
  v[1] = t;
}
template <int DIR>
DGPE_HD void fx_bf3(fxc *v) {
  const fxc t = v[1] + v[2], d = v[1] - v[2];
  const fxc m = {v[0].re - (t.re >> 1), v[0].im - (t.im >> 1)};
  const fxc s = fx_rot<DIR>(fxc{fx_const<1, 0xddb3d742c265539eull>(d.re), fx_const<1, 0xddb3d742c265539eull>(d.im)});
  v[0] = v[0] + t;
  v[1] = m + s;
  v[2] = m - s;
}
template <int DIR>
DGPE_HD void fx_bf4(fxc *v) {
  const fxc a = v[0] + v[2], b = v[0] - v[2], c = v[1] + v[3], d = fx_rot<DIR>(v[1] - v[3]);
  v[0] = a + c;
  v[1] = b + d;
  v[2] = a - c;
  v[3] = b - d;
}
template <int DIR>
DGPE_HD void fx_bf5(fxc *v) {
  const fxc t1 = v[1] + v[4], t2 = v[2] + v[3], d1 = v[1] - v[4], d2 = v[2] - v[3], t = t1 + t2, e = t1 - t2;
  const fxc m = {v[0].re - (t.re >> 2), v[0].im - (t.im >> 2)};
  const fxc q = {fx_const<1, 0x8f1bbcdcbfa53e0bull>(e.re), fx_const<1, 0x8f1bbcdcbfa53e0bull>(e.im)};
  auto s1 = [](fxc a) { return fxc{fx_const<1, 0xf378709a22a7faf3ull>(a.re), fx_const<1, 0xf378709a22a7faf3ull>(a.im)}; };
  auto s2 = [](fxc a) { return fxc{fx_const<1, 0x96791823aad2ef6eull>(a.re), fx_const<1, 0x96791823aad2ef6eull>(a.im)}; };
  const fxc a = m + q, b = m - q;
  const fxc x = fx_rot<DIR>(s1(d1) + s2(d2)), y = fx_rot<DIR>(s2(d1) - s1(d2));
  v[0] = v[0] + t;
  v[1] = a + x;
  v[4] = a - x;
  v[2] = b + y;
  v[3] = b - y;
}
template <int DIR>
DGPE_HD void fx_bf7(fxc *v) {
  const fxc t[3] = {v[1] + v[6], v[2] + v[5], v[3] + v[4]}, d[3] = {v[1] - v[6], v[2] - v[5], v[3] - v[4]};
  auto c1 = [](fxc a) { return fxc{fx_const<1, 0x9f9d07145f6e8b66ull>(a.re), fx_const<1, 0x9f9d07145f6e8b66ull>(a.im)}; };
  auto c2 = [](fxc a) { return fxc{fx_const<0, 0xc708de39fb74fb2dull>(a.re), fx_const<0, 0xc708de39fb74fb2dull>(a.im)}; };
  auto c3 = [](fxc a) { return fxc{fx_const<-1, 0x195a1ab1a51c796dull>(a.re), fx_const<-1, 0x195a1ab1a51c796dull>(a.im)}; };
  auto s1 = [](fxc a) { return fxc{fx_const<1, 0xc8261ba82ef2585eull>(a.re), fx_const<1, 0xc8261ba82ef2585eull>(a.im)}; };
  auto s2 = [](fxc a) { return fxc{fx_const<1, 0xf994e02ac74b471dull>(a.re), fx_const<1, 0xf994e02ac74b471dull>(a.im)}; };
  auto s3 = [](fxc a) { return fxc{fx_const<0, 0x6f130135c6af0401ull>(a.re), fx_const<0, 0x6f130135c6af0401ull>(a.im)}; };
  const fxc p1 = v[0] + c1(t[0]) + c2(t[1]) + c3(t[2]), q1 = fx_rot<DIR>(s1(d[0]) + s2(d[1]) + s3(d[2]));
  const fxc p2 = v[0] + c2(t[0]) + c3(t[1]) + c1(t[2]), q2 = fx_rot<DIR>(s2(d[0]) - s3(d[1]) - s1(d[2]));
  const fxc p3 = v[0] + c3(t[0]) + c1(t[1]) + c2(t[2]), q3 = fx_rot<DIR>(s3(d[0]) - s1(d[1]) + s2(d[2]));
  v[0] = v[0] + t[0] + t[1] + t[2];
  v[1] = p1 + q1;
  v[6] = p1 - q1;
  v[2] = p2 + q2;
  v[5] = p2 - q2;
  v[3] = p3 + q3;
  v[4] = p3 - q3;
}
template <int DIR>
DGPE_HD void fx_bf8(fxc *v) {
  fxc a[4], b[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    a[k] = v[k] + v[k + 4];
    b[k] = v[k] - v[k + 4];
  }
  auto r = [](long long x) { return fx_const<1, 0xb504f333f9de6484ull>(x); };   // 1/sqrt 2
  // e^{DIR i pi/4} = (1 + DIR i)/sqrt 2, e^{DIR 3 i pi/4} = (-1 + DIR i)/sqrt 2
  const fxc i1 = fx_rot<DIR>(b[1]), i3 = fx_rot<DIR>(b[3]);
  b[1] = {r(b[1].re + i1.re), r(b[1].im + i1.im)};
  b[2] = fx_rot<DIR>(b[2]);
  b[3] = {r(i3.re - b[3].re), r(i3.im - b[3].im)};
  fx_bf4<DIR>(a);
  fx_bf4<DIR>(b);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[2 * k] = a[k];
    v[2 * k + 1] = b[k];
  }
}
template <int DIR>
DGPE_HD void fx_bf6(fxc *v) {   // 2 x 3: n = 3 n1 + 2 n2, k = 3 k1 + 4 k2 (mod 6)
  fxc a[3] = {v[0], v[2], v[4]}, b[3] = {v[3], v[5], v[1]};
  fx_bf3<DIR>(a);
  fx_bf3<DIR>(b);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    v[(4 * k) % 6] = a[k] + b[k];
    v[(4 * k + 3) % 6] = a[k] - b[k];
  }
}
template <int DIR>
DGPE_HD void fx_bf10(fxc *v) {   // 2 x 5: n = 5 n1 + 2 n2, k = 5 k1 + 6 k2 (mod 10)
  fxc a[5] = {v[0], v[2], v[4], v[6], v[8]}, b[5] = {v[5], v[7], v[9], v[1], v[3]};
  fx_bf5<DIR>(a);
  fx_bf5<DIR>(b);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    v[(6 * k) % 10] = a[k] + b[k];
    v[(6 * k + 5) % 10] = a[k] - b[k];
  }
}
template <int DIR>
DGPE_HD void fx_bf9(fxc *v) {   // 3 x 3 with the twiddles e^{DIR 2 pi i n2 k1 / 9}
  auto c1 = [](long long a) { return fx_const<1, 0xc41b7d167a81c991ull>(a); };
  auto s1 = [](long long a) { return fx_const<1, 0xa48dba91e0b0e55dull>(a); };
  auto c2 = [](long long a) { return fx_const<0, 0x2c7434fc16e71346ull>(a); };
  auto s2 = [](long long a) { return fx_const<1, 0xfc1c5c6408e0bad0ull>(a); };
  auto c4 = [](long long a) { return fx_const<-1, 0x0f704ded6e972329ull>(a); };
  auto s4 = [](long long a) { return fx_const<0, 0x578ea1d2282fd573ull>(a); };
  auto tw = [](fxc z, auto c, auto s) {
    return DIR < 0 ? fxc{c(z.re) + s(z.im), c(z.im) - s(z.re)} : fxc{c(z.re) - s(z.im), c(z.im) + s(z.re)};
  };
  fxc c[3][3];   // [n2][k1]
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    c[n2][0] = v[n2];
    c[n2][1] = v[n2 + 3];
    c[n2][2] = v[n2 + 6];
    fx_bf3<DIR>(c[n2]);
  }
  c[1][1] = tw(c[1][1], c1, s1);
  c[1][2] = tw(c[1][2], c2, s2);
  c[2][1] = tw(c[2][1], c2, s2);
  c[2][2] = tw(c[2][2], c4, s4);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    fxc t[3] = {c[0][k1], c[1][k1], c[2][k1]};
    fx_bf3<DIR>(t);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = t[k2];
  }
}
template <int DIR, int P>
DGPE_HD void fx_bf(fxc *v) {
  if constexpr (P == 2) fx_bf2<DIR>(v);
  else if constexpr (P == 3) fx_bf3<DIR>(v);
  else if constexpr (P == 4) fx_bf4<DIR>(v);
  else if constexpr (P == 5) fx_bf5<DIR>(v);
  else if constexpr (P == 6) fx_bf6<DIR>(v);
  else if constexpr (P == 7) fx_bf7<DIR>(v);
  else if constexpr (P == 8) fx_bf8<DIR>(v);
  else if constexpr (P == 9) fx_bf9<DIR>(v);
  else fx_bf10<DIR>(v);
}

// ---- FP64 <-> fixed point ----------------------------------------------------------------
// The tile's exponent is the largest biased exponent emax of its values, at least kFxMinBiased (0x7ff:
// some value is not finite, and the tile's results are NaN): x = v 2^(emax - 1075 - UP), |v| < 2^(53 + UP)
// (a tile's: 2^58), cut off at bit 0; subnormal values, 2^-63 below the least tile exponent, are 0.
constexpr int kFxMinBiased = 64;
DGPE_HD long long fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
DGPE_HD double fx_value(long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
DGPE_HD int fx_exponent_bits(double x) { return (int)(fx_bits(x) >> 32) & 0x7fffffff; }   // orders by exponent
template <int UP = 5>
DGPE_HD long long fx_from(double x, int emax) {
  const long long b = fx_bits(x);
  const int s = emax - ((int)(b >> 52) & 0x7ff);
  const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 1ull << 52;
  const long long v = (long long)((m << UP) >> (s < 63 ? s : 63));
  const long long g = b >> 63;
  return (v ^ g) - g;
}
// v 2^(exp - 1086) rounded to FP64, |v| < 2^62: the conversion and a shift of the exponent field where
// every nonzero v gives a normal number, else through fx_to_any (below 2^-1022 the result is 0).
__host__ __device__ __noinline__ static double fx_to_any(long long v, int exp) {
  const double x = (double)v;
  const int f = (int)((fx_bits(x) >> 52) & 0x7ff) + exp - 1086;
  if (v == 0 || f < 1) return 0.0;
  if (f > 2046) return fx_value(v < 0 ? (long long)0xfff0000000000000ull : 0x7ff0000000000000ll);
  return fx_value(fx_bits(x) + ((long long)(exp - 1086) << 52));
}
DGPE_HD double fx_to_normal(long long v, int exp) {   // 64 <= exp <= 2047
  const double x = (double)v;
  return v == 0 ? 0.0 : fx_value(fx_bits(x) + ((long long)(exp - 1086) << 52));
}
DGPE_HD double fx_to(long long v, int exp) {
  return (unsigned)(exp - 64) < 1984u ? fx_to_normal(v, exp) : fx_to_any(v, exp);
}
DGPE_HD cplx<double> fx_to(fxc v, int exp) {
  if ((unsigned)(exp - 64) < 1984u) return {fx_to_normal(v.re, exp), fx_to_normal(v.im, exp)};
  return {fx_to_any(v.re, exp), fx_to_any(v.im, exp)};
}
// The same without the conversion instruction, for the kernels whose FP64 pipe has other work or whose
// chains wait for it: about 20 integer instructions.
DGPE_HD double fx_to_int(long long v, int exp) {
  const long long g = v >> 63;
  const unsigned long long a = (unsigned long long)((v ^ g) - g);
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  const int f = exp - lz - 1;   // the biased exponent less 1; the leading bit, at bit 52 below, adds it
  const unsigned long long m = a << ((lz - 1) & 63);
  unsigned long long b = ((m + 0x1ff + (((unsigned)m >> 10) & 1)) >> 10) + ((unsigned long long)(unsigned)f << 52);
  if ((unsigned)f >= 2046u || a == 0) b = f >= 2046 && a != 0 ? 0x7ff0000000000000ull : 0;
  return fx_value((long long)(b | ((unsigned long long)g & 0x8000000000000000ull)));
}
DGPE_HD cplx<double> fx_to_int(fxc v, int exp) { return {fx_to_int(v.re, exp), fx_to_int(v.im, exp)}; }

// ---- one value with its own exponent: v 2^e ------------------------------------------------
// The recurrences along a line keep every point's precision relative to that point (the tails of a
// cloud as well as its middle), so the running value carries its own exponent: components just
// below 2^62 (fx_up's range) after every step.  One exponent for both components: complex coefficients
// (real time) mix them in every product, and each is good to 2^-56 of the point's magnitude.  (Imaginary
// time, whose real coefficients leave the two parts apart, runs its sweeps in FP64.)
// A long run repeats each rounding at each step, so none of them may lean to one side (the packing's
// cut-off did: the phase of a state turned by 4e-17 a step, coherently).
struct fxv {
  fxc v;
  int e;
};
constexpr int kFxMinExp = kFxMinBiased - 1081;   // (values below 2^-960 lose bits from here on)
DGPE_HD int fx_min(int a, int b) { return a < b ? a : b; }
DGPE_HD long long fx_shl(long long a, int n) { return (long long)((unsigned long long)a << n); }
DGPE_HD fxv fx_norm(fxc s, int e) {   // components of s below 2^62
#ifdef __CUDA_ARCH__
  const int n = __clz(fx_mag(s)) - 2;
#else
  const int mg = fx_mag(s), n = (mg ? __builtin_clz(mg) : 32) - 2;
#endif
  return {{fx_shl(s.re, n), fx_shl(s.im, n)}, e - n};
}
// a w / 8 for a coefficient w of magnitude at most 1 (words of w 2^61): below 2^59.5 for a normalised a
DGPE_HD fxc fx_coef(fxc a, fxw w) { return fx_twiddle<-1>(a, w); }
constexpr int kFxCoefBits = 61;
// a 2^-s, s >= 0, rounded (halves up)
DGPE_HD long long fx_sar(long long a, int s) {
#ifdef __CUDA_ARCH__
  long long h;   // 2^(s - 1), 0 for s = 0 (shl.b64 gives 0 for amounts above 63)
  asm("shl.b64 %0, 1, %1;" : "=l"(h) : "r"(min(s, 63) - 1));
  return (a + h) >> min(s, 63);
#else
  const int k = s < 63 ? s : 63;
  return (a + (k ? 1LL << (k - 1) : 0)) >> k;
#endif
}
// psi + p (p: components below 2^60, exponent ep; key: psi's exponent key), normalised
DGPE_HD fxv fx_forward(double re, double im, int key, fxc p, int ep) {
  const int em = (key >> 20) - 1081;
  int e = em > ep ? em : ep;
  if (e < kFxMinExp) e = kFxMinExp;
  return fx_norm({fx_from<6>(re, e + 1081) + fx_sar(p.re, e - ep), fx_from<6>(im, e + 1081) + fx_sar(p.im, e - ep)}, e);
}
// y + p for an unpacked y (whose low bits are zero: its shift is exact unless p is far above it)
DGPE_HD fxv fx_backward(fxv y, fxc p, int ep) {
  const int e = y.e + 3 > ep ? y.e + 3 : ep;
  const int s = fx_min(e - y.e, 63);
  return fx_norm({(y.v.re >> s) + fx_sar(p.re, e - ep), (y.v.im >> s) + fx_sar(p.im, e - ep)}, e);
}
// 16 bytes of a normalised value: 56 bits of each component, rounded to even, the exponent in the low
// 6 bits of both
DGPE_HD fxc fx_pack(fxv y) {
  const int b = y.e + 1300;
  return {((y.v.re + 31 + ((y.v.re >> 6) & 1)) & ~63ll) | (b & 63), ((y.v.im + 31 + ((y.v.im >> 6) & 1)) & ~63ll) | (b >> 6)};
}
DGPE_HD fxv fx_unpack(fxc q) {
  return {{q.re & ~63ll, q.im & ~63ll}, ((((int)q.im & 63) << 6) | ((int)q.re & 63)) - 1300};
}

// ---- sine, cosine and exponential of the potential step, in fixed point ------------------------
// An angle as theta 2^58, |theta| < 18.
constexpr long long kFxOne58 = 1LL << 58;
// x 2^58 rounded, for |x| < 4; `slow` set otherwise
DGPE_HD long long fx_angle(double x, bool &slow) {
  const long long b = fx_bits(x);
  const int e = (int)(b >> 52) & 0x7ff, s = 1027 - e;
  slow |= e > 1024;
  const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (1ull << 52);
  const int k = s > 63 ? 63 : s < 0 ? 0 : s;
  const long long v = (long long)(((m << 10) + ((1ull << k) >> 1)) >> k);
  const long long g = b >> 63;
  return (v ^ g) - g;
}
// p w / 2^64 + c
DGPE_HD long long fx_horner(long long p, int wh, int wl, long long c) {
  const int ph = fx_hi(p), pl = fx_lo(p);
  const long long mid = fx_mad(ph, wl, fx_mad(pl, wh, kFxHalf));
  return fx_mad(ph, wh, (mid >> 32) + c);
}
// (cos theta, -sin theta) 2^60, the factor e^{-i theta}: up to |theta| = 1/8 the least-squares fits of
// sin_cos(double); beyond (fx_cis_any, out of line: seldom taken, and twice the code) a reduction by
// quarter turns and Taylor series to r^17 and r^18 in u / 2, u = r^2 (r <= pi / 4: the remainders are
// below 2^-63).  Absolute error below 2^-57, so the result's rounding to FP64 dominates.
__host__ __device__ __noinline__ static fxc fx_cis_any(long long th) {
  // quarter turns q and the rest f in [-1/2, 1/2), 2^58
  const long long t = fx_const<1, 0xa2f9836e4e44152aull>(th);   // 2 / pi
  const int q = (int)((t + (kFxOne58 >> 1)) >> 58);
  const long long f = t - ((long long)q << 58);
  const long long f62 = f * 16, r = 2 * (2 * f62 + fx_mul(f62, -1843415740, 1121027178));   // r 2^63, pi/2 = 2 - ...
  const long long u = 2 * fx_mul(r, fx_hi(r), fx_lo(r));   // (r^2 / 2) 2^64
  const int uh = fx_hi(u), ul = fx_lo(u);
  long long ps = fx_horner(1659591, uh, ul, -225704436);   // (-1)^(k+1) 2^k / (2 k + 3)! 2^62
  ps = fx_horner(ps, uh, ul, 23698965738ll);
  ps = fx_horner(ps, uh, ul, -1848519327572ll);
  ps = fx_horner(ps, uh, ul, 101668563016477ll);
  ps = fx_horner(ps, uh, ul, -3660068268593165ll);
  ps = fx_horner(ps, uh, ul, 76861433640456465ll);
  ps = fx_horner(ps, uh, ul, -768614336404564651ll);
  long long pc = fx_horner(-184399, uh, ul, 28213054);     // (-1)^(k+1) 2^k / (2 k + 2)! 2^62
  pc = fx_horner(pc, uh, ul, -3385566534ll);
  pc = fx_horner(pc, uh, ul, 308086554595ll);
  pc = fx_horner(pc, uh, ul, -20333712603295ll);
  pc = fx_horner(pc, uh, ul, 915017067148291ll);
  pc = fx_horner(pc, uh, ul, -25620477880152155ll);
  pc = fx_horner(pc, uh, ul, 384307168202282325ll);
  pc = fx_horner(pc, uh, ul, -2305843009213693952ll);
  const long long ru = fx_mul(r, uh, ul);   // r u 2^62
  const long long s = (r >> 3) + fx_mul(ps, fx_hi(ru), fx_lo(ru));   // 2^60
  const long long c = fx_horner(pc, uh, ul, 1LL << 61) >> 1;
  return (q & 1) ? ((q & 2) ? fxc{s, c} : fxc{-s, -c}) : ((q & 2) ? fxc{-c, s} : fxc{c, -s});
}
DGPE_HD fxc fx_cis(long long th) {
  if (th <= (kFxOne58 >> 3) && th >= -(kFxOne58 >> 3)) {
    const long long x = th * 64;   // theta 2^64
    const int xh = fx_hi(x), xl = fx_lo(x);
    const long long u = fx_mul(x, xh, xl);   // theta^2 2^64
    const int uh = fx_hi(u), ul = fx_lo(u);
    long long ps = fx_horner(12704960496226ll, uh, ul, -915017031897204ll);   // 2^62 times the fits
    ps = fx_horner(ps, uh, ul, 38430716820118072ll);
    ps = fx_horner(ps, uh, ul, -768614336404564608ll);
    long long pc = fx_horner(114337425721235ll, uh, ul, -6405119082289318ll);
    pc = fx_horner(pc, uh, ul, 192153584099929472ll);
    pc = fx_horner(pc, uh, ul, -2305843009213693440ll);
    const long long xu = fx_mul(x, uh, ul);   // theta^3 2^64
    const long long s = (x >> 2) + fx_mul(ps, fx_hi(xu), fx_lo(xu));   // 2^62
    const long long c = fx_horner(pc, uh, ul, 1LL << 62);
    return {c >> 2, -(s >> 2)};
  }
  return fx_cis_any(th);
}
// e^-theta = p 2^(n - 60): 2^f, f in [-1/2, 1/2), by its Taylor series in f / 2 to the 14th power
// (remainder below 2^-66)
DGPE_HD long long fx_exp(long long th, int &n) {
  const long long t = -fx_const<1, 0x71547652b82fe177ull>(th);   // log2 e
  n = (int)((t + (kFxOne58 >> 1)) >> 58);
  const long long w = (t - ((long long)n << 58)) * 32;   // (f / 2) 2^64
  const int wh = fx_hi(w), wl = fx_lo(w);
  long long p = fx_horner(1280465205, wh, wl, 12931245613ll);   // (2 ln 2)^k / k! 2^60
  p = fx_horner(p, wh, wl, 121262985468ll);
  p = fx_horner(p, wh, wl, 1049673046670ll);
  p = fx_horner(p, wh, wl, 8328969544420ll);
  p = fx_horner(p, wh, wl, 60080815287248ll);
  p = fx_horner(p, wh, wl, 390052324203650ll);
  p = fx_horner(p, wh, wl, 2250906215263282ll);
  p = fx_horner(p, wh, wl, 11365799319932687ll);
  p = fx_horner(p, wh, wl, 49192146943818121ll);
  p = fx_horner(p, wh, wl, 177423166116318949ll);
  p = fx_horner(p, wh, wl, 511935043789664227ll);
  p = fx_horner(p, wh, wl, 1107849223398934356ll);
  p = fx_horner(p, wh, wl, 1598288580650331957ll);
  return fx_horner(p, wh, wl, 1152921504606846976ll);
}
// d = c 2^x with |c| < 2^62 (0 for a subnormal d)
struct fxs {
  int h, l, x;
};
DGPE_HD fxs fx_scalar(double d) {
  const long long b = fx_bits(d);
  const int e = (int)(b >> 52) & 0x7ff;
  const long long m = e ? (long long)(((unsigned long long)b & 0xfffffffffffffull) | (1ull << 52)) << 9 : 0;
  const long long c = b < 0 ? -m : m;
  return {fx_hi(c), fx_lo(c), e - 1084};
}
// One point of the potential step: z e^{-i theta} (z e^{-theta}), theta = v + g |z|^2 + dd phi with
// v 2^58 (a sum of two terms below 4) and phi 2^(exp - 1086) in integers, sd = the shift of dd phi
// (not below -1: |theta| < 4 + 4 + 2 + 8).  False, and z as it was, where the interaction or z itself is out of range.
template <bool IMAG>
DGPE_HD bool fx_phase(double &zre, double &zim, long long v, fxs g, fxs dd, int sd, long long phi) {
  const int ka = fx_exponent_bits(zre) >> 20, kb = fx_exponent_bits(zim) >> 20;
  int em = ka > kb ? ka : kb;
  if (em < kFxMinBiased) em = kFxMinBiased;
  // imaginary time: each component under its own exponent, as its factor is real: it keeps its 53 bits
  const int er = !IMAG ? em : ka > kFxMinBiased ? ka : kFxMinBiased, ei = !IMAG ? em : kb > kFxMinBiased ? kb : kFxMinBiased;
  const fxc z = {fx_from<9>(zre, er), fx_from<9>(zim, ei)};   // z.re 2^(er - 1084), ..
  const long long n = (fx_mul(z.re, fx_hi(z.re), fx_lo(z.re)) >> fx_min(2 * (em - er), 63)) +
                      (fx_mul(z.im, fx_hi(z.im), fx_lo(z.im)) >> fx_min(2 * (em - ei), 63));
  const int sg = -(g.x + 2 * (em - 1084) + 186);
  if (em == 0x7ff || sg < 0) return false;
  const long long th = v + fx_sar(fx_mul(n, g.h, g.l), sg) + fx_sar(2 * fx_mul(phi, dd.h, dd.l), sd + 1);
  if constexpr (IMAG) {
    int k;
    const long long p = fx_exp(th, k);
    const int ph = fx_hi(p), pl = fx_lo(p);
    zre = fx_to(fx_mul(z.re, ph, pl), er + 6 + k);
    zim = fx_to(fx_mul(z.im, ph, pl), ei + 6 + k);
  } else {
    const fxc c = fx_cis(th);
    const cplx<double> r = fx_to(fx_twiddle<-1>(z, fx_words(c.re, c.im)), em + 6);
    zre = r.re;
    zim = r.im;
  }
  return true;
}
DGPE_HD int fx_phase_shift(fxs dd, int exp) { return -(64 + dd.x + exp - 1028); }

// The kernels' side of a real type: the exponent key of a value (ordered), the tile's largest key
// -> exponent, values -> integers and back under `exp`, v 2^(exp - 1086).
template <typename R>
struct FxIO;
template <>
struct FxIO<double> {
  static constexpr int kKeyShift = 20, kBad = 0x7ff, kExp = 6;   // exp = emax + kExp
  DGPE_HD static int key(double x) { return fx_exponent_bits(x); }
  DGPE_HD static long long from(double x, int emax) { return fx_from(x, emax); }
  DGPE_HD static double to(long long v, int exp) { return fx_to(v, exp); }
  DGPE_HD static cplx<double> to(fxc v, int exp) { return fx_to(v, exp); }
};
template <typename R>
DGPE_HD int fx_key(cplx<R> z) {
  const int a = FxIO<R>::key(z.re), b = FxIO<R>::key(z.im);
  return a > b ? a : b;
}

// ---- plans: the radices of the staged transforms (dgpe_stages.cuh) ---------------------------
template <int N>
struct FxPlan {
  using S = Stages<N>;
  static constexpr int R1 = S::R1, R2 = S::R2, R3 = S::R3;
  static constexpr int PL = R3 > 1 ? R3 : R2, NBL = N / PL;                     // the last stage
  static constexpr int TWL = R3 > 1 ? R1 * (R2 - 1) : 0;                        // its twiddles
  static constexpr int SLOTS = st_slots<R1, R2, R3, 8>();                       // per line
};
// Threads per CTA of a tile of `lines` lines in `smem` bytes of shared memory: at most 256, enough
// for about 21 warps per SM (what 96 registers a thread allow) with the tiles that fit, and of
// those the fewest thread-elements over the stages (a thread takes whole butterflies, so a stage
// rounds up).
constexpr int fx_threads(int n, int lines, int smem) {
  int best = 256, cost = 0;
  for (int nt = 256; nt >= 64 && nt * (225 * 1024 / (smem + 1024)) >= 640; nt -= 32) {
    int c = 0;
    for (int s = 0; s < 3; ++s) {
      const int r = st_radix(n, s);
      if (r > 1) c += (lines * (n / r) + nt - 1) / nt * r * nt;
    }
    if (!cost || c < cost) {
      cost = c;
      best = nt;
    }
  }
  return best;
}

// Or (or maximum) over the CTA of a per-thread value, with the barrier that orders the shared
// memory written before it.  One slot array per use.
struct FxSlots {
  int w[8];
};
template <int NT>
__device__ __forceinline__ int fx_all_or(int v, FxSlots &s) {
  v = (int)__reduce_or_sync(0xffffffffu, (unsigned)v);
  if ((threadIdx.x & 31) == 0) s.w[threadIdx.x >> 5] = v;
  __syncthreads();
  int r = s.w[0];
#pragma unroll
  for (int k = 1; k < NT / 32; ++k) r |= s.w[k];
  return r;
}
template <int NT>
__device__ __forceinline__ int fx_all_max(int v, FxSlots &s) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) s.w[threadIdx.x >> 5] = v;
  __syncthreads();
  int r = s.w[0];
#pragma unroll
  for (int k = 1; k < NT / 32; ++k) r = max(r, s.w[k]);
  return r;
}

__device__ __forceinline__ fxw fx_ldw(const fxw *p) {
  const int4 q = __ldg(reinterpret_cast<const int4 *>(p));
  return {q.x, q.y, q.z, q.w};
}
// the inputs of a stage: scaled by the tile's shift d, times the twiddles of output index k
template <int DIR, int P, int NS>
__device__ __forceinline__ void fx_inputs(fxc *v, const fxw *__restrict__ tw, int k, int d) {
  v[0] = {fx_scale(v[0].re, d), fx_scale(v[0].im, d)};
#pragma unroll
  for (int r = 1; r < P; ++r) v[r] = fx_twiddle<DIR>(fx_up(v[r], d), fx_ldw(tw + (r - 1) * NS + k));
}
template <int P>
__device__ __forceinline__ int fx_mags(const fxc *v) {
  int m = 0;
#pragma unroll
  for (int r = 0; r < P; ++r) m |= fx_mag(v[r]);
  return m;
}

// Stages after the first of a tile of nl <= L lines (SL slots each), element slots in the layouts
// of dgpe_stages.cuh; the middle stage of three, and the last one, whose outputs go to
// out(line, j, v): elements j + s NBL.
template <int DIR, int N, int NT, int SL>
__device__ __forceinline__ int fx_middle(const fxc *x0, fxc *y0, const fxw *tw, int nl, int d) {
  using F = FxPlan<N>;
  constexpr int R1 = F::R1, R2 = F::R2, NB = N / R2, GAP = st_pad2_gap<R1, R2, 8>();
  int mag = 0;
  for (int it = threadIdx.x; it < nl * NB; it += NT) {
    const int l = it / NB, j = it - l * NB, jb = j / R1, k = j - jb * R1;
    const fxc *x = x0 + l * SL + st_pad1<R1>(j);
    fxc v[R2];
#pragma unroll
    for (int r = 0; r < R2; ++r) v[r] = x[st_pad1<R1>(r * NB)];
    fx_inputs<DIR, R2, R1>(v, tw, k, d);
    fx_bf<DIR, R2>(v);
    mag |= fx_mags<R2>(v);
    fxc *y = y0 + l * SL + jb * (R1 * R2 + GAP) + k;
#pragma unroll
    for (int s = 0; s < R2; ++s) y[s * R1] = v[s];
  }
  return mag;
}
template <int DIR, int N, int NT, int SL, typename Out>
__device__ __forceinline__ void fx_last(const fxc *x0, const fxw *tw, int nl, int d, Out out) {
  using F = FxPlan<N>;
  constexpr int R1 = F::R1, PL = F::PL, NB = F::NBL, GAP = st_pad2_gap<R1, F::R2, 8>();
  for (int it = threadIdx.x; it < nl * NB; it += NT) {
    const int l = it / NB, j = it - l * NB;
    const fxc *x = x0 + l * SL + (F::R3 > 1 ? j : st_pad1<R1>(j));
    fxc v[PL];
#pragma unroll
    for (int r = 0; r < PL; ++r) v[r] = x[F::R3 > 1 ? r * (NB + GAP) : st_pad1<R1>(r * NB)];
    fx_inputs<DIR, PL, NB>(v, tw + F::TWL, j, d);
    fx_bf<DIR, PL>(v);
    out(l, j, v);
  }
}
template <typename R>
__device__ __forceinline__ R fx_nan() { return R(__longlong_as_double(0x7ff8000000000000ll)); }

// ---- K2 / K4: y lines ---------------------------------------------------------------------
template <int N>
struct FxY {
  static constexpr int L = N >= 1024 ? 1 : N <= 32 ? 32 : 1024 / N;
  static constexpr int SL = FxPlan<N>::SLOTS | 1;
  static constexpr size_t smem = (size_t)(FxPlan<N>::R3 > 1 ? 2 : 1) * L * SL * sizeof(fxc);
  static constexpr int NT = fx_threads(N, L, smem);
};
template <typename R, int DIR, int N>
__global__ void __launch_bounds__(FxY<N>::NT) k_ffty_fx(const __grid_constant__ KArgs a) {
  using C = cplx<R>;
  using Y = FxY<N>;
  using F = FxPlan<N>;
  using IO = FxIO<R>;
  constexpr int R1 = F::R1, SL = Y::SL, NT = Y::NT, NB = N / R1, IT = (Y::L * NB + NT - 1) / NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxSlots slot[3];
  fxc *sa = reinterpret_cast<fxc *>(smem_raw), *sb = sa + Y::L * SL;
  const int total = a.nzh * a.nx, l0 = blockIdx.x * Y::L, nl = min(Y::L, total - l0);
  C *g = reinterpret_cast<C *>(a.spec) + (size_t)l0 * N;
  const fxw *tw = reinterpret_cast<const fxw *>(a.tw_st[1]);
  C x[IT][R1];
  int key = 0;
#pragma unroll
  for (int u = 0; u < IT; ++u) {
    const int it = threadIdx.x + u * NT, l = it / NB, j = it - l * NB;
    if (it < nl * NB) {
#pragma unroll
      for (int r = 0; r < R1; ++r) x[u][r] = g[l * N + j + r * NB];
#pragma unroll
      for (int r = 0; r < R1; ++r) key = max(key, fx_key(x[u][r]));
    }
  }
  const int emax = max(fx_all_max<NT>(key, slot[0]) >> IO::kKeyShift, kFxMinBiased);
  if (emax == IO::kBad) {
    for (int e = threadIdx.x; e < nl * N; e += NT) g[e] = {fx_nan<R>(), fx_nan<R>()};
    return;
  }
  int mag = 0;
#pragma unroll
  for (int u = 0; u < IT; ++u) {
    const int it = threadIdx.x + u * NT, l = it / NB, j = it - l * NB;
    if (it < nl * NB) {
      fxc v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = {IO::from(x[u][r].re, emax), IO::from(x[u][r].im, emax)};
      fx_bf<DIR, R1>(v);
      mag |= fx_mags<R1>(v);
      fxc *y = sa + l * SL + st_pad1<R1>(j * R1);
#pragma unroll
      for (int s = 0; s < R1; ++s) y[s] = v[s];
    }
  }
  int d = fx_shift(fx_all_or<NT>(mag, slot[1])), exp = emax + IO::kExp + d;
  if constexpr (F::R3 > 1) {
    mag = fx_middle<DIR, N, NT, SL>(sa, sb, tw, nl, d);
    d = fx_shift(fx_all_or<NT>(mag, slot[2]));
    exp += d;
  }
  fx_last<DIR, N, NT, SL>(F::R3 > 1 ? sb : sa, tw, nl, d, [&](int l, int j, const fxc *v) {
    C *y = g + l * N + j;
#pragma unroll
    for (int s = 0; s < F::PL; ++s) y[s * F::NBL] = IO::to(v[s], exp);
  });
}

// ---- K3: x lines, 4 columns per CTA (64-byte rows) -------------------------------------------
template <int N>
struct FxX {
  using S = Stages<N>;
  static constexpr int B = 4;
  static constexpr int SLA = st_slots<S::R1, S::R2, S::R3, 2>(), SLB = st_slots<S::R3, S::R2, S::R1, 2>();
  static constexpr int SLOTS = SLA > SLB ? SLA : SLB;
  static constexpr size_t smem = 2 * (size_t)SLOTS * B * sizeof(fxc);
  static constexpr int NT = fx_threads(N, B, smem);
};
template <int DIR, int N, int P1, int P2, int P3, int B, int NT>
__device__ __forceinline__ int fx_middle_x(const fxc *x0, fxc *y0, const fxw *tw, int b, int d) {
  constexpr int NB = N / P2, GAP = st_pad2_gap<P1, P2, 2>();
  int mag = 0;
  for (int j = threadIdx.x / B; j < NB; j += NT / B) {
    const int jb = j / P1, k = j - jb * P1;
    const fxc *x = x0 + st_pad1<P1>(j) * B + b;
    fxc v[P2];
#pragma unroll
    for (int r = 0; r < P2; ++r) v[r] = x[st_pad1<P1>(r * NB) * B];
    fx_inputs<DIR, P2, P1>(v, tw, k, d);
    fx_bf<DIR, P2>(v);
    mag |= fx_mags<P2>(v);
    fxc *y = y0 + (jb * (P1 * P2 + GAP) + k) * B + b;
#pragma unroll
    for (int s = 0; s < P2; ++s) y[s * P1 * B] = v[s];
  }
  return mag;
}
template <typename R, int N>
__global__ void __launch_bounds__(FxX<N>::NT) k3_fx(const __grid_constant__ KArgs a) {
  using C = cplx<R>;
  using X = FxX<N>;
  using IO = FxIO<R>;
  constexpr int R1 = X::S::R1, R2 = X::S::R2, R3 = X::S::R3, B = X::B, NT = X::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxSlots slot[6];
  fxc *sa = reinterpret_cast<fxc *>(smem_raw), *sb = sa + X::SLOTS * B;
  const int b = threadIdx.x % B, m = blockIdx.y, jy = blockIdx.x * B + b, ny = a.ny;
  const bool on = jy < ny;
  const size_t col = (size_t)m * a.nx * ny + (on ? jy : 0);
  C *g = reinterpret_cast<C *>(a.spec) + col;
  const fxw *tw = reinterpret_cast<const fxw *>(a.tw_st[0]), *twr = tw + st_table(N);
  int mag = 0, d, exp;
  {
    constexpr int NB = N / R1, IT = (NB * B + NT - 1) / NT;
    C x[IT][R1];
    int key = 0;
#pragma unroll
    for (int u = 0; u < IT; ++u) {
      const int j = threadIdx.x / B + u * (NT / B);
      if (j < NB) {
#pragma unroll
        for (int r = 0; r < R1; ++r) x[u][r] = on ? g[(size_t)(j + r * NB) * ny] : czero<R>();
#pragma unroll
        for (int r = 0; r < R1; ++r) key = max(key, fx_key(x[u][r]));
      }
    }
    const int emax = max(fx_all_max<NT>(key, slot[0]) >> IO::kKeyShift, kFxMinBiased);
    if (emax == IO::kBad) {
      for (int j = threadIdx.x / B; j < N; j += NT / B)
        if (on) g[(size_t)j * ny] = {fx_nan<R>(), fx_nan<R>()};
      return;
    }
    exp = emax + IO::kExp;
#pragma unroll
    for (int u = 0; u < IT; ++u) {
      const int j = threadIdx.x / B + u * (NT / B);
      if (j < NB) {
        fxc v[R1];
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = {IO::from(x[u][r].re, emax), IO::from(x[u][r].im, emax)};
        fx_bf<-1, R1>(v);
        mag |= fx_mags<R1>(v);
        fxc *y = sa + st_pad1<R1>(j * R1) * B + b;
#pragma unroll
        for (int s = 0; s < R1; ++s) y[s * B] = v[s];
      }
    }
  }
  d = fx_shift(fx_all_or<NT>(mag, slot[1]));
  exp += d;
  if constexpr (R3 > 1) {
    mag = fx_middle_x<-1, N, R1, R2, R3, B, NT>(sa, sb, tw, b, d);
    d = fx_shift(fx_all_or<NT>(mag, slot[2]));
    exp += d;
  }
  // the last forward stage and the product by Ut(k) (table: Ut 2^61), in place; then, at the
  // products' range, the first inverse stage on the same elements
  constexpr int P = R3 > 1 ? R3 : R2, NBL = N / P, GAP = st_pad2_gap<R1, R2, 2>();
  fxc *x0 = R3 > 1 ? sb : sa, *y0 = R3 > 1 ? sa : sb;
  mag = 0;
  {
    const long long *ut = reinterpret_cast<const long long *>(a.utab) + col;
    for (int j = threadIdx.x / B; j < NBL; j += NT / B) {
      fxc *x = x0 + (R3 > 1 ? j : st_pad1<R1>(j)) * B + b;
      fxc v[P];
      long long u[P];
#pragma unroll
      for (int s = 0; s < P; ++s) u[s] = __ldg(ut + (size_t)(j + s * NBL) * ny);
#pragma unroll
      for (int r = 0; r < P; ++r) v[r] = x[(R3 > 1 ? r * (NBL + GAP) : st_pad1<R1>(r * NBL)) * B];
      fx_inputs<-1, P, NBL>(v, R3 > 1 ? tw + R1 * (R2 - 1) : tw, j, d);
      fx_bf<-1, P>(v);
#pragma unroll
      for (int s = 0; s < P; ++s) {
        const int uh = fx_hi(u[s]), ul = fx_lo(u[s]);
        v[s] = {fx_mul(v[s].re, uh, ul), fx_mul(v[s].im, uh, ul)};
      }
      mag |= fx_mags<P>(v);
#pragma unroll
      for (int r = 0; r < P; ++r) x[(R3 > 1 ? r * (NBL + GAP) : st_pad1<R1>(r * NBL)) * B] = v[r];
    }
  }
  d = fx_shift(fx_all_or<NT>(mag, slot[3]));
  exp += 3 + d;
  mag = 0;
  for (int j = threadIdx.x / B; j < NBL; j += NT / B) {
    const fxc *x = x0 + (R3 > 1 ? j : st_pad1<R1>(j)) * B + b;
    fxc v[P];
#pragma unroll
    for (int r = 0; r < P; ++r) {
      const fxc t = x[(R3 > 1 ? r * (NBL + GAP) : st_pad1<R1>(r * NBL)) * B];
      v[r] = {fx_scale(t.re, d), fx_scale(t.im, d)};
    }
    fx_bf<+1, P>(v);
    mag |= fx_mags<P>(v);
    fxc *y = y0 + st_pad1<P>(j * P) * B + b;
#pragma unroll
    for (int s = 0; s < P; ++s) y[s * B] = v[s];
  }
  d = fx_shift(fx_all_or<NT>(mag, slot[4]));
  exp += d;
  if constexpr (R3 > 1) {
    mag = fx_middle_x<+1, N, R3, R2, R1, B, NT>(sa, sb, twr, b, d);
    d = fx_shift(fx_all_or<NT>(mag, slot[5]));
    exp += d;
  }
  {
    constexpr int NB = N / R1, GAPR = st_pad2_gap<R3, R2, 2>();
    for (int j = threadIdx.x / B; j < NB; j += NT / B) {
      const fxc *x = sb + (R3 > 1 ? j : st_pad1<P>(j)) * B + b;
      fxc v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = x[(R3 > 1 ? r * (NB + GAPR) : st_pad1<P>(r * NB)) * B];
      fx_inputs<+1, R1, NB>(v, R3 > 1 ? twr + R3 * (R2 - 1) : twr, j, d);
      fx_bf<+1, R1>(v);
      if (on) {
#pragma unroll
        for (int s = 0; s < R1; ++s) g[(size_t)(j + s * NB) * ny] = IO::to(v[s], exp);
      }
    }
  }
}

// ---- z lines: tiles of 2 PZ real lines, packed in pairs ------------------------------------
template <int N>
struct FxZ {
  static constexpr int PZ = N <= 64 ? 16 : N <= 128 ? 8 : 4;
  // line stride: PZ lines by 8 / PZ elements on distinct banks
  static constexpr int SL0 = FxPlan<N>::SLOTS > N ? FxPlan<N>::SLOTS : N;
  static constexpr int SL = PZ == 4 ? SL0 + (10 - SL0 % 8) % 8 : SL0 | 1;
  static constexpr size_t smem = 2 * (size_t)PZ * SL * sizeof(fxc);
  static constexpr size_t smem5 = smem + N * sizeof(long long);   // K5: and the trap's angles along z
  static constexpr int NT = fx_threads(N, PZ, smem);
};

// K1: densities, forward transform, separation of the two real spectra
template <typename R, int N>
__global__ void __launch_bounds__(FxZ<N>::NT) k1_fx(const __grid_constant__ KArgs a) {
  using C = cplx<R>;
  using Z = FxZ<N>;
  using F = FxPlan<N>;
  using IO = FxIO<R>;
  constexpr int R1 = F::R1, SL = Z::SL, NT = Z::NT, PZ = Z::PZ, NB = N / R1, IT = (PZ * NB + NT - 1) / NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxSlots slot[3];
  fxc *sa = reinterpret_cast<fxc *>(smem_raw), *sb = sa + PZ * SL;
  const int i = blockIdx.y, j0 = blockIdx.x * (2 * PZ), np = min(2 * PZ, a.ny - j0) >> 1;
  const C *psi = reinterpret_cast<const C *>(a.psi) + ((size_t)i * a.ny + j0) * N;
  const R s2 = a.unit_scale ? R(1) : scale_sq_of<R>(a.state);
  const bool scaled = (double)s2 != 1.0;
  R x[IT][R1], y[IT][R1];
  int key = 0;
#pragma unroll
  for (int u = 0; u < IT; ++u) {
    const int it = threadIdx.x + u * NT, p = it / NB, j = it - p * NB;
    if (it < np * NB) {
#pragma unroll
      for (int r = 0; r < R1; ++r) {
        const C v = psi[(size_t)(2 * p) * N + j + r * NB], w = psi[(size_t)(2 * p + 1) * N + j + r * NB];
        x[u][r] = v.re * v.re + v.im * v.im;
        y[u][r] = w.re * w.re + w.im * w.im;
      }
      if (scaled) {
#pragma unroll
        for (int r = 0; r < R1; ++r) {
          x[u][r] = x[u][r] * s2;
          y[u][r] = y[u][r] * s2;
        }
      }
#pragma unroll
      for (int r = 0; r < R1; ++r) key = max(key, max(IO::key(x[u][r]), IO::key(y[u][r])));
    }
  }
  const int emax = max(fx_all_max<NT>(key, slot[0]) >> IO::kKeyShift, kFxMinBiased);
  const bool bad = emax == IO::kBad;
  int mag = 0;
#pragma unroll
  for (int u = 0; u < IT; ++u) {
    const int it = threadIdx.x + u * NT, p = it / NB, j = it - p * NB;
    if (it < np * NB) {
      fxc v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = {IO::from(x[u][r], emax), IO::from(y[u][r], emax)};
      fx_bf<-1, R1>(v);
      mag |= fx_mags<R1>(v);
      fxc *q = sa + p * SL + st_pad1<R1>(j * R1);
#pragma unroll
      for (int s = 0; s < R1; ++s) q[s] = v[s];
    }
  }
  const fxw *tw = reinterpret_cast<const fxw *>(a.tw_st[2]);
  int d = fx_shift(fx_all_or<NT>(mag, slot[1])), exp = emax + IO::kExp - 1 + d;   // - 1: the half of the separation
  if constexpr (F::R3 > 1) {
    mag = fx_middle<-1, N, NT, SL>(sa, sb, tw, np, d);
    d = fx_shift(fx_all_or<NT>(mag, slot[2]));
    exp += d;
  }
  fxc *res = F::R3 > 1 ? sa : sb;
  fx_last<-1, N, NT, SL>(F::R3 > 1 ? sb : sa, tw, np, d, [&](int p, int j, const fxc *v) {
#pragma unroll
    for (int s = 0; s < F::PL; ++s) res[p * SL + j + s * F::NBL] = v[s];
  });
  __syncthreads();
  C *spec = reinterpret_cast<C *>(a.spec) + (size_t)i * a.ny + j0;
  const size_t plane = (size_t)a.nx * a.ny;
  const int p = threadIdx.x % PZ;
  if (p < np) {
    for (int m = threadIdx.x / PZ; m <= N / 2; m += NT / PZ) {
      const fxc zm = res[p * SL + m], zc = res[p * SL + (m ? N - m : 0)];
      C o1 = fx_to_int(fxc{zm.re + zc.re, zm.im - zc.im}, exp), o2 = fx_to_int(fxc{zm.im + zc.im, zc.re - zm.re}, exp);
      if (bad) o1 = o2 = {fx_nan<R>(), fx_nan<R>()};
      C *dst = spec + m * plane + 2 * p;
      dst[0] = o1;
      dst[1] = o2;
    }
  }
}

// the potential step of one point in FP64
static __device__ __noinline__ cplx<double> phase_fp64(cplx<double> z, double phi, double v, double dtg, double dtgdd, bool imag) {
  const double theta = fma(dtg, z.re * z.re + z.im * z.im, fma(dtgdd, phi, v));
  if (imag) return scale(z, exp_r(-theta));
  double sn, cs;
  sin_cos(theta, &sn, &cs);
  return {z.re * cs + z.im * sn, z.im * cs - z.re * sn};
}
// K5's phase pass: packing of the two half spectra, inverse transform (Phi), potential step.  Bound by
// integer issue; at 256^3, real time, 1100 us in FP64, 765 with the transform in integers, 295 with
// the angle and its factor too (imaginary time, whose exponential was CUDA's, at 480x480x250: 3060 ->
// 1500, 80 of them for an exponent per component).
template <typename R, int N>
__global__ void __launch_bounds__(FxZ<N>::NT) k5_fx(const __grid_constant__ KArgs a) {
  using C = cplx<R>;
  using Z = FxZ<N>;
  using F = FxPlan<N>;
  using IO = FxIO<R>;
  constexpr int R1 = F::R1, SL = Z::SL, NT = Z::NT, PZ = Z::PZ, M = N / 2 + 1, IT = (PZ * M + NT - 1) / NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxSlots slot[4];
  fxc *sa = reinterpret_cast<fxc *>(smem_raw), *sb = sa + PZ * SL;
  long long *tz = reinterpret_cast<long long *>(sb + PZ * SL);   // dt V_z 2^58
  const int i = blockIdx.y, j0 = blockIdx.x * (2 * PZ), np = min(2 * PZ, a.ny - j0) >> 1;
  int emax;
  {
    const C *spec = reinterpret_cast<const C *>(a.spec) + (size_t)i * a.ny + j0;
    const size_t plane = (size_t)a.nx * a.ny;
    C x1[IT], x2[IT];
    int key = 0;
    const int p = threadIdx.x % PZ;
#pragma unroll
    for (int u = 0; u < IT; ++u) {
      const int m = threadIdx.x / PZ + u * (NT / PZ);
      if (m < M && p < np) {
        const C *src = spec + m * plane + 2 * p;
        x1[u] = src[0];
        x2[u] = src[1];
      }
    }
#pragma unroll
    for (int u = 0; u < IT; ++u) {
      const int m = threadIdx.x / PZ + u * (NT / PZ);
      if (m < M && p < np) key = max(key, max(fx_key(x1[u]), fx_key(x2[u])));
    }
    emax = max(fx_all_max<NT>(key, slot[0]) >> IO::kKeyShift, kFxMinBiased) + 1;   // + 1: the sums of the packing
#pragma unroll
    for (int u = 0; u < IT; ++u) {
      const int m = threadIdx.x / PZ + u * (NT / PZ);
      if (m < M && p < np) {
        const bool end = m == 0 || m == N / 2;   // real bins of a real field's spectrum
        const fxc v1 = {IO::from(x1[u].re, emax), end ? 0 : IO::from(x1[u].im, emax)};
        const fxc v2 = {IO::from(x2[u].re, emax), end ? 0 : IO::from(x2[u].im, emax)};
        sa[p * SL + m] = {v1.re - v2.im, v1.im + v2.re};
        if (!end) sa[p * SL + N - m] = {v1.re + v2.im, v2.re - v1.im};
      }
    }
  }
  const bool bad = emax > IO::kBad;
  __syncthreads();
  const fxw *tw = reinterpret_cast<const fxw *>(a.tw_st[2]);
  int mag = 0;
  {
    constexpr int NB = N / R1;
    for (int it = threadIdx.x; it < np * NB; it += NT) {
      const int p = it / NB, j = it - p * NB;
      fxc v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = sa[p * SL + j + r * NB];
      fx_bf<+1, R1>(v);
      mag |= fx_mags<R1>(v);
      fxc *q = sb + p * SL + st_pad1<R1>(j * R1);
#pragma unroll
      for (int s = 0; s < R1; ++s) q[s] = v[s];
    }
  }
  int d = fx_shift(fx_all_or<NT>(mag, slot[1])), exp = emax + IO::kExp + d;
  if constexpr (F::R3 > 1) {
    mag = fx_middle<+1, N, NT, SL>(sb, sa, tw, np, d);
    d = fx_shift(fx_all_or<NT>(mag, slot[2]));
    exp += d;
  }
  // theta = dt (V + g n + gdd Phi), 1/(nx ny nz) of the inverse transform folded into gdd; the
  // angles and factors in integers (fx_phase), or in FP64 where one of them is out of their range
  // (a CTA whose trap angles or Phi can be, or a point)
  C *psi = reinterpret_cast<C *>(a.psi) + ((size_t)i * a.ny + j0) * N;
  const double *dtv_y = reinterpret_cast<const double *>(a.dtv[1]) + j0, *dtv_z = reinterpret_cast<const double *>(a.dtv[2]);
  const double dtvx = ldg(reinterpret_cast<const double *>(a.dtv[0]) + i);
  const double sr = scale_of<double>(a.state);
  const bool scaled = sr != 1.0;
  const fxs g = fx_scalar(a.dtg), dd = fx_scalar(a.dtgdd_n);
  const int sd = fx_phase_shift(dd, exp);
  bool out = bad || sd < -1;
  if (threadIdx.x < 2 * np) fx_angle(dtvx + ldg(dtv_y + threadIdx.x), out);
  for (int n = threadIdx.x; n < N; n += NT) tz[n] = fx_angle(ldg(dtv_z + n), out);
  const bool slow = __syncthreads_or(out);
  auto phase = [&](auto imag) {
    constexpr bool IMAG = decltype(imag)::value;
    fx_last<+1, N, NT, SL>(F::R3 > 1 ? sa : sb, tw, np, d, [&](int p, int j, const fxc *v) {
#pragma unroll 1   // (the code of a point is long: one copy for both lines)
      for (int h = 0; h < 2; ++h) {
        C *row = psi + (size_t)(2 * p + h) * N + j;
        const double vxy = dtvx + ldg(dtv_y + 2 * p + h);
        bool any = false;
        const long long v0 = fx_angle(vxy, any);
        C w[F::PL];
#pragma unroll
        for (int s = 0; s < F::PL; ++s) w[s] = row[s * F::NBL];
#pragma unroll
        for (int s = 0; s < F::PL; ++s) {
          C z = w[s];
          if (scaled) z = scale(z, sr);
          const long long phi = h ? v[s].im : v[s].re;
          if (slow || !fx_phase<IMAG>(z.re, z.im, v0 + tz[j + s * F::NBL], g, dd, sd, phi))
            z = phase_fp64(z, bad ? fx_nan<double>() : IO::to(phi, exp), vxy + ldg(dtv_z + j + s * F::NBL), a.dtg, a.dtgdd_n, IMAG);
          row[s * F::NBL] = z;
        }
      }
    });
  };
  if (a.imag) phase(std::true_type{});
  else phase(std::false_type{});
}

// ---- Crank-Nicolson sweeps ------------------------------------------------------------------
// Coefficients of the sweeps, behind the FP64 table of the same axis and direction (at fx_cn_offset).
// Imaginary time: the FP64 values alpha_s for s < h + 2, then 2 beta_s (h = m/2).  Real time: a header {ka, kb}, then alpha_s 2^ka for s < h + 2, then 2 beta_s 2^kb for
// s < h + 2, as words of kFxCoefBits bits (the largest powers of two that keep every magnitude at most 1).
__host__ __device__ constexpr size_t fx_cn_offset(int chunk) { return ((size_t)4 * kWarp * chunk + 11 * kWarp) * 16; }
__global__ inline void k_fx_cn_tables(CnJobs jobs) {
  const CnJob &jb = jobs.job[blockIdx.x];
  const int m = jb.m, chunk = jb.chunk, mp = kWarp * chunk, n = m / 2 + 2;
  const double *tab = static_cast<const double *>(jb.tab);
  fxw *out = reinterpret_cast<fxw *>(static_cast<char *>(jb.tab) + fx_cn_offset(chunk));
  // (entries past m are the padding of the FP64 table, and within it: n <= m + 1 <= 32 chunk)
  auto at = [&](int q, int i) { return q * mp + (i % chunk) * kWarp + i / chunk; };
  auto get = [&](int q, int i) {
    if (i >= m) return Z64{0.0, 0.0};
    const double f = q ? 2.0 : 1.0;
    return Z64{f * tab[2 * at(q, i)], f * tab[2 * at(q, i) + 1]};
  };
  if (jobs.imag) {
    for (int q = 0; q < 2; ++q)
      for (int i = threadIdx.x; i < n; i += kWarp) reinterpret_cast<double *>(out)[q * n + i] = i < m ? (q ? 2.0 : 1.0) * tab[at(q, i)] : 0.0;
    return;
  }
  double mx[2] = {0.0, 0.0};
  for (int q = 0; q < 2; ++q) {
    for (int i = threadIdx.x; i < n; i += kWarp) {
      const Z64 z = get(q, i);
      mx[q] = fmax(mx[q], sqrt(z.re * z.re + z.im * z.im));
    }
    for (int o = kWarp / 2; o > 0; o >>= 1) mx[q] = fmax(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], o));
  }
  int k[2];
  for (int q = 0; q < 2; ++q) {
    int e = 0;
    frexp(mx[q] * (1.0 + 1e-15), &e);
    k[q] = mx[q] > 0.0 ? min(-e, 60) : 60;
  }
  if (threadIdx.x == 0) out[0] = {k[0], k[1], 0, 0};
  for (int q = 0; q < 2; ++q)
    for (int i = threadIdx.x; i < n; i += kWarp) {
      const Z64 z = get(q, i);
      const long long re = __double2ll_rn(ldexp(z.re, kFxCoefBits + k[q])), im = __double2ll_rn(ldexp(z.im, kFxCoefBits + k[q]));
      out[1 + q * n + i] = fx_words(re, im);
    }
}

// The sweep along AXIS: two threads per line, the twisted ("burn at both ends") factorization of the
// Cayley form psi' = 2 (1 - c D)^-1 psi - psi.  The matrix tridiag(-c, 1 + 2c, -c) reads the same from
// either end, so the top thread eliminates points 0 .. h-1 downwards and the bottom thread points
// m-1 .. h+1 upwards with the same table entry s at their s-th step; they meet at h = m/2,
//   gamma x_h = psi_h + alpha_h y_{h-1} + alpha_{m-1-h} z_{h+1}   (in FP64),
// and substitute back away from it:
//   y_i = psi_i + alpha_i y_{i-1},  x_i = y_i + alpha_{i+2} x_{i+1}  (x = chi / beta),
//   psi'_i = 2 beta_i x_i - psi_i.
// Real time: the running values are integers with their own exponent (fxv).  In FP64 arithmetic a sweep is
// 12 FP64 instructions per point, 0.32 ms of that pipe at 256^3; this is about 330 integer ones (0.14 ms)
// and two FP64 subtractions.  Imaginary time: FP64 arithmetic.  Its real coefficients make a sweep 6 FP64
// instructions per point, no more than the integers take (us at 256^3, integers -> FP64: y 254 -> 238, x with
// its sums 341 -> 381, z 296 -> 272; a step at 64^3 104 -> 98), and each component of psi keeps its own 53 bits.  Persistent CTAs: y waits for the way back in a scratch of the CTA's own
// (packed, 16 bytes a point), so few enough lines are under way for much of it and of their psi to
// stay in L2.  psi and y come through shared memory by cp.async, two chunks of four points ahead;
// along z, where a thread's points are consecutive, the lanes of a warp copy each other's chunks as
// segments of 64 bytes, both ways.  Bound by the latency of the recurrence (a warp issues every 4 to 5
// cycles; half of the issue slots at 12 warps per SM; DRAM 1.1 GB, 165 us).  Measured at 256^3, real
// time, us, FP64 arithmetic (without these pipelines) -> now: y 411 -> 292, x with its sums 515 -> 378, z
// 410 -> 325; errors against extended precision 0.7 of the FP64 sweep's (1.1e-16 and 1.6e-16).
constexpr int kFxcThreads = 128, kFxcChunk = 4, kFxcStages = 3;
template <int AXIS>
constexpr size_t fx_cn_smem(bool reduce, int nx) {
  const size_t row = AXIS == 2 ? kFxcChunk + 1 : kFxcChunk;
  return (size_t)kFxcStages * kFxcThreads * (row + kFxcChunk) * 16 + (reduce ? (size_t)nx * 8 : 0);
}
template <bool CPLX, int AXIS, bool RED>
__global__ void __launch_bounds__(kFxcThreads, 4) k_cn_fx(const __grid_constant__ KArgs a, int renorm) {
  using C = cplx<double>;
  constexpr int K = kFxcChunk, S = kFxcStages, T = kFxcThreads, ROW = AXIS == 2 ? K + 1 : K;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C *pbuf = reinterpret_cast<C *>(smem_raw);                       // psi: [stage][step][thread], z: [stage][thread][step]
  fxc *ybuf = reinterpret_cast<fxc *>(pbuf + S * T * ROW);         // y: [stage][step][thread]
  double *wxtab = reinterpret_cast<double *>(ybuf + S * T * K);    // quadrature weights along x
  const int tid = threadIdx.x, lane = tid & (kWarp - 1);
  const bool bottom = lane >= kWarp / 2;
  if constexpr (RED) {
    for (int n = tid; n < a.nx; n += T) wxtab[n] = quad_weight(n, a.nx, a.simpson);
    __syncthreads();
  }
  const int nfixed = AXIS == 0 ? a.ny : a.nx;
  const int nlines = AXIS == 2 ? a.nx * a.ny : nfixed * a.nz;
  const int ntiles = (nlines + T / 2 - 1) / (T / 2);
  const ptrdiff_t stride = AXIS == 2 ? 1 : AXIS == 1 ? (ptrdiff_t)a.nz : (ptrdiff_t)a.ny * a.nz;
  const int m = a.cn[AXIS].m, lc = a.cn[AXIS].lchunk, chunk = 1 << lc, mp = kWarp << lc, h = m / 2;
  using Coef = typename std::conditional<CPLX, C, double>::type;
  const Coef *tab = reinterpret_cast<const Coef *>(a.cn[AXIS].tab);
  const fxw *ft = reinterpret_cast<const fxw *>(static_cast<const char *>(a.cn[AXIS].tab) + fx_cn_offset(chunk));
  const fxw head = CPLX ? fx_ldw(ft) : fxw{0, 0, 0, 0};
  const int ka = head.rh, kb = head.rl;
  const fxw *fal = ft + 1, *fbe = ft + 1 + h + 2;
  const double *dal = reinterpret_cast<const double *>(ft), *dbe = dal + h + 2;   // imaginary time
  const double r = a.cn_r[AXIS];
  fxc *scratch = reinterpret_cast<fxc *>(a.ybuf) + (size_t)blockIdx.x * h * T + tid;   // y of step s at s T
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int line0 = tile * (T / 2) + tid / kWarp * (kWarp / 2);   // the warp's first line
    const int line = line0 + (lane & 15);
    const bool active = line < nlines;
    const int ln = active ? line : 0, k = ln % a.nz, fixed = ln / a.nz;
    C *p = reinterpret_cast<C *>(a.psi) +
           (AXIS == 2 ? (size_t)ln * a.nz : (AXIS == 1 ? (size_t)fixed * a.ny * a.nz : (size_t)fixed * a.nz) + k) + stride;
    const int nf = active ? (bottom ? m - 1 - h : h) : 0;   // elimination steps of this half
    // psi of this half's points b + d s for the steps s of chunk c, to stage c % S (z: lane by lane
    // of the warp's rows, whose b and d follow from the row)
    auto load_psi = [&](int c, bool back) {
      if constexpr (AXIS == 2) {
#pragma unroll
        for (int q = 0; q < K; ++q) {
          const int row = q * (kWarp / K) + lane / K, s = c * K + lane % K, l = line0 + (row & 15);
          const bool bt = row >= kWarp / 2;
          const int len = bt ? m - 1 - h : h;
          const int i = back ? (bt ? h + 1 + s : h - 1 - s) : (bt ? m - 1 - s : s);
          if (l < nlines && s < len)
            cp_async(pbuf + ((c % S) * T + (tid - lane) + row) * ROW + lane % K, reinterpret_cast<C *>(a.psi) + (size_t)l * a.nz + 1 + i);
        }
      } else {
#pragma unroll
        for (int e = 0; e < K; ++e) {
          const int s = c * K + e;
          const int i = back ? (bottom ? h + 1 + s : h - 1 - s) : (bottom ? m - 1 - s : s);
          if (s < nf) cp_async(pbuf + ((c % S) * K + e) * T + tid, p + i * stride);
        }
      }
    };
    auto psi_at = [&](int c, int e) -> C & { return AXIS == 2 ? pbuf[((c % S) * T + tid) * ROW + e] : pbuf[((c % S) * K + e) * T + tid]; };
    const int nc = (h + K - 1) / K, nwhole = line0 + 15 < nlines ? (m - 1 - h) / K : 0;
    // elimination
    fxv y = {{0, 0}, kFxMinExp};
    C yf = czero<double>();   // imaginary time: in FP64
    int kmax = 0;
#pragma unroll
    for (int c = 0; c < S - 1; ++c) {
      load_psi(c, false);
      cp_async_commit();
    }
    for (int c = 0; c < nc; ++c) {
      load_psi(c + S - 1, false);
      cp_async_commit();
      cp_async_wait_group<S - 1>();
      if constexpr (AXIS == 2) __syncwarp();
      // (whole chunks of whole warps without conditions: straight-line code, so that the parts off the
      // recurrence fill its latency)
      auto steps = [&](auto whole) {
        C vs[K];
#pragma unroll
        for (int e = 0; e < K; ++e) vs[e] = psi_at(c, e);   // (past the half's end: not used)
#pragma unroll
        for (int e = 0; e < K; ++e) {
          const int s = c * K + e;
          if (decltype(whole)::value || s < nf) {
            const C v = vs[e];
            if constexpr (CPLX) {
              const int key = fx_key(v);
              kmax = max(kmax, key);
              const fxc t = fx_coef(y.v, fx_ldw(fal + s));
              y = fx_forward(v.re, v.im, key, t, y.e + 3 - ka);
              scratch[(size_t)s * T] = fx_pack(y);
            } else {
              yf = cfma(__ldg(dal + s), yf, v);
              reinterpret_cast<C *>(scratch)[(size_t)s * T] = yf;
            }
          }
        }
      };
      if (c < nwhole) steps(std::true_type{});
      else steps(std::false_type{});
      if constexpr (AXIS == 2) __syncwarp();
    }
    cp_async_wait_all();
    __threadfence();   // the scratch is read back through cp.async
    // y and psi of the way back, step j: the half's step nf - 1 - j
    auto load_y = [&](int c) {
#pragma unroll
      for (int e = 0; e < K; ++e) {
        const int j = c * K + e;
        if (j < nf) cp_async(ybuf + ((c % S) * K + e) * T + tid, scratch + (size_t)(nf - 1 - j) * T);
      }
    };
    if constexpr (AXIS == 2) __syncwarp();
#pragma unroll
    for (int c = 0; c < S - 1; ++c) {
      load_psi(c, true);
      load_y(c);
      cp_async_commit();
    }
    // the twist point, in FP64: gamma x_h = psi_h + alpha_h y_{h-1} + alpha_{m-1-h} z_{h+1}
    const C yd = CPLX ? fx_to(y.v, y.e + 1086) : yf;
    const C yt = shfl_xor(yd, kWarp / 2);
    C xh = czero<double>(), ph = czero<double>();
    if (bottom && active) {
      auto slot = [&](int s) { return ((s & (chunk - 1)) << 5) + (s >> lc); };
      ph = p[h * stride];
      if constexpr (CPLX) kmax = max(kmax, fx_key(ph));
      xh = mul(ldg(tab + 4 * mp + 10 * kWarp), cfma(ldg(tab + slot(m - 1 - h)), yd, cfma(ldg(tab + slot(h)), yt, ph)));
    }
    const C xt = shfl_xor(xh, kWarp / 2);
    if (!bottom) xh = xt;
    if constexpr (CPLX) kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, kWarp / 2));
    double s0 = 0.0;
    auto add = [&](int i, C o) {
      if constexpr (RED) {
        if (a.simpson) s0 = fma(wxtab[i + 1], fma(o.re, o.re, o.im * o.im), s0);
        else s0 = fma(o.im, o.im, fma(o.re, o.re, s0));
      }
    };
    if (bottom && active) {
      const C o = {twice_minus(xh.re, ph.re), twice_minus(xh.im, ph.im)};
      p[h * stride] = o;
      add(h, o);
    }
    // c x_h starts both halves' way back
    const C cx = CPLX ? C{-r * xh.im, r * xh.re} : C{r * xh.re, r * xh.im};
    const int ex = max(fx_key(cx) >> 20, kFxMinBiased);
    fxc t = {fx_from<6>(cx.re, ex), fx_from<6>(cx.im, ex)};
    int et = ex - 1081;
    C xf = xh;
    double ap = r;   // imaginary time: x_i = y_i + ap x of the point before
    for (int c = 0; c < nc; ++c) {
      load_psi(c + S - 1, true);
      load_y(c + S - 1);
      cp_async_commit();
      cp_async_wait_group<S - 1>();
      if constexpr (AXIS == 2) __syncwarp();
      auto steps = [&](auto whole) {
        C vs[K];
        fxc ys[K];
#pragma unroll
        for (int e = 0; e < K; ++e) {
          vs[e] = psi_at(c, e);
          ys[e] = ybuf[((c % S) * K + e) * T + tid];
        }
#pragma unroll
        for (int e = 0; e < K; ++e) {
          const int j = c * K + e;
          if (decltype(whole)::value || j < nf) {
            const int q = nf - 1 - j, i = bottom ? h + 1 + j : h - 1 - j;
            const C v = vs[e];
            C o;
            if constexpr (!CPLX) {
              xf = cfma(ap, xf, C{__longlong_as_double(ys[e].re), __longlong_as_double(ys[e].im)});
              o = cfma(__ldg(dbe + q), xf, C{-v.re, -v.im});
              ap = __ldg(dal + q + 1);
            } else {
              const fxv x = fx_backward(fx_unpack(ys[e]), t, et);
              const fxc b = fx_coef(x.v, fx_ldw(fbe + q));
              t = fx_coef(x.v, fx_ldw(fal + q + 1));   // (q = 0: the last point, unused)
              et = x.e + 3 - ka;
              const int eb = x.e + 3 - kb;
              if constexpr (RED) {
                // the difference in integers: the FP64 pipe has the sums to do
                const int ev = (fx_key(v) >> 20) - 1081, ed = max(max(eb, ev), kFxMinExp);
                o = fx_to_int(fxc{fx_sar(b.re, ed - eb) - fx_from<6>(v.re, ed + 1081), fx_sar(b.im, ed - eb) - fx_from<6>(v.im, ed + 1081)}, ed + 1086);
              } else {
                o = fx_to_int(b, eb + 1086) - v;
              }
            }
            if constexpr (AXIS == 2) psi_at(c, e) = o;
            else p[i * stride] = o;
            add(i, o);
          }
        }
      };
      if (c < nwhole) steps(std::true_type{});
      else steps(std::false_type{});
      if constexpr (AXIS == 2) {
        __syncwarp();
#pragma unroll
        for (int q = 0; q < K; ++q) {
          const int row = q * (kWarp / K) + lane / K, s = c * K + lane % K, l = line0 + (row & 15);
          const bool bt = row >= kWarp / 2;
          if (l < nlines && s < (bt ? m - 1 - h : h))
            reinterpret_cast<C *>(a.psi)[(size_t)l * a.nz + 1 + (bt ? h + 1 + s : h - 1 - s)] = pbuf[((c % S) * T + (tid - lane) + row) * ROW + lane % K];
        }
        __syncwarp();
      }
    }
    cp_async_wait_all();
    if (kmax >= 0x7ff00000) {   // a value that is not finite: so is its line
      const C nan = {fx_nan<double>(), fx_nan<double>()};
      for (int s = 0; s < nf; ++s) p[(bottom ? m - 1 - s : s) * stride] = nan;
      if (bottom && active) p[h * stride] = nan;
      s0 = fx_nan<double>();
    }
    if (active) {
      // the walls (grid points 0 and N-1)
      if (!bottom) p[-stride] = czero<double>();
      else p[m * stride] = czero<double>();
      if constexpr (RED) {
        const double wyz = quad_weight_r<double>(fixed, a.ny, a.simpson) * quad_weight_r<double>(k, a.nz, a.simpson);
        const double yv = (fixed - a.ny / 2) * a.hy, zv = (k - a.nz / 2) * a.hz, tt = wyz * s0;
        acc[0] += tt;
        acc[2] = fma(yv * yv, tt, acc[2]);
        acc[3] = fma(zv * zv, tt, acc[3]);
      }
    }
  }
  if constexpr (RED) finish_sweep_sums(a, acc, 1.0, 1.0, 1.0, renorm);
}

// ---- set-up ---------------------------------------------------------------------------------
// The twiddles of the plan of length n and of its radices in reverse order (layout: dgpe_stages.cuh)
__global__ inline void k_fx_twiddles(fxw *tw, int n, int r1, int r2, int r3) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * n) return;
  const bool rev = t >= n;
  int e = rev ? t - n : t;
  const int nst = r3 > 1 ? 3 : 2;
  const int p1 = rev ? (nst == 3 ? r3 : r2) : r1, p2 = rev ? (nst == 3 ? r2 : r1) : r2, p3 = nst == 3 ? (rev ? r1 : r3) : 1;
  int ns = p1, p = p2;
  if (e >= p1 * (p2 - 1)) {
    e -= p1 * (p2 - 1);
    ns = p1 * p2;
    p = p3;
    if (e >= ns * (p - 1)) return;
  }
  const int r = e / ns + 1, k = e % ns;
  double s, c;
  sincospi(2.0 * (double)(r * k) / (double)(ns * p), &s, &c);
  const long long qc = __double2ll_rn(c * 1152921504606846976.0), qs = __double2ll_rn(-s * 1152921504606846976.0);   // 2^60
  tw[t] = fx_words(qc, qs);
}

// One translation unit's lengths: every kFxParts-th of the list.
constexpr int kFxParts = 8;
constexpr int fx_index(int n) {
  int i = 0, at = -1;
#define DGPE_AT(m) \
  if (m == n) at = i; \
  ++i;
  DGPE_STAGE_ALL(DGPE_AT)
#undef DGPE_AT
  return at;
}
template <int PART>
struct FxLaunch {
  template <typename F>
  static bool with(int n, F &&f) {
    switch (n) {
#define DGPE_CASE(m) \
  case m: \
    if constexpr (fx_index(m) % kFxParts == PART) { \
      f(std::integral_constant<int, m>{}); \
      return true; \
    } \
    break;
      DGPE_STAGE_ALL(DGPE_CASE)
#undef DGPE_CASE
      default: break;
    }
    return false;
  }
  // kernel `which` (kK1DensityR2Cz .. kK4IfftY, kK5C2RzPhaseCnz: the phase pass)
  template <typename R>
  static bool run(int which, const KArgs &a, cudaStream_t st) {
    const int n = which == kK3FftXDipolar ? a.nx : which == kK2FftY || which == kK4IfftY ? a.ny : a.nz;
    return with(n, [&](auto len) {
      constexpr int N = decltype(len)::value;
      using Y = FxY<N>;
      using X = FxX<N>;
      using Z = FxZ<N>;
      const unsigned gy = (a.nzh * a.nx + Y::L - 1) / Y::L;
      const dim3 gz((a.ny + 2 * Z::PZ - 1) / (2 * Z::PZ), a.nx);
      if (which == kK2FftY) k_ffty_fx<R, -1, N><<<gy, Y::NT, Y::smem, st>>>(a);
      else if (which == kK4IfftY) k_ffty_fx<R, +1, N><<<gy, Y::NT, Y::smem, st>>>(a);
      else if (which == kK3FftXDipolar) k3_fx<R, N><<<dim3((a.ny + X::B - 1) / X::B, a.nzh), X::NT, X::smem, st>>>(a);
      else if constexpr (N % 2 == 0) {
        if (which == kK1DensityR2Cz) k1_fx<R, N><<<gz, Z::NT, Z::smem, st>>>(a);
        else k5_fx<R, N><<<gz, Z::NT, Z::smem5, st>>>(a);
      }
    });
  }
  template <typename R>
  static cudaError_t init(int nx, int ny, int nz) {
    cudaError_t e = cudaSuccess;
    auto opt = [&](auto k, size_t sm) {
      if (e == cudaSuccess && sm > 40 * 1024) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    };
    with(nx, [&](auto len) { opt(k3_fx<R, decltype(len)::value>, FxX<decltype(len)::value>::smem); });
    with(ny, [&](auto len) {
      opt(k_ffty_fx<R, -1, decltype(len)::value>, FxY<decltype(len)::value>::smem);
      opt(k_ffty_fx<R, +1, decltype(len)::value>, FxY<decltype(len)::value>::smem);
    });
    with(nz, [&](auto len) {
      opt(k1_fx<R, decltype(len)::value>, FxZ<decltype(len)::value>::smem);
      opt(k5_fx<R, decltype(len)::value>, FxZ<decltype(len)::value>::smem5);
    });
    return e;
  }
};

}  // namespace dgpe
