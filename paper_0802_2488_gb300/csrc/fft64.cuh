// Double-precision transforms on the integer pipes (fft_seq<double, ...>).
//
// GB300 issues one FP64 warp instruction per 19 clocks and SM (64 on its
// scheduler), a 64-bit integer add (two instructions) about every 1.5 and a
// 32 x 32 + 64 bit multiply-add every 2.1 clocks (measured).  A transform is
// additions and multiplications by numbers of modulus 1, so it is done in
// 64-bit fixed point on a block exponent: each sequence is read as doubles,
// its largest exponent found, and each number x of it held as the integer
// x 2^B of a common B.  (One B for all sequences of a call is not enough:
// components that do not couple, or rows, far below the largest would lose
// bits that FP64 butterflies, whose error follows the sequence's own norm, keep.
// A component 1e-10 of the others: 6e-8 of its norm against 1e-16.)  A stage of radix R
// multiplies by its twiddles scaled by 2^64 / R and keeps the upper 64 bits
// of the 128-bit product, which divides by R, so no sum can overflow
// whatever the data are:
//
//   |z| <= 2^62.5 before a stage (|re|, |im| <= 2^62 at the first), at most
//   2^62.5 / R after the multiplication, and a sum of R such numbers has
//   modulus <= 2^62.5 again.
//
// The last stage's integers are rounded to doubles.  Precision: an input is
// held to 2^-60 of the sequence's largest number, each stage rounds to the last
// bit of numbers whose RMS falls by sqrt(R) a stage from 2^60 or so, which
// leaves an error of 2^-55 (N = 512) to 2^-53 (N = 4096) of the output's RMS,
// below that of the FP64 butterflies it replaces (their 53 bits are rounded at
// every operation).  A NaN or infinity in a sequence makes every output of it
// NaN.
//
// Measured (8 x L = 512, CUDA events): FP64 butterflies 581 us (column pass) and
// 787 us (row pass); 207 and 332 us with the transforms and the twists in fixed
// point, the pixel step of local_step64 and the CTA shapes this left room for
// (Cfg in passes.cuh); what is left on the FP64 pipe is the Green operator and
// the pixel step.  L = 4096: 5.69 -> 2.88 ms and 7.83 -> 4.32 ms.  (One block
// exponent for all sequences of a call instead of one each: 205 and 330 us, 2.86
// and 4.25 ms.)
// Against long double: projection at L = 64, 256 1.8e-16, 1.8e-16 relative
// (FP64 butterflies 3.2e-16, 3.6e-16), 20 iterations at L = 256 7.0e-16
// (1.25e-15).
#pragma once
#include "common.cuh"

#ifdef __CUDACC__
#define EPFFT_HD __host__ __device__ __forceinline__
#else
#define EPFFT_HD inline
#endif

namespace epfft {

using i64 = long long;

// High word of a for the balanced split a = hi 2^32 + lo with lo the signed
// low word.
EPFFT_HD int bal_lo(i64 a) { return (int)(unsigned)(unsigned long long)a; }
EPFFT_HD int bal_hi(i64 a) { return (int)(a >> 32) + (int)(((unsigned)(unsigned long long)a) >> 31); }

// A twiddle is stored as balanced words: re / im = hi 2^32 + lo, in the
// 16 bytes of a complex double.  conj for the inverse kernel is a change of
// sign of the imaginary words (the host keeps lo above -2^31).
struct Tw64 {
  int rl, rh, il, ih;
};

// Products keep the words' cross terms in one 64-bit sum (the lowest words'
// product is below the last bit kept); its upper half joins the product of
// the high words.  Bounds: |a| <= 2^62.5, |w| <= 2^62: the four cross terms
// of a complex product stay below 2^62.8 and the high ones below 2^62.5.
// a w / 2^64 (complex).
template <bool INV>
EPFFT_HD void cmul_hi(i64& re, i64& im, const Tw64& w) {
  const int rl = bal_lo(re), rh = bal_hi(re), il = bal_lo(im), ih = bal_hi(im);
  const int wl = INV ? -w.il : w.il, wh = INV ? -w.ih : w.ih;  // imaginary part of w
  i64 m = 0x80000000ll;
  m += (i64)rh * w.rl;
  m += (i64)rl * w.rh;
  m += (i64)ih * -wl;
  m += (i64)il * -wh;
  i64 n = 0x80000000ll;
  n += (i64)rh * wl;
  n += (i64)rl * wh;
  n += (i64)ih * w.rl;
  n += (i64)il * w.rh;
  re = (m >> 32) + (i64)rh * w.rh + (i64)ih * -wh;
  im = (n >> 32) + (i64)rh * wh + (i64)ih * w.rh;
}
// a w / 2^63 (complex) with w of scale 2^62, i.e. half the product.
EPFFT_HD void cmul_half(i64& re, i64& im, const Tw64& w) {
  const int rl = bal_lo(re), rh = bal_hi(re), il = bal_lo(im), ih = bal_hi(im);
  i64 m = 0x40000000ll, n = 0x40000000ll;
  m += (i64)rh * w.rl;
  m += (i64)rl * w.rh;
  m += (i64)ih * -w.il;
  m += (i64)il * -w.ih;
  n += (i64)rh * w.il;
  n += (i64)rl * w.ih;
  n += (i64)ih * w.rl;
  n += (i64)il * w.rh;
  const i64 p = (i64)rh * w.rh + (i64)ih * -w.ih, q = (i64)rh * w.ih + (i64)ih * w.rh;
  re = (m >> 31) + (i64)((unsigned long long)p << 1);
  im = (n >> 31) + (i64)((unsigned long long)q << 1);
}
// a w / 2^S (complex), for products of twiddles of scale 2^S (S = 64 - log2 R).
template <int S>
EPFFT_HD Tw64 tw_mul(const Tw64& a, const Tw64& w) {
  i64 m = (i64)a.rh * w.rl + (i64)a.rl * w.rh - (i64)a.ih * w.il - (i64)a.il * w.ih;
  i64 n = (i64)a.rh * w.il + (i64)a.rl * w.ih + (i64)a.ih * w.rl + (i64)a.il * w.rh;
  i64 p = (i64)a.rh * w.rh - (i64)a.ih * w.ih;
  i64 q = (i64)a.rh * w.ih + (i64)a.ih * w.rh;
  // odd, so that no low word is -2^31 (the words change sign in cmul_hi)
  const i64 re = ((i64)((unsigned long long)p << (64 - S)) + (m >> (S - 32))) | 1;
  const i64 im = ((i64)((unsigned long long)q << (64 - S)) + (n >> (S - 32))) | 1;
  return Tw64{bal_lo(re), bal_hi(re), bal_lo(im), bal_hi(im)};
}
// a c / 2^64 for a constant c (its balanced words), real.
EPFFT_HD i64 mul_hi(i64 a, int cl, int ch) {
  const int al = bal_lo(a), ah = bal_hi(a);
  i64 m = 0x80000000ll;
  m += (i64)ah * cl;
  m += (i64)al * ch;
  return (m >> 32) + (i64)ah * ch;
}
// a c for c = cos(pi/4), cos(pi/8), sin(pi/8) of the small butterflies; the
// ones above 1/2 as a - a (1 - c), so that the constant fits 2^63.
#define EPFFT_C64(name, num, sub)                                   \
  EPFFT_HD i64 name(i64 a) {                                        \
    constexpr i64 C = (i64)((num) * 18446744073709551616.0L);       \
    constexpr int CL = (int)(unsigned)(unsigned long long)C;        \
    constexpr int CH = (int)(C >> 32) + (CL < 0 ? 1 : 0);           \
    const i64 p = mul_hi(a, CL, CH);                                \
    return (sub) ? a - p : p;                                       \
  }
EPFFT_C64(mul_cos4, 1.0L - 0.70710678118654752440084436210484904L, true)
EPFFT_C64(mul_cos8, 1.0L - 0.92387953251128675612818318939678828682L, true)
EPFFT_C64(mul_sin8, 0.38268343236508977172845998403039886676L, false)
#undef EPFFT_C64

// (a + 2^(k-1)) >> k
template <int k>
EPFFT_HD i64 rshift(i64 a) { return k == 0 ? a : (a + ((i64)1 << (k > 0 ? k - 1 : 0))) >> k; }

EPFFT_HD int hi_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  union { double d; unsigned long long u; } c{x};
  return (int)(c.u >> 32);
#endif
}
EPFFT_HD unsigned lo_word(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  union { double d; unsigned long long u; } c{x};
  return (unsigned)c.u;
#endif
}
EPFFT_HD double make_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((i64)b);
#else
  union { unsigned long long u; double d; } c{b};
  return c.d;
#endif
}

// Block exponent of the largest high word mx (sign bit cleared): the biased
// exponent, at least 1, or FIX_NAN for an infinity or a NaN (far above any
// exponent, so that the shifts between stages leave it one).  to_fixed takes
// exponents from FIX_LOW on: numbers of a sequence below that (2^-957) are
// converted as 2^64 times themselves (lift64, exact) on an exponent 64 larger;
// the callers write this as a loop, which the compiler leaves a branch (as
// predicated FP64 instructions it cost every sequence 5 %).  Results below the
// normal range (2^-1022) become zero.
constexpr int FIX_NAN = 1 << 20, FIX_LOW = 65;
EPFFT_HD int block_exp(unsigned mx) {
  const int e = (int)(mx >> 20);
  return e < 1 ? 1 : (e >= 2047 ? FIX_NAN : e);
}
EPFFT_HD double lift64(double x) { return x * 18446744073709551616.0; }
// x 2^(B - emax + 1022), B = 62 - G: below 2^B in modulus for |x| <
// 2^(emax - 1022).
template <int G>
EPFFT_HD i64 to_fixed(double x, int emax) {
  const int hi = hi_word(x);
  const unsigned lo = lo_word(x);
  const unsigned long long m =
      ((unsigned long long)((((unsigned)hi & 0xfffffu) | 0x100000u) << 10 | lo >> 22) << 32) | (lo << 10);
  int r = 1 + G + emax - (int)(((unsigned)hi >> 20) & 0x7ffu);
  r = r > 63 ? 63 : r;
  const i64 t = (i64)(m >> r), sg = (i64)(hi >> 31);
  return (t ^ sg) - sg;
}
// v 2^(emax - 1084 + LG) rounded to the nearest double: the output of a
// length 2^LG transform of numbers made by to_fixed (every stage divides by
// its radix).  Underflow gives 0, overflow infinity, FIX_NAN NaN.
template <int LG>
EPFFT_HD double from_fixed(i64 v, int emax) {
  const unsigned sg = (unsigned)((unsigned long long)v >> 32) & 0x80000000u;
  const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
#ifdef __CUDA_ARCH__
  const int lz = __clzll((i64)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  const unsigned long long n = a << (lz & 63);
  const int E = emax + LG + 2 - lz;
  unsigned long long b = (n >> 11) + ((n >> 10) & 1ull);
  b += (unsigned long long)(unsigned)(E - 1) << 52;
  if (a == 0 || E <= 0) b = 0;
  // (with FIX_NAN, E is as large for every v)
  if (E >= 2047) b = (unsigned long long)(emax >= FIX_NAN / 2 ? 0x7ff80000u : 0x7ff00000u) << 32;
  return make_double(b | (unsigned long long)sg << 32);
}

// Radix-R butterflies on fixed-point numbers (kernel signs as Bfly).
template <int R, bool INV>
struct Bfly64;
template <bool INV>
struct Bfly64<2, INV> {
  static EPFFT_HD void run(C2<i64>* v) {
    const C2<i64> a = v[0], b = v[1];
    v[0].re = a.re + b.re;
    v[0].im = a.im + b.im;
    v[1].re = a.re - b.re;
    v[1].im = a.im - b.im;
  }
};
template <bool INV>
struct Bfly64<4, INV> {
  static EPFFT_HD void run(C2<i64>* v) {
    const C2<i64> x0 = v[0], x1 = v[1], x2 = v[2], x3 = v[3];
    const i64 a0r = x0.re + x2.re, a0i = x0.im + x2.im, a1r = x0.re - x2.re, a1i = x0.im - x2.im;
    const i64 a2r = x1.re + x3.re, a2i = x1.im + x3.im, dr = x1.re - x3.re, di = x1.im - x3.im;
    v[0].re = a0r + a2r;
    v[0].im = a0i + a2i;
    v[2].re = a0r - a2r;
    v[2].im = a0i - a2i;
    // v[1] = a1 -+ i d (forward -i d = (di, -dr))
    v[1].re = INV ? a1r - di : a1r + di;
    v[1].im = INV ? a1i + dr : a1i - dr;
    v[3].re = INV ? a1r + di : a1r - di;
    v[3].im = INV ? a1i - dr : a1i + dr;
  }
};
template <bool INV>
struct Bfly64<8, INV> {
  static EPFFT_HD void run(C2<i64>* v) {
    C2<i64> e[4] = {v[0], v[2], v[4], v[6]};
    C2<i64> o[4] = {v[1], v[3], v[5], v[7]};
    Bfly64<4, INV>::run(e);
    Bfly64<4, INV>::run(o);
    // o[k] exp(-+ i pi k / 4), k = 1, 2, 3
    C2<i64> t[4];
    t[0] = o[0];
    const i64 p1 = mul_cos4(o[1].re + o[1].im), m1 = mul_cos4(o[1].im - o[1].re);
    t[1].re = INV ? -m1 : p1;
    t[1].im = INV ? p1 : m1;
    t[2].re = INV ? -o[2].im : o[2].im;
    t[2].im = INV ? o[2].re : -o[2].re;
    const i64 p3 = mul_cos4(o[3].re + o[3].im), m3 = mul_cos4(o[3].im - o[3].re);
    t[3].re = INV ? -p3 : m3;
    t[3].im = INV ? -m3 : -p3;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      v[k].re = e[k].re + t[k].re;
      v[k].im = e[k].im + t[k].im;
      v[k + 4].re = e[k].re - t[k].re;
      v[k + 4].im = e[k].im - t[k].im;
    }
  }
};
template <bool INV>
struct Bfly64<16, INV> {
  // z exp(-+ 2 pi i m / 16) for m = 1, 2, 3, 6, 9
  template <int m>
  static EPFFT_HD C2<i64> rot(const C2<i64>& z) {
    C2<i64> o;
    i64 cr, ci, sr, si;  // z cos, z sin of the angle 2 pi m' / 16 reduced to the first octant pair
    if (m == 1 || m == 9) {
      cr = mul_cos8(z.re), ci = mul_cos8(z.im), sr = mul_sin8(z.re), si = mul_sin8(z.im);
    } else if (m == 3) {
      cr = mul_sin8(z.re), ci = mul_sin8(z.im), sr = mul_cos8(z.re), si = mul_cos8(z.im);
    } else {
      cr = sr = mul_cos4(z.re), ci = si = mul_cos4(z.im);
    }
    if (m == 6) cr = -cr, ci = -ci;                          // (cos, sin) = (-h, h)
    if (m == 9) cr = -cr, ci = -ci, sr = -sr, si = -si;  // (-c1, -s1)
    // forward: (re c + im s, im c - re s); inverse: the other sign of s
    o.re = INV ? cr - si : cr + si;
    o.im = INV ? ci + sr : ci - sr;
    return o;
  }
  static EPFFT_HD void run(C2<i64>* v) {
    C2<i64> y[4][4];
#pragma unroll
    for (int n = 0; n < 4; n++) {
#pragma unroll
      for (int k = 0; k < 4; k++) y[n][k] = v[4 * k + n];
      Bfly64<4, INV>::run(y[n]);
    }
    y[1][1] = rot<1>(y[1][1]);
    y[1][2] = rot<2>(y[1][2]);
    y[1][3] = rot<3>(y[1][3]);
    y[2][1] = rot<2>(y[2][1]);
    const C2<i64> z = y[2][2];
    y[2][2].re = INV ? -z.im : z.im;
    y[2][2].im = INV ? z.re : -z.re;
    y[2][3] = rot<6>(y[2][3]);
    y[3][1] = rot<3>(y[3][1]);
    y[3][2] = rot<6>(y[3][2]);
    y[3][3] = rot<9>(y[3][3]);
#pragma unroll
    for (int k = 0; k < 4; k++) {
      C2<i64> w[4] = {y[0][k], y[1][k], y[2][k], y[3][k]};
      Bfly64<4, INV>::run(w);
#pragma unroll
      for (int j = 0; j < 4; j++) v[k + 4 * j] = w[j];
    }
  }
};

// Twiddles w^r, r = 1 .. R - 1, of a stage block (see stage_twiddles in
// fft.cuh; scale 2^(64 - log2 R)).
template <int R, int NS, bool FULL>
EPFFT_HD void stage_twiddles64(const Tw64* tb, int jm, Tw64 (&w)[R]) {
  constexpr int S = R == 4 ? 62 : (R == 8 ? 61 : 60);
  if constexpr (FULL) {
#pragma unroll
    for (int r = 1; r < R; r++) w[r] = tb[(r - 1) * NS + jm];
  } else {
#pragma unroll
    for (int p = 1, i = 0; p < R; p *= 2, i++) {
      w[p] = tb[i * NS + jm];
#pragma unroll
      for (int r = 1; r < p; r++) w[p + r] = tw_mul<S>(w[r], w[p]);
    }
  }
}

}  // namespace epfft
