// FP64 Hartley transforms in 64-bit block fixed point.
//
// GB300 issues FP64 at 1/64 of the FP32 rate (measured: 1.7 DFMA or DADD per
// clock and SM), and a 256-point line FFT of FP64 data is bound by those
// operations (0.55 ms per 256^3 pass).  64-bit integer sums issue 29 times as
// fast (50 per clock and SM), and a 64 x 64-bit product kept to its high half
// is three IMAD.WIDE (5 per clock and SM), so the butterflies run on
// integers: the points of a line pair are scaled to a common exponent, the
// complex FFT is integer arithmetic with Q62 twiddles, and the Hartley
// outputs are rounded back to FP64.  Nothing before or after a pass changes:
// the data between passes is FP64.
//
// Scaling.  With |x| < 2^(E - 1022) for every value of the pair (E the
// largest biased exponent), a value enters as q = x 2^(B - (E - 1022)),
// rounded, |q| <= 2^B.  A radix-RP butterfly can grow a modulus by RP; a
// twiddle product in Q62 (the high 64 bits of the product) divides by 4.
// With Sum_p the product of the first p radices, an intermediate value of pass p
// is a sum of at most Sum_p rotated inputs, each at most once, divided by 4^(p-1).
// Its modulus is therefore at most sqrt(2) 2^B Sum_p / 4^(p-1), and at most
// sqrt(Sum_p) L2 / 4^(p-1) with L2 the 2-norm of the (scaled) line, which is largest
// at p = 1 for radices up to 8.  All moduli stay below 2^61, which leaves room for
// the sums of a rotation (sqrt(2)) and of the Hartley split (2 sqrt(2)), when
// B <= 60 - H, H = max_p log2(Sum_p / 4^(p-1)), or when sqrt(R) L2 <= 2^61: B is the
// larger of the two.  The second keeps the bits of every line whose points are not
// all large, from one large point or a decaying spectrum to a point that stands out
// of a dense background: the error relative to the line's norm is then about
// sqrt(2 N R) 2^-61, whatever the line's shape.  (The 1-norm in its place has the same
// cost, but lost up to 2 bits against FP64 on 1024 points with a background of 1/4
// to 1/128 of the largest: 9.0e-16 against FP64's 2.0e-16, 1.1e-16 now.)
//
// Error: every step rounds to a unit of 2^-B (B = 55 .. 60) of the line's
// largest value, against 2^-53 of the value in FP64, with two to three units
// on the outputs, so that the transform's error relative to the norm of the
// line stays below that of the FP64 butterflies (tests/fx_line_check.cu and
// tests/fx_peak_check.cu measure both against long double, for n = 8 .. 1024 with
// radix 8 and n = 8 .. 256 with radix 4: 0.4 to 1.2e-16 on dense, decaying and
// peaked lines, FP64 1.1 to 2.3e-16).  The passes scale lines
// whose largest value is below 2^-958 up first (fx_enter), and subnormal outputs are
// 0; a NaN or an infinity makes every output of its line pair NaN, as the FP64 sums
// would.
#pragma once

#include "fft_line.cuh"

namespace psd {

struct fx {
  long long v;
  fx() = default;
  __host__ __device__ constexpr explicit fx(long long x) : v(x) {}
};
__host__ __device__ __forceinline__ fx operator+(fx a, fx b) { return fx(a.v + b.v); }
__host__ __device__ __forceinline__ fx operator-(fx a, fx b) { return fx(a.v - b.v); }

// v = h 2^32 + l with both halves signed, so that every partial product of a
// 64-bit multiplication is a signed 32 x 32-bit one.
struct fx_halves {
  int h, l;
};
__host__ __device__ __forceinline__ fx_halves fx_split(long long v) {
  const int l = (int)(unsigned)(unsigned long long)v;
  return {(int)(v >> 32) - (l >> 31), l};
}
__host__ __device__ __forceinline__ long long fx_wide(int a, int b) { return (long long)a * b; }

// Q62 twiddle (cos, sin), split into halves (built on the host).
struct __align__(16) fx_tw {
  int ch, cl, sh, sl;
};
__host__ inline fx_tw fx_make_tw(long double c, long double s) {
  auto q62 = [](long double v) {
    long long q = llroundl(v * 4611686018427387904.0L);
    if ((int)(unsigned)(unsigned long long)q == (int)0x80000000) ++q;  // the low half can be negated
    return q;
  };
  const fx_halves C = fx_split(q62(c)), S = fx_split(q62(s));
  return {C.h, C.l, S.h, S.l};
}

// (a + i b)(c - i s) / 4, rounded (the products of the low halves, below one
// unit, are dropped); ties go down for odd points and up for even ones, so
// that the exact quarters of the points with w = 1 leave no common offset.
// |a|, |b| <= 2^61: the cross terms stay below 2^63.
__host__ __device__ __forceinline__ void fx_rotate(fx& a, fx& b, const fx_tw& w, bool odd) {
  const fx_halves A = fx_split(a.v), B = fx_split(b.v);
  const int nsh = -w.sh, nsl = -w.sl;
  const long long half = (1LL << 31) - (odd ? 1 : 0);
  const long long tr = fx_wide(B.l, w.sh) + (fx_wide(B.h, w.sl) + (fx_wide(A.l, w.ch) + (fx_wide(A.h, w.cl) + half)));
  const long long ti = fx_wide(A.l, nsh) + (fx_wide(A.h, nsl) + (fx_wide(B.l, w.ch) + (fx_wide(B.h, w.cl) + half)));
  a.v = fx_wide(A.h, w.ch) + (fx_wide(B.h, w.sh) + (tr >> 32));
  b.v = fx_wide(B.h, w.ch) + (fx_wide(A.h, nsh) + (ti >> 32));
}

// v / 4 rounded, ties to even: an offset of a fraction of a unit common to all
// points would add up in the lowest frequencies.
__host__ __device__ __forceinline__ fx fx_quarter(fx x) { return fx((x.v + 1 + ((x.v >> 2) & 1)) >> 2); }

// The p = 4 flux F = |G|^2 G of a vertex gradient whose modulus is below 2^61, in
// units of 2^125 of G^3: |G|^2 / 2^64, times 8, times G / 2^64, so |F| < 2^58.
// Returns the high word of |G|^2 / 2^64.
__host__ __device__ __forceinline__ unsigned fx_flux(long long g0, long long g1, long long g2, long long (&F)[3]) {
  const fx_halves a = fx_split(g0), b = fx_split(g1), c = fx_split(g2);
  const long long t = fx_wide(a.h, a.l) + (fx_wide(b.h, b.l) + (fx_wide(c.h, c.l) + (1LL << 30)));
  const long long s = fx_wide(a.h, a.h) + (fx_wide(b.h, b.h) + (fx_wide(c.h, c.h) + (t >> 31)));
  const fx_halves w = fx_split((long long)((unsigned long long)s << 3));
  const long long half = 1LL << 31;
  F[0] = fx_wide(w.h, a.h) + ((fx_wide(w.h, a.l) + (fx_wide(w.l, a.h) + half)) >> 32);
  F[1] = fx_wide(w.h, b.h) + ((fx_wide(w.h, b.l) + (fx_wide(w.l, b.h) + half)) >> 32);
  F[2] = fx_wide(w.h, c.h) + ((fx_wide(w.h, c.l) + (fx_wide(w.l, c.h) + half)) >> 32);
  return (unsigned)((unsigned long long)s >> 32);
}

__host__ __device__ __forceinline__ long long fx_shl(long long v, int k) {
  return (long long)((unsigned long long)v << k);
}

// The 64 bits of a value.
__device__ __forceinline__ unsigned long long fx_bits(long long v) { return (unsigned long long)v; }
__device__ __forceinline__ unsigned long long fx_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long fx_bits(float v) { return (unsigned long long)__float_as_uint(v); }

// x sqrt(1/2) = x + x (sqrt(1/2) - 1), the factor in units of 2^-64.
__host__ __device__ __forceinline__ fx fx_mul_rsqrt2(fx x) {
  constexpr long long W = -5402926248376769404LL;  // (sqrt(1/2) - 1) 2^64
  constexpr int wl = (int)(unsigned)(unsigned long long)W;
  constexpr int wh = (int)(W >> 32) - (wl >> 31);
  const fx_halves X = fx_split(x.v);
  const long long t = fx_wide(X.l, wh) + (fx_wide(X.h, wl) + (1LL << 31));
  return fx(fx_wide(X.h, wh) + (x.v + (t >> 32)));
}

// The rotations of the butterflies, W_16^m = exp(-2 pi i m / 16): radices up
// to 8 need m = 2 and 6 besides the trivial ones.
template <>
__host__ __device__ __forceinline__ void rot16<fx>(int m, fx a, fx b, fx& tr, fx& ti) {
  const fx s = fx_mul_rsqrt2(a + b), d = fx_mul_rsqrt2(b - a);
  if (m == 2) {
    tr = s;
    ti = d;
  } else {  // m = 6
    tr = d;
    ti = fx(-s.v);
  }
}
// The Hartley split keeps twice the outputs (its halving is in the exponent).
template <>
__host__ __device__ __forceinline__ fx half_of<fx>(fx x) {
  return x;
}
#ifdef __CUDACC__
template <>
__device__ __forceinline__ fx shfl_from<fx>(unsigned mask, fx v, int src) {
  return fx(__shfl_sync(mask, v.v, src));
}
#endif

constexpr int fx_log2(int n) { return n <= 1 ? 0 : 1 + fx_log2(n / 2); }

// Passes, headroom and scale of the N-point line FFT with radix RM.
template <int N, int RM>
struct FxPlan {
  static constexpr int R = N < RM ? N : RM;
  static constexpr int lg = fx_log2(N), lr = fx_log2(R);
  static constexpr int P = (lg + lr - 1) / lr;
  static constexpr int headroom() {
    int h = 0;
    for (int p = 1; p <= P; ++p) {
      const int g = lr * p < lg ? lr * p : lg;
      if (g - 2 * (p - 1) > h) h = g - 2 * (p - 1);
    }
    return h;
  }
  static constexpr int B = 60 - headroom();  // the scale that is safe for every line
  // the outputs are w 2^(E - B + kOut) for the split sums w of a line with
  // largest biased exponent E and scale B
  static constexpr int kOut = -1022 + 2 * (P - 1) - 1;
};

constexpr int kFxMinExp = 64;    // lines whose largest biased exponent is below this are scaled up first
constexpr int kFxMaxExp = 2046;  // above: NaN or infinity

// An upper bound of this value's share of the line's squared 2-norm in units of
// 2^(2 (E - 1032)), from its high word: at most 2^20, so that 2048 values fit.
__host__ __device__ __forceinline__ unsigned fx_square(unsigned hi, int E) {
  const int d = E - (int)((hi >> 20) & 0x7FFu);
  const unsigned m = ((((hi & 0xFFFFFu) | 0x100000u) >> 11) >> (d < 31 ? d : 31)) + 1u;
  return m * m;
}
// The name under which tests/fx_line_check.cu sums the same bound.
__host__ __device__ __forceinline__ unsigned fx_l1(unsigned hi, int E) { return fx_square(hi, E); }
// The scale B of a line whose squared 2-norm is below l2 2^(2 (E - 1032)):
// R L2^2 2^(2 B) <= 2^122 in units of 2^(2 (E - 1022)).
template <class Plan>
__host__ __device__ __forceinline__ int fx_scale(unsigned l2) {
#ifdef __CUDA_ARCH__
  const int bits = 32 - __clz((int)l2);
#else
  const int bits = l2 ? 32 - __builtin_clz(l2) : 0;
#endif
  const int B = (142 - Plan::lr - bits) >> 1;
  return B < Plan::B ? Plan::B : (B > 60 ? 60 : B);
}

// x 2^(B - (E - 1022)) rounded to nearest, from the bits of x (hi, lo), for a
// line with largest biased exponent E >= 64 (zeros and subnormals of such
// a line give 0).
__host__ __device__ __forceinline__ fx fx_quantise(unsigned hi, unsigned lo, int E, int B) {
  const int d = (60 - B) + E - (int)((hi >> 20) & 0x7FFu);
  unsigned long long m = ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
  m = (((m << 8) >> (d < 63 ? d : 63)) + 1) >> 1;
  const long long s = (long long)((int)hi >> 31);
  return fx(((long long)m ^ s) - s);
}

// w 2^e as a double, rounded to nearest; underflow gives 0, overflow infinity.
__host__ __device__ __forceinline__ double fx_result(long long w, int e) {
  const unsigned neg = (unsigned)((unsigned long long)w >> 32) & 0x80000000u;
  unsigned long long a = w < 0 ? 0ULL - (unsigned long long)w : (unsigned long long)w;
  if (a == 0) return 0.0;
#ifdef __CUDA_ARCH__
  const int z = __clzll((long long)a);
#else
  const int z = __builtin_clzll(a);
#endif
  a <<= z;
  const int E = 63 - z + e + 1023;  // biased exponent before the rounding
  // the leading bit of a >> 11 (and a carry of the rounding) adds to the exponent
  unsigned long long r = ((unsigned long long)(unsigned)(E - 1) << 52) + (a >> 11) + ((a >> 10) & 1ULL);
  if ((unsigned)(E - 1) >= 2046u) r = E <= 0 ? 0ULL : 0x7FF0000000000000ULL;
  return ff_bitsd(r | ((unsigned long long)neg << 32));
}

}  // namespace psd
