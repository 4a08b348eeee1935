// fx64.cuh - 64-bit block fixed-point arithmetic for the FFT passes of the FP64 paths.
//
// GB300 issues about two FP64 operations a clock per SM, but about 48 64-bit integer additions
// (measured: DADD and DFMA 1.7 lanes a clock per SM, 64-bit adds 48, 32 x 32 -> 64-bit
// multiply-adds 25).  A transform is mostly additions, so the passes run it on 64-bit integers
// with an exponent per block of values, and meet FP64 only at their ends:
//   a value is v 2^u, v a signed 64-bit integer, u the unit exponent that a block shares.
//   Stage A: the R points of one thread are a block.  They are brought below 2^head(R) (their
//     largest exponent sets the unit: doubles lose nothing that lies within 2^-3 of the largest),
//     so that an R-point transform, whose outputs are at most R sqrt(2) times its inputs, stays
//     below 2^62.
//   Twiddles: x w / 4 with w scaled by 2^62, rounded to nearest.
//   Stage B: the blocks that meet in it (the threads of one pencil) are brought to a common unit,
//     the finest in which the largest value still stays below 2^head(R).
// Rounding therefore happens at 2^-57 or so of the largest value of a block instead of at 2^-53 of
// each value, and additions are exact: against long double the transform of 16 to 256 points comes
// out 1.8 to 3.6 times nearer (relative 2-norm) than the same two stages in FP64: 1.9 to 3.3 for white and
// zero-padded pencils, 1.8 to 2.8 for spikes and for spectra that fall off (what is left is the
// rounding of the results to doubles).  A block that holds an infinity or a NaN gives NaN (unit kNanUnit).
// Subnormal doubles are read and written (a unit below that of the smallest normal is as good as any).
//
// Unit exponents are kept in the bias of FP64: value = v 2^(u - 1075).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_core.cuh"

namespace scfft {

constexpr int kNanUnit = 1 << 14;  // unit of a block with an infinity or a NaN

// Bits a value may have before an R-point transform: R sqrt(2) 2^head < 2^62.
__host__ __device__ constexpr int fx_head(int R) { return R <= 4 ? 59 : 57; }

// v = hi 2^32 + lo with lo a signed 32-bit number: products of the halves need no sign fix-up
FXHD int fx_lo(long long v) { return (int)v; }
FXHD int fx_hi(long long v) { return (int)(v >> 32) + (int)((unsigned)v >> 31); }
constexpr long long kHalf32 = 0x80000000ll;

// x c (|x| < 2^62) for the compile-time constant 0 < c < 1 given as C = 2^64 c, or 2^64 (c - 1)
// when c >= 1/2 (ONE); rounded to nearest, but for the product of the low halves
template <long long C, bool ONE> FXHD long long fx_mulc(long long x) {
  constexpr int cl = (int)C, ch = (int)(C >> 32) + (int)((unsigned)C >> 31);
  const int xl = fx_lo(x), xh = fx_hi(x);
  const long long mid = (long long)xh * cl + kHalf32 + (long long)xl * ch;
  const long long r = (long long)xh * ch + (mid >> 32);
  return ONE ? r + x : r;
}

// v / 2^k rounded to nearest, ties away from zero, k >= 1.  A short shift meets a tie often (every
// second value at one bit): ties that all went up would add the same fraction of a unit to every
// value, an error of the zero frequency that is the same in every pencil and adds up over passes
// and iterations, and would break the mirror symmetries that the method keeps exactly.
FXHD long long fx_shr(long long v, int k) { return (v + (1ll << (k - 1)) + (v >> 63)) >> k; }
template <int K> FXHD long long fx_shr(long long v) { return fx_shr(v, K); }

// 2^64 cos(k pi / 24), less 2^64 from 1/2 on, k = 1 .. 11
__host__ __device__ constexpr long long fx_cos24(int k) {
  return k == 1 ? -157814452752426473ll : k == 2 ? -628557561968679382ll : k == 3 ? -1404174782535421627ll
       : k == 4 ? -2471395088767036514ll : k == 5 ? -3811958045334532105ll : k == 6 ? -5402926248376769404ll
       : k == 7 ? -7217077790839976240ll : k == 8 ? (-0x7fffffffffffffffll - 1) : k == 9 ? 7059263338087549767ll
       : k == 10 ? 4774368686408090022ll : 2407783262799110479ll;
}

// a (cos t - i sin t) forward, a (cos t + i sin t) inverse, t = k pi / 24, 0 < k < 12
template <int K, bool INV> FXHD fxc fx_rot(fxc a) {
  if constexpr (K == 6) {  // cos = sin
    constexpr long long H = fx_cos24(6);
    return INV ? mk(fx_mulc<H, true>(a.x - a.y), fx_mulc<H, true>(a.x + a.y))
               : mk(fx_mulc<H, true>(a.x + a.y), fx_mulc<H, true>(a.y - a.x));
  } else {
    constexpr long long C = fx_cos24(K), S = fx_cos24(12 - K);
    constexpr bool C1 = K <= 8, S1 = K >= 4;  // the cosine, the sine is at least 1/2
    constexpr int cl = (int)C, ch = (int)(C >> 32) + (int)((unsigned)C >> 31);
    constexpr int sl = (int)S, sh = (int)(S >> 32) + (int)((unsigned)S >> 31);
    const long long p = a.x, q = INV ? -a.y : a.y;  // re = p c + q s, im' = q c - p s (conjugated for INV)
    const long long np = -p;
    const int pl = fx_lo(p), ph = fx_hi(p), ql = fx_lo(q), qh = fx_hi(q), nl = fx_lo(np), nh = fx_hi(np);
    const long long m0 = (long long)ph * cl + kHalf32 + (long long)pl * ch + (long long)qh * sl + (long long)ql * sh;
    const long long m1 = (long long)qh * cl + kHalf32 + (long long)ql * ch + (long long)nh * sl + (long long)nl * sh;
    long long re = (long long)ph * ch + (long long)qh * sh + (m0 >> 32);
    long long im = (long long)qh * ch + (long long)nh * sh + (m1 >> 32);
    if (C1) { re += p; im += q; }
    if (S1) { re += q; im += np; }
    return mk(re, INV ? -im : im);
  }
}

template <int R, bool INV> struct TwiddleConst<fxc, R, INV> {
  static FXHD fxc apply(fxc a, int m) {
    const int q = ((2 * m * 24 / R) % 48 + 48) % 48;  // a constant at every call site
    // a quarter turn at a time, then the rest (each branch folds)
    const int k = q % 12, t = q / 12;
    fxc b = a;
    if (t == 1) b = INV ? mk(-a.y, a.x) : mk(a.y, -a.x);
    if (t == 2) b = mk(-a.x, -a.y);
    if (t == 3) b = INV ? mk(a.y, -a.x) : mk(-a.y, a.x);
    switch (k) {
      case 1: return fx_rot<1, INV>(b);
      case 2: return fx_rot<2, INV>(b);
      case 3: return fx_rot<3, INV>(b);
      case 4: return fx_rot<4, INV>(b);
      case 5: return fx_rot<5, INV>(b);
      case 6: return fx_rot<6, INV>(b);
      case 7: return fx_rot<7, INV>(b);
      case 8: return fx_rot<8, INV>(b);
      case 9: return fx_rot<9, INV>(b);
      case 10: return fx_rot<10, INV>(b);
      case 11: return fx_rot<11, INV>(b);
      default: return b;
    }
  }
};

template <bool INV> struct DFT<3, INV, fxc> {
  static FXHD void run(fxc* v) {
    const fxc s = v[1] + v[2], d = v[1] - v[2];
    const fxc m = mk(v[0].x - fx_shr<1>(s.x), v[0].y - fx_shr<1>(s.y));
    constexpr long long C = fx_cos24(4);  // sqrt(3) / 2
    const fxc r = mk(fx_mulc<C, true>(d.x), fx_mulc<C, true>(d.y));
    v[0] = v[0] + s;
    v[1] = INV ? mk(m.x - r.y, m.y + r.x) : mk(m.x + r.y, m.y - r.x);
    v[2] = INV ? mk(m.x + r.y, m.y - r.x) : mk(m.x - r.y, m.y + r.x);
  }
};

// a w / 4 forward, a conj(w) / 4 inverse; w = 2^62 (cos, sin) of the forward angle as the halves
// (cos hi, cos lo, sin hi, sin lo), low halves odd (so their negatives are 32-bit numbers too);
// the forward twiddle is cos - i sin
template <bool INV> FXHD fxc fx_twiddle(fxc a, int4 w) {
  const int ch = w.x, cl = w.y, sh = INV ? -w.z : w.z, sl = INV ? -w.w : w.w;
  const int pl = fx_lo(a.x), ph = fx_hi(a.x), ql = fx_lo(a.y), qh = fx_hi(a.y);
  const long long m0 = (long long)ph * cl + kHalf32 + (long long)pl * ch + (long long)qh * sl + (long long)ql * sh;
  const long long m1 = (long long)qh * cl + kHalf32 + (long long)ql * ch + (long long)ph * (-sl) + (long long)pl * (-sh);
  return mk((long long)ph * ch + (long long)qh * sh + (m0 >> 32), (long long)qh * ch + (long long)ph * (-sh) + (m1 >> 32));
}
// the unit twiddle
FXHD fxc fx_quarter(fxc a) { return mk(fx_shr<2>(a.x), fx_shr<2>(a.y)); }

// ((a ka + b kb) / 2^64, rounded; |a|, |b| < 2^62, |ka|, |kb| < 2^62, k as halves (hi, lo)
FXHD long long fx_mac2(long long a, int2 ka, long long b, int2 kb) {
  const int al = fx_lo(a), ah = fx_hi(a), bl = fx_lo(b), bh = fx_hi(b);
  const long long m =
      (long long)ah * ka.y + kHalf32 + (long long)al * ka.x + (long long)bh * kb.y + (long long)bl * kb.x;
  return (long long)ah * ka.x + (long long)bh * kb.x + (m >> 32);
}
FXHD int2 fx_neg(int2 k) { return make_int2(-k.x, -k.y); }
// halves of a factor; its last bit is set, which keeps the low half off -2^31
FXHD int2 fx_split(long long k) {
  k |= 1;
  return make_int2(fx_hi(k), fx_lo(k));
}

// ---------------------------------------------------------------- FP64 at the ends
FXHD int fx_clz(unsigned v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}
// Largest |high word| of a thread's doubles so far; the exponent of a block.
FXHD int fx_top(int m, int hi) {
  const int a = hi & 0x7fffffff;
  return a > m ? a : m;
}
FXHD int fx_exp_of(int m) { return (m >> 20) > 1 ? (m >> 20) : 1; }
FXHD int fx_unit_of(int et, int head) { return et >= 0x7ff ? kNanUnit : et - (head - 53); }
// the double (hi, lo) in the unit fx_unit_of(et, HEAD), cut toward zero.  Zeros and subnormals have
// the exponent 1 and no leading bit.
template <int HEAD> FXHD long long fx_from_double(int hi, unsigned lo, int et) {
  const int a = hi & 0x7fffffff, e = fx_exp_of(a);
  const int d = et - e < 63 ? et - e : 63;
  unsigned long long m = ((unsigned long long)(unsigned)(a - ((e - 1) << 20)) << 32) | lo;
  m = (m << (HEAD - 53)) >> d;
  return hi < 0 ? -(long long)m : (long long)m;
}
// v 2^(u - 1075) as a double, rounded to nearest (ties away from zero); NaN from kNanUnit / 2 on.
// PLAIN: for a unit in which every value but 0 is a normal double (fx_plain).
FXHD bool fx_plain(int u) { return (unsigned)(u - 53) <= 2036u - 53u; }
template <bool PLAIN> FXHD unsigned long long fx_to_bits(long long v, int u) {
  const unsigned long long a = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  const int z = ah ? fx_clz(ah) : 32 + fx_clz(al);  // 1 .. 64
  const int e = u + 11 - z;
  const unsigned long long n = a << (z - 1);
  unsigned long long m = (n + 0x200) >> 10;
  m += (unsigned long long)(unsigned)(e - 1) << 52;
  if (a == 0) m = 0;
  if (!PLAIN) {
    if (a != 0 && e <= 0) m = e > -53 ? (n + (1ull << (10 - e))) >> (11 - e) : 0;  // subnormal
    if (a != 0 && e > 2046) m = 0x7ff0000000000000ull;
    if (u >= kNanUnit / 2) return 0x7ff8000000000000ull;
  }
  return m | ((unsigned long long)v & 0x8000000000000000ull);
}
// bits a block's values may use, from the OR of their high words' magnitudes (fx_or)
FXHD int fx_or(int m, long long v) {
  const int h = (int)(v >> 32);
  return m | (h ^ (h >> 31));
}
FXHD int fx_bits(int m) { return 64 - fx_clz((unsigned)m); }  // |v| <= 2^bits
}  // namespace scfft
