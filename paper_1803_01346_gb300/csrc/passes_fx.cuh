// passes_fx.cuh - the FFT passes of the FP64 paths, on 64-bit block fixed point (fx64.cuh): spectra
// and fields are doubles in memory, transforms and spectral products run on 64-bit integers, the
// node-wise steps in FP64.
//
// What bounds them is latency and issue on the integer pipes (additions 2, twiddles about 20
// instructions a point): the padded z pass of 192 points runs 8 warps an SM (211 registers) at 46% issue, the
// y passes 19 warps at 60%; not the FP64 pipe, which kept the FP64 passes before these 76% busy.
// Measured on 64 x 64 x 96 with a shield's box, us a launch, FP64 |
// double-float passes before | these: padded z 589 | 306 | 136, Eq. 5 update 177 | 122 | 63, padded y
// inverse 127 | 71 | 32, curl z 79 | 51 | 32; one right-hand side 10.4 | 6.2 | 2.8 ms.  A length L = R1 R2
// transform is two register stages with one shared-memory transpose; every length is compiled on its
// own; the component loops stay rolled, so that a kernel's four unrolled DFT bodies stay within the
// instruction cache.  (Reading a component's input during the transform before it, in the z pass: no gain.
// The z pass of 192 points held to five CTAs an SM, 200 registers: Phi 96^3's 314 us against 292.)
#pragma once
#include <limits.h>

#include "fx64.cuh"
#include "passes_wide.cuh"

namespace scfft {
namespace fx {

using wide::cmax;

// the real and imaginary double of one complex value as raw words: (re lo, re hi, im lo, im hi)
__device__ __forceinline__ int4 ld_raw(const double2* p) { return *reinterpret_cast<const int4*>(p); }
__device__ __forceinline__ int4 raw_of(double2 v) {
  return make_int4(__double2loint(v.x), __double2hiint(v.x), __double2loint(v.y), __double2hiint(v.y));
}
__device__ __forceinline__ int top_of(int m, int4 r) { return fx_top(fx_top(m, r.y), r.w); }
template <int HEAD> __device__ __forceinline__ fxc fx_of(int4 r, int et) {
  return mk(fx_from_double<HEAD>(r.y, (unsigned)r.x, et), fx_from_double<HEAD>(r.w, (unsigned)r.z, et));
}
template <bool PLAIN> __device__ __forceinline__ double2 dbl_of(fxc v, int u) {
  return make_double2(__longlong_as_double((long long)fx_to_bits<PLAIN>(v.x, u)),
                      __longlong_as_double((long long)fx_to_bits<PLAIN>(v.y, u)));
}
// A thread's block of doubles (R points, those from N on zero) in fixed point; m: its fx_top, made 0 for
// a block of zeros alone and 1 for one that lies below 2^-1042.  Returns the block's exponent.
template <int R, int N> __device__ __forceinline__ int block_in(fxc* v, const int4* raw, int& m) {
  if (m == 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) m |= raw[i].x | raw[i].z;
    m = m != 0;
  }
  const int et = fx_exp_of(m);
#pragma unroll
  for (int i = 0; i < R; ++i) v[i] = i < N ? fx_of<fx_head(R)>(raw[i < N ? i : 0], et) : mk(0ll, 0ll);
  return et;
}
// The unit of a block of zeros, which has no part in the choice of a pencil's unit.
constexpr int kNoUnit = -(1 << 20);
// Writing results: whether the unit is plain (fx_plain; zeros alone are) is asked once a block and f called
// with std::true_type or std::false_type: with the checks at every value a 64 x 64 x 96 right-hand side took
// 3.02 ms, without 2.79, and Phi at 96^3 569 us, without 500.
__device__ __forceinline__ bool plain_unit(int u) { return fx_plain(u) || u < kNoUnit / 2; }
template <typename F> __device__ __forceinline__ void by_unit(bool plain, F&& f) {
  if (__builtin_expect(plain, 1)) f(std::true_type{});
  else f(std::false_type{});
}
__device__ __forceinline__ fxc shfl_fx(fxc v, int s) {
  return mk(__shfl_sync(0xffffffffu, v.x, s), __shfl_sync(0xffffffffu, v.y, s));
}
// the unit that a block (own unit u, magnitude bits m) needs in a stage of R points
template <int R> __device__ __forceinline__ int want_unit(int u, int m) {
  const int w = u + fx_bits(m) - fx_head(R);
  return w > u ? w : u;
}
// Largest p over the threads of a column (same t % TC) into slot[c], for a CTA of NT threads.  With 48
// threads the second warp has 16 lanes, and a shuffle must not read the others: the butterfly stays within
// groups of W lanes, which exist whole in every warp, and atomicMax joins the groups.
template <int TC, int NT> __device__ __forceinline__ void column_max(int* slot, int p) {
  constexpr int W = NT % 32 ? NT % 32 : 32;
  static_assert((W & (W - 1)) == 0 && W >= TC && W % TC == 0, "a CTA ends in a power of two of lanes, whole columns");
#pragma unroll
  for (int o = TC; o < W; o <<= 1) {
    const int q = __shfl_xor_sync(0xffffffffu, p, o);
    p = q > p ? q : p;
  }
  const int lane = threadIdx.x & (W - 1);
  if (lane < TC) atomicMax(slot + lane, p);
}
// v, in unit u, to unit U >= u
template <int R> __device__ __forceinline__ void to_unit(fxc* v, int u, int U) {
  const int k = U - u < 63 ? U - u : 63;
  if (k > 0) {
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = mk(fx_shr(v[i].x, k), fx_shr(v[i].y, k));
  }
}

// ---------------------------------------------------------------- y passes
struct YArgs {
  double2* base;
  int rows, sx, HX, nzs;
  const int4* tw;
  const Ctrl* ctrl;
  int check_done;
  // planes z = zoff + blockIdx.y; rows outside [ylo, yhi): the forward pass reads them as zero, the
  // inverse pass does not write them
  int zoff, ylo, yhi;
};

// grid (ceil(HX / TC), planes, 3), TC columns of one (component, plane) per CTA.  PAD: the
// zero-padded transform (forward: only the first half of the rows is read; inverse: only the
// first half is kept).  192 points (R2 = 12) are held to ten CTAs an SM: left alone the compiler takes registers
// for nine (forward y on the lens's box at 96 x 96 x 64: 25.4 us against 18.4).
template <int R1, int R2, int TC, bool INV, bool PAD>
__global__ void __launch_bounds__(TC * R1, R2 == 12 ? 10 : 0) ypass_kernel(const YArgs a) {
  constexpr int L = R1 * R2, NT = TC * R1;
  constexpr int S2 = R1 * TC + (TC < 8 ? TC : 0);  // 8 lanes of a 16-byte access on distinct banks
  constexpr bool HALF = PAD && !INV;
  constexpr int NL = HALF ? R2 / 2 : R2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int unit[TC];
  after_previous();
  if (a.check_done && a.ctrl->done) return;
  int4* tw = reinterpret_cast<int4*>(smem_raw);
  fxc* sm = reinterpret_cast<fxc*>(tw + L);
  const int t = threadIdx.x;
  const int c = t % TC, n1 = t / TC;
  const int z = a.zoff + blockIdx.y, kx = blockIdx.x * TC + c;
  const bool colok = kx < a.HX;
  double2* col = a.base + ((size_t)(blockIdx.z * a.nzs + z) * a.rows) * a.sx + kx;
  int4 raw[NL];
  int m = 0;
#pragma unroll
  for (int n2 = 0; n2 < NL; ++n2) {
    const int row = n1 + R1 * n2;
    raw[n2] = (colok && (INV || (row >= a.ylo && row < a.yhi))) ? ld_raw(col + (size_t)row * a.sx)
                                                               : make_int4(0, 0, 0, 0);
  }
  for (int i = t; i < L; i += NT) tw[i] = a.tw[i];
  if (t < TC) unit[t] = kNoUnit;
#pragma unroll
  for (int n2 = 0; n2 < NL; ++n2) m = top_of(m, raw[n2]);
  fxc v[R2];
  const int et = block_in<R2, NL>(v, raw, m);
  const bool some = m != 0;
  dft_maybe_half<R2, INV, HALF>(v);
  __syncthreads();  // twiddles staged, units cleared
  const int u = fx_unit_of(et, fx_head(R2)) + 2;
  m = 0;
#pragma unroll
  for (int k2 = 0; k2 < R2; ++k2) {
    v[k2] = k2 == 0 ? fx_quarter(v[0]) : fx_twiddle<INV>(v[k2], tw[n1 * k2]);
    m = fx_or(fx_or(m, v[k2].x), v[k2].y);
  }
  column_max<TC, NT>(unit, some ? want_unit<R1>(u, m) : kNoUnit);
  __syncthreads();
  const int U = unit[c];
  to_unit<R2>(v, u, U);
#pragma unroll
  for (int k2 = 0; k2 < R2; ++k2) sm[k2 * S2 + n1 * TC + c] = v[k2];
  __syncthreads();
  if (n1 < R2) {
    fxc w[R1];
#pragma unroll
    for (int i = 0; i < R1; ++i) w[i] = sm[n1 * S2 + i * TC + c];
    DFT<R1, INV, fxc>::run(w);
    if (colok)
      by_unit(plain_unit(U), [&](auto plain) {
#pragma unroll
        for (int k1 = 0; k1 < (PAD && INV ? R1 / 2 : R1); ++k1) {
          const int row = n1 + R2 * k1;
          if (!INV || (row >= a.ylo && row < a.yhi)) col[(size_t)row * a.sx] = dbl_of<plain.value>(w[k1], U);
        }
      });
  }
}

// ---------------------------------------------------------------- z passes
struct ZArgs {
  double2* base;
  int rows, sx, HX, nzs;
  const int4* tw;
  // curl: per-axis wavenumbers and smoothing; along z as integers (t1 = S 2^(62-e1), t2 = S k 2^(62-e2))
  const double* kt0; const double* kt1;
  const double* st0; const double* st1;
  const long long* t1; const long long* t2;
  int e1, e2;
  double scale;
  // kernel: the octant as integers, K 2^(62 - ek(ky, kx))
  const long long* kap;
  const int* ek;
  int nx, ny, nz;
  const Ctrl* ctrl;
  int check_done;
  int ilo, ihi, olo, ohi;  // planes outside [ilo, ihi) read as zero, planes outside [olo, ohi) are not written
};

// |c| < 2^dexp(c)
__device__ __forceinline__ int dexp(double c) { return ((__double2hiint(c) >> 20) & 0x7ff) - 1022; }
// c 2^(62 - e), |c| < 2^e (0 for what is below 2.2e-308)
__device__ __forceinline__ long long scaled62(double c, int e) {
  if (dexp(c) == -1022) return 0;
  return fx_from_double<62>(__double2hiint(c), (unsigned)__double2loint(c), e + 1022);
}

// One CTA takes TC columns (kx, y) of all three components: forward z transforms one after
// another, the product on the points each thread itself finished (its "own slots" of the transpose
// buffer, so the product needs no barrier), inverse transforms.  KIND 0: the smoothed curl on the
// unpadded grid; KIND 1: the Biot-Savart kernel on the padded grid (half of the input planes are
// zero and half of the output planes are kept).  Omega's box: KIND 1 reads and KIND 0 writes its
// planes only; TB, the transposed iteration's form, the other way round (run-time ranges on both
// sides of both cost Phi 96^3 1%).  A 1-D grid: TC consecutive kx of one row per
// CTA; the columns left over when HX is not a multiple of TC are packed TC (row, kx) pairs to a
// CTA and run first.
template <int R1, int R2, int TC, int KIND, bool TB>
__global__ void __launch_bounds__(TC * R1) zpass_kernel(const ZArgs a) {
  constexpr int L = R1 * R2, NT = TC * R1;
  constexpr bool PR = KIND == 1;
  constexpr int NL = PR ? R2 / 2 : R2;
  constexpr int PADZ = TC < 8 ? TC : 0;  // 8 lanes of a 16-byte access on distinct banks
  constexpr int S2 = R1 * TC + PADZ;     // forward transpose [k2][n1][c]
  constexpr int S1 = R2 * TC + PADZ;     // inverse transpose [m1][k2][c]
  constexpr int CS = cmax(R2 * S2, R1 * S1);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int unit[6][TC];  // units of the three spectra, of the three products' transforms
  after_previous();
  if (a.check_done && a.ctrl->done) return;
  int4* tw = reinterpret_cast<int4*>(smem_raw);
  fxc* F = reinterpret_cast<fxc*>(tw + L);
  const int t = threadIdx.x;
  const int c = t % TC, n1 = t / TC;
  const int nfull = a.HX / TC, rem = a.HX - nfull * TC;
  const int ntail = (a.rows * rem + TC - 1) / TC;
  int y, kx;
  bool colok = true;
  if ((int)blockIdx.x >= ntail) {
    const int b = blockIdx.x - ntail;
    y = b / nfull;
    kx = (b - y * nfull) * TC + c;
  } else {
    const int e = blockIdx.x * TC + c;
    colok = e < a.rows * rem;
    y = colok ? e / rem : 0;
    kx = colok ? nfull * TC + (e - y * rem) : 0;
  }
  const size_t zstride = (size_t)a.rows * a.sx;
  const size_t cstride = (size_t)a.nzs * zstride;
  double2* col = a.base + (size_t)y * a.sx + kx;
  for (int i = t; i < L; i += NT) tw[i] = a.tw[i];
  for (int i = t; i < 6 * TC; i += NT) unit[i / TC][i % TC] = kNoUnit;
  bool z0 = true, z1 = true;  // whether the x, the y component has anything on the thread's points that k_z multiplies
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    fxc* Fq = F + q * CS;
    int4 raw[NL];
    int m = 0;
#pragma unroll
    for (int n2 = 0; n2 < NL; ++n2) {
      const int l = n1 + R1 * n2;
      raw[n2] = (colok && (!(PR || TB) || (l >= a.ilo && l < a.ihi))) ? ld_raw(col + q * cstride + l * zstride)
                                                   : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int n2 = 0; n2 < NL; ++n2) m = top_of(m, raw[n2]);
    fxc v[R2];
    const int et = block_in<R2, NL>(v, raw, m);
    const bool some = m != 0;
    dft_maybe_half<R2, false, PR>(v);
    if (q == 0) __syncthreads();  // twiddles staged, units cleared
    const int u = fx_unit_of(et, fx_head(R2)) + 2;
    m = 0;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      v[k2] = k2 == 0 ? fx_quarter(v[0]) : fx_twiddle<false>(v[k2], tw[n1 * k2]);
      m = fx_or(fx_or(m, v[k2].x), v[k2].y);
    }
    column_max<TC, NT>(unit[q], some ? want_unit<R1>(u, m) : kNoUnit);
    __syncthreads();
    to_unit<R2>(v, u, unit[q][c]);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) Fq[k2 * S2 + n1 * TC + c] = v[k2];
    __syncthreads();
    if (n1 < R2) {
      fxc w[R1];
#pragma unroll
      for (int i = 0; i < R1; ++i) w[i] = Fq[n1 * S2 + i * TC + c];
      DFT<R1, false, fxc>::run(w);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) Fq[n1 * S2 + k1 * TC + c] = w[k1];
      if (!PR) {
        long long any = 0;
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1)
          if (k1 % (R1 / 2) != 0 || n1 != 0) any |= w[k1].x | w[k1].y;  // (k_z = 0 on DC and Nyquist)
        if (q == 0) z0 = any != 0;
        if (q == 1) z1 = any != 0;
      }
    }
  }
  // product at kz = k2 + R2 k1 on the thread's own slots: G = i (k x F), |k| < 2^62 in units 2^(ec-62)
  int mg[3] = {0, 0, 0};  // magnitudes of the thread's products
  int ug[3];              // their units
  {
    const int k2 = n1;
    fxc* F0 = F + k2 * S2 + c;
    const int u0 = unit[0][c], u1 = unit[1][c], u2 = unit[2][c];
    int ux = u1 > u2 ? u1 : u2, uy = u0 > u2 ? u0 : u2, uz = u0 > u1 ? u0 : u1;
    int ec;
    long long cx = 0, cy = 0, cz = 0;
    const size_t plane = (size_t)(a.ny + 1) * (a.nx + 1), oct = plane * (a.nz + 1);
    const int fy = y <= a.ny ? y : 2 * a.ny - y;
    const long long* K = PR ? a.kap + (size_t)fy * (a.nx + 1) + kx : nullptr;
    if (PR) {
      ec = a.ek[fy * (a.nx + 1) + kx];
    } else {
      const double s = a.st0[kx] * a.st1[y] * a.scale;
      const double dx = s * a.kt0[kx], dy = s * a.kt1[y];
      ec = cmax(cmax(dexp(dx), dexp(dy)) + a.e1, dexp(s) + a.e2);
      cx = scaled62(dx, ec - a.e1);
      cy = scaled62(dy, ec - a.e1);
      cz = scaled62(s, ec - a.e2);
    }
    // A spectrum whose factor vanishes does not set the unit of the product when the other one would lose bits by
    // it (the curl on k_x = 0 or k_y = 0, and off the DC of a component that does not vary along z: a uniform
    // background must not cost the rest its low bits; within 2^4 of each other nothing is lost, the factors having
    // 62).  An infinity or a NaN does, as 0 times it is a NaN.
    if (!PR) {
      const bool tx = cx != 0, ty = cy != 0;
      auto unit_of = [](int ua, bool a_on, int ub, bool b_on) {
        if (!a_on && b_on && ua > ub + 4 && ua < kNanUnit / 2) return ub;
        if (a_on && !b_on && ub > ua + 4 && ub < kNanUnit / 2) return ua;
        return max(ua, ub);
      };
      ux = unit_of(u1, z1, u2, ty);
      uy = unit_of(u2, tx, u0, z0);
      uz = unit_of(u0, ty, u1, tx);
    }
    ug[0] = ux + ec + 2;
    ug[1] = uy + ec + 2;
    ug[2] = uz + ec + 2;
    if (n1 < R2) {
      // right shifts that bring the two spectra of an output to their common unit, taken on the
      // factors, which have bits to spare
      auto shift = [](int U, int u) { return PR || U >= u ? min(U - u, 63) : 63; };
      const int s1x = shift(ux, u1), s2x = shift(ux, u2), s0y = shift(uy, u0), s2y = shift(uy, u2), s0z = shift(uz, u0),
                s1z = shift(uz, u1);
#pragma unroll 2
      for (int k1 = 0; k1 < R1; ++k1) {
        const int kz = k2 + R2 * k1;
        long long ax, ay, az;
        if (PR) {
          // K^ is odd in ky (component y) and in kz (component z) about the fold
          const size_t off = (size_t)(kz <= L / 2 ? kz : L - kz) * plane;
          ax = K[off];
          ay = K[oct + off];
          az = K[2 * oct + off];
          if (y > a.ny) ay = -ay;
          if (kz > L / 2) az = -az;
        } else {
          const long long t1 = a.t1[kz], t2 = a.t2[kz];
          ax = __mul64hi(cx, t1) << 2;
          ay = __mul64hi(cy, t1) << 2;
          az = __mul64hi(cz, t2) << 2;
        }
        const fxc G0 = F0[k1 * TC], G1 = F0[CS + k1 * TC], G2 = F0[2 * CS + k1 * TC];
        fxc hx, hy, hz;
        {
          const int2 p = fx_split(az >> s1x), q = fx_split(ay >> s2x);
          hx = mk(fx_mac2(G1.y, p, G2.y, fx_neg(q)), fx_mac2(G2.x, q, G1.x, fx_neg(p)));
        }
        {
          const int2 p = fx_split(ax >> s2y), q = fx_split(az >> s0y);
          hy = mk(fx_mac2(G2.y, p, G0.y, fx_neg(q)), fx_mac2(G0.x, q, G2.x, fx_neg(p)));
        }
        {
          const int2 p = fx_split(ay >> s0z), q = fx_split(ax >> s1z);
          hz = mk(fx_mac2(G0.y, p, G1.y, fx_neg(q)), fx_mac2(G1.x, q, G0.x, fx_neg(p)));
        }
        F0[k1 * TC] = hx;
        F0[CS + k1 * TC] = hy;
        F0[2 * CS + k1 * TC] = hz;
        mg[0] = fx_or(fx_or(mg[0], hx.x), hx.y);
        mg[1] = fx_or(fx_or(mg[1], hy.x), hy.y);
        mg[2] = fx_or(fx_or(mg[2], hz.x), hz.y);
      }
    }
  }
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    fxc* Fq = F + q * CS;
    fxc w[R1];
    int u = INT_MIN, p = INT_MIN;
    if (n1 < R2) {
      // the products to fx_head(R1) bits (they use up to 61)
      const int mq = q == 0 ? mg[0] : q == 1 ? mg[1] : mg[2];
      const int uq = q == 0 ? ug[0] : q == 1 ? ug[1] : ug[2];
      const int lz = fx_head(R1) - fx_bits(mq);
      u = uq - lz + 2;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) w[k1] = Fq[n1 * S2 + k1 * TC + c];
      if (lz >= 0) {
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) w[k1] = mk(w[k1].x << lz, w[k1].y << lz);
      } else {
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) w[k1] = mk(fx_shr(w[k1].x, -lz), fx_shr(w[k1].y, -lz));
      }
      DFT<R1, true, fxc>::run(w);
      int m = 0;
#pragma unroll
      for (int m1 = 0; m1 < R1; ++m1) {
        w[m1] = m1 == 0 ? fx_quarter(w[0]) : fx_twiddle<true>(w[m1], tw[n1 * m1]);
        m = fx_or(fx_or(m, w[m1].x), w[m1].y);
      }
      p = want_unit<R2>(u, m);
    }
    column_max<TC, NT>(unit[3 + q], p);
    __syncthreads();  // units known, every own slot of this buffer read
    const int U = unit[3 + q][c];
    if (n1 < R2) {
      to_unit<R1>(w, u, U);
#pragma unroll
      for (int m1 = 0; m1 < R1; ++m1) Fq[m1 * S1 + n1 * TC + c] = w[m1];
    }
    __syncthreads();
    fxc v[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = Fq[n1 * S1 + k2 * TC + c];
    DFT<R2, true, fxc>::run(v);
    if (colok)
      by_unit(plain_unit(U), [&](auto plain) {
#pragma unroll
        for (int m2 = 0; m2 < (PR ? R2 / 2 : R2); ++m2) {
          const int l = n1 + R1 * m2;
          if (PR != TB || (l >= a.olo && l < a.ohi)) col[q * cstride + l * zstride] = dbl_of<plain.value>(v[m2], U);
        }
      });
  }
}

// ---------------------------------------------------------------- x passes
// As xwide_kernel (passes_wide.cuh), with the transforms in fixed point.  The rows between the
// transforms are doubles in shared memory.
// SPLIT: each work item is one component of a tile (the passes that multiply by chi).  The power-law,
// assemble and update passes whose C2R is R1i 16 points are held to six CTAs an SM (168 registers): left alone
// they take 188 to 210 (64 x 64 x 96: update 89 us against 63, power law 117 against 107).
template <int CIN, int COUT, int R1i, int R2i, int R2o, bool SPLIT>
__global__ void __launch_bounds__(64, R1i <= 8 && R2i == 16 && CIN > 0 && COUT == 1 ? 6 : 0)
    xpass_kernel(const XArgs<double> a, const int4* __restrict__ tw_in, const int4* __restrict__ tw_out) {
  typedef WX<CIN, COUT, R1i, R2i, R2o> S;
  constexpr int TP = S::TP, P = S::P, NT = S::NT, XL = S::XL, TT = S::TT, Li = S::Li, Lo = S::Lo, R1o = S::R1o;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  if (a.check_done && a.ctrl->done) return;
  const UpdateArgs<double> up = update_args(a);
  int4* twi = reinterpret_cast<int4*>(smem_raw);  // [k2][n1]: the lanes of a pair read consecutive words
  int4* two = twi + S::TWI;
  double2* RS = reinterpret_cast<double2*>(two + S::TWO);  // [3][P][XL] real rows of the pairs
  fxc* Tb = reinterpret_cast<fxc*>(RS + 3 * P * XL);
  const int tid = threadIdx.x;
  const int p = tid / TP, r = tid % TP;
  for (int i = tid; i < S::TWI; i += NT) twi[i] = tw_in[(i % R1i) * (i / R1i)];
  for (int i = tid; i < S::TWO; i += NT) two[i] = tw_out[(i % R1o) * (i / R1o)];
  const int ny = a.g.ny, nz = a.g.nz;
  const long long N = a.g.N;
  const int hp = (a.use_box ? a.by1 - a.by0 : ny) >> 1;
  const int npairs = (a.use_box ? a.bz1 - a.bz0 : nz) * hp;
  const int ntiles = (npairs + P - 1) / P;
  fxc* Tp = Tb + p * TT;
  double part = 0.0;
  __syncthreads();
  for (int item = blockIdx.x; item < (SPLIT ? 3 * ntiles : ntiles); item += gridDim.x) {
    const int tile = SPLIT ? item / 3 : item;
    const int q0 = SPLIT ? item - 3 * tile : 0, q1 = SPLIT ? q0 + 1 : 3;
    const int gp = tile * P + p;
    const bool pok = gp < npairs;
    const int gq = pok ? gp : 0;
    const int zb = gq / hp;
    const int z = (a.use_box ? a.bz0 : 0) + zb, ya = (a.use_box ? a.by0 : 0) + 2 * (gq - zb * hp);
    const size_t na0 = ((size_t)z * ny + ya) * XL;  // first node of the pair's first row
    if constexpr (CIN > 0) {
#pragma unroll 1
      for (int q = q0; q < q1; ++q) {
        fxc v[R2i];
        int u = kNoUnit, want = kNoUnit;
        if (r < R1i) {
          const double2* ra = a.spec_in + ((size_t)(q * nz + z) * a.in_rows + ya) * a.in_sx;
          const double2* rb = ra + a.in_sx;
          int4 raw[R2i];
          int m = 0;
#pragma unroll
          for (int n2 = 0; n2 < R2i; ++n2) {
            // Z[k] = A[k] + i B[k], Z[L-k] = conj(A[k]) + i conj(B[k]); only the real parts of
            // DC and Nyquist are read
            const int k = r + R1i * n2;
            const bool lo = k <= Li / 2;
            const int kk = lo ? k : Li - k;
            double2 A = make_double2(0.0, 0.0), B = make_double2(0.0, 0.0);
            if (pok) { A = ra[kk]; B = rb[kk]; }
            if (kk == 0 || kk == Li / 2) { A.y = 0; B.y = 0; }
            raw[n2] = raw_of(lo ? make_double2(A.x - B.y, A.y + B.x) : make_double2(A.x + B.y, B.x - A.y));
            m = top_of(m, raw[n2]);
          }
          const int et = block_in<R2i, R2i>(v, raw, m);
          const bool some = m != 0;
          DFT<R2i, true, fxc>::run(v);
          u = fx_unit_of(et, fx_head(R2i)) + 2;
          m = 0;
#pragma unroll
          for (int k2 = 0; k2 < R2i; ++k2) {
            v[k2] = k2 == 0 ? fx_quarter(v[0]) : fx_twiddle<true>(v[k2], twi[k2 * R1i + r]);
            m = fx_or(fx_or(m, v[k2].x), v[k2].y);
          }
          if (some) want = want_unit<R1i>(u, m);
        }
#pragma unroll
        for (int o = 1; o < TP; o <<= 1) want = max(want, __shfl_xor_sync(0xffffffffu, want, o));
        if (r < R1i) {
          to_unit<R2i>(v, u, want);
#pragma unroll
          for (int k2 = 0; k2 < R2i; ++k2) Tp[k2 * (R1i + 1) + r] = v[k2];
        }
        __syncwarp();
        if (r < R2i) {
          fxc w[R1i];
#pragma unroll
          for (int i = 0; i < R1i; ++i) w[i] = Tp[r * (R1i + 1) + i];
          DFT<R1i, true, fxc>::run(w);
          by_unit(plain_unit(want), [&](auto plain) {
#pragma unroll
            for (int k1 = 0; k1 < S::KX; ++k1) RS[(q * P + p) * XL + r + R2i * k1] = dbl_of<plain.value>(w[k1], want);
          });
        }
        __syncwarp();
      }
      // the node-wise step on the nodes x = r + TP j of both rows of the lane's pair
      auto step = [&](int x) {
        double2 w[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) w[q] = RS[(q * P + p) * XL + x];
        double va[3] = {w[0].x, w[1].x, w[2].x}, vb[3] = {w[0].y, w[1].y, w[2].y};
        part += node_step<double>(a, up, na0 + x, va);
        part += node_step<double>(a, up, na0 + XL + x, vb);
        if (COUT > 0) {
#pragma unroll
          for (int q = 0; q < 3; ++q) RS[(q * P + p) * XL + x] = make_double2(va[q], vb[q]);
        }
      };
      if constexpr (SPLIT) {
        if (pok) {
          for (int x = r; x < XL; x += TP) {
            double2* w = RS + (q0 * P + p) * XL + x;
            if (!a.mask[na0 + x]) w->x = 0.0;
            if (!a.mask[na0 + XL + x]) w->y = 0.0;
          }
        }
      } else if (pok) {
#pragma unroll 1
        for (int x = r; x < XL; x += TP) step(x);
      }
      __syncwarp();
    } else {
#pragma unroll 1
      for (int q = 0; q < 3; ++q) {
        constexpr int J = XL / TP;
        double2 w[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const size_t na = na0 + r + TP * j, nb = na + XL;
          double va = 0, vb = 0;
          if (pok) {
            const size_t o = (size_t)q * N;
            const double* src = a.src_t ? a.src_t : a.src_f64;
            va = src[o + na];
            vb = src[o + nb];
            if (a.mode == X_ADJ_PAD) {  // (1 - chi)
              if (a.mask[na]) va = 0;
              if (a.mask[nb]) vb = 0;
            }
            if (a.mode == X_ADJ_IN) {  // chi
              if (!a.mask[na]) va = 0;
              if (!a.mask[nb]) vb = 0;
            }
          }
          w[j] = make_double2(va, vb);
        }
#pragma unroll
        for (int j = 0; j < J; ++j) RS[(q * P + p) * XL + r + TP * j] = w[j];
      }
      __syncwarp();
    }
    if constexpr (COUT > 0) {
#pragma unroll 1
      for (int q = q0; q < q1; ++q) {
        constexpr bool HALF = COUT == 2;
        constexpr int NL = HALF ? R2o / 2 : R2o;
        fxc v[R2o];
        int u = kNoUnit, want = kNoUnit;
        if (r < R1o) {
          int4 raw[NL];
          int m = 0;
#pragma unroll
          for (int n2 = 0; n2 < NL; ++n2) {
            raw[n2] = ld_raw(RS + (q * P + p) * XL + r + R1o * n2);
            m = top_of(m, raw[n2]);
          }
          const int et = block_in<R2o, NL>(v, raw, m);
          const bool some = m != 0;
          dft_maybe_half<R2o, false, HALF>(v);
          u = fx_unit_of(et, fx_head(R2o)) + 2;
          m = 0;
#pragma unroll
          for (int k2 = 0; k2 < R2o; ++k2) {
            v[k2] = k2 == 0 ? fx_quarter(v[0]) : fx_twiddle<false>(v[k2], two[k2 * R1o + r]);
            m = fx_or(fx_or(m, v[k2].x), v[k2].y);
          }
          if (some) want = want_unit<R1o>(u, m);
        }
#pragma unroll
        for (int o = 1; o < TP; o <<= 1) want = max(want, __shfl_xor_sync(0xffffffffu, want, o));
        if (r < R1o) {
          to_unit<R2o>(v, u, want);
#pragma unroll
          for (int k2 = 0; k2 < R2o; ++k2) Tp[k2 * (R1o + 1) + r] = v[k2];
        }
        __syncwarp();
        const int k2 = r;
        fxc Zr[R1o];
#pragma unroll
        for (int i = 0; i < R1o; ++i) Zr[i] = mk(0ll, 0ll);
        if (k2 < R2o) {
#pragma unroll
          for (int i = 0; i < R1o; ++i) Zr[i] = Tp[k2 * (R1o + 1) + i];
          DFT<R1o, false, fxc>::run(Zr);
        }
        // separate the two rows: A = (Z[k] + conj Z[Lo-k])/2, B = (Z[k] - conj Z[Lo-k])/(2i).
        // Thread k2 holds Z[k2 + R2o k1]; the mirror Lo - k lives in thread R2o - k2 at register
        // R1o - 1 - k1 (k2 > 0) or in this thread at (R1o - k1) mod R1o (k2 = 0).
        const int lane = tid & 31;
        const int src = lane - k2 + (k2 == 0 ? 0 : (k2 < R2o ? R2o - k2 : k2));
        double2* ra = a.spec_out + ((size_t)(q * nz + z) * a.out_rows + ya) * a.out_sx;
        double2* rb = ra + a.out_sx;
        by_unit(__all_sync(0xffffffffu, plain_unit(want - 1)), [&](auto plain) {  // (the lanes shuffle together)
#pragma unroll
          for (int k1 = 0; k1 <= R1o / 2; ++k1) {
            const fxc sh = shfl_fx(Zr[R1o - 1 - k1], src);
            const fxc Zk = Zr[k1];
            const fxc Zm = k2 == 0 ? Zr[(R1o - k1) % R1o] : sh;
            const int k = k2 + R2o * k1;
            if (k2 < R2o && pok && k <= Lo / 2) {
              ra[k] = dbl_of<plain.value>(mk(Zk.x + Zm.x, Zk.y - Zm.y), want - 1);
              rb[k] = dbl_of<plain.value>(mk(Zk.y + Zm.y, Zm.x - Zk.x), want - 1);
            }
          }
        });
        __syncwarp();  // the next component's first stage overwrites Tp
      }
    }
    __syncwarp();  // the pair's rows are reused by the next tile
  }
  if (CIN == 2 && a.mode == X_UPDATE) residual_finish<NT>(a, part, up.it);
  if (CIN == 1 && a.mode == X_ASSEMBLE && blockIdx.x == 0 && tid == 0) begin_loop(a);
}

// ---------------------------------------------------------------- launchers
template <int CIN, int COUT, int R1i, int R2i, int R2o, bool SPLIT = false>
cudaError_t go_x(const Launch<double>& L, const XArgs<double>& a) {
  typedef WX<CIN, COUT, R1i, R2i, R2o> S;
  if constexpr (S::MASKS && !SPLIT)
    if (a.comp_split) return go_x<CIN, COUT, R1i, R2i, R2o, true>(L, a);
  constexpr auto k = xpass_kernel<CIN, COUT, R1i, R2i, R2o, SPLIT>;
  const size_t smem = sizeof(fxc) * S::SM;
  allow_smem<k>();
  static const int resident = wide::resident_ctas(k, S::NT, smem);
  const int hp = (a.use_box ? a.by1 - a.by0 : a.g.ny) / 2;
  const int ntiles = ((a.use_box ? a.bz1 - a.bz0 : a.g.nz) * hp + S::P - 1) / S::P * (SPLIT ? 3 : 1);
  const int grid = ntiles < resident ? ntiles : resident;
  const Work<double>& w = *L.w;
  launch_chained(k, dim3(grid), S::NT, smem, L.st, a, CIN == 2 ? w.fxp[0] : w.fxu[0], COUT == 2 ? w.fxp[0] : w.fxu[0]);
  return checked_launch("fx xpass_kernel", dim3(grid), S::NT, smem);
}
template <int CIN, int COUT> cudaError_t go_x_n(const Launch<double>& L, const XArgs<double>& a) {
#define XN(NN, A_, B_, C_, D_)                                                                                  \
  case NN:                                                                                                      \
    if constexpr (CIN == 0) return go_x<CIN, COUT, 1, B_, COUT == 2 ? 2 * A_ : A_>(L, a);                       \
    else if constexpr (CIN == 1) return go_x<CIN, COUT, A_, B_, COUT == 2 ? 2 * A_ : COUT == 1 ? A_ : 1>(L, a); \
    else return go_x<CIN, COUT, C_, D_, COUT == 1 ? C_ / 2 : 1>(L, a);
  switch (a.g.nx) {
    XN(16, 4, 4, 8, 4)
    XN(32, 4, 8, 8, 8)
    XN(48, 4, 12, 8, 12)
    XN(64, 4, 16, 8, 16)
    XN(96, 8, 12, 16, 12)
    XN(128, 8, 16, 16, 16)
  }
#undef XN
  return cudaErrorInvalidValue;
}

}  // namespace fx
}  // namespace scfft
