// passes_small.cuh - the FP64 passes of small grids (every axis at most 32: transforms of 16, 32
// and 64 points), in native FP64.
//
// What bounds them is the depth of a warp's instruction stream: an FP64 instruction of a warp
// takes its quarter of the SM 64 clocks whatever its lanes do, and a 16^3 grid has fewer warps of
// whole transforms than the GPU has quarters (608).  So the points of a transform lie in the lanes
// of a warp, one to a lane (two for 64 points), and a butterfly is a shuffle and one instruction
// for each part: 16 points are about 16 FP64 instructions deep, 32 points 18, against 160 and 116
// for a thread that transforms 16 or 8 points in its registers.  Measured on 16^3: one curl 55.3 ->
// 22.3 us, an adaptive run 42.3 -> 23.1 ms (12.1 us and 12.7 ms since the passes follow each other as
// dependent launches and the Eq. 5 loop is a graph).  The y and z passes of 64 points (32^3 and its like on the
// padded grid) have enough warps, so what counts is the number of instructions, about 17 a
// point with 8 points to a thread against 24 in lanes, and they keep that form.
// The operations are those of the register transforms (fft_core.cuh: 16 = 4 x 4, 32 = 4 x 8,
// 64 = 8 x 8), fused multiply-adds included, in the same order: a small grid's step sequence
// depends on the last bits of its error estimates, and stays what it was.
#pragma once
#include "passes_wide.cuh"

namespace scfft {
namespace small {

// ---------------------------------------------------------------- transforms across lanes
__device__ __forceinline__ double neg_if(double v, bool f) {  // (an integer instruction)
  return __hiloint2double(__double2hiint(v) ^ (f ? (int)0x80000000 : 0), __double2loint(v));
}
__device__ __forceinline__ bool bit(int e, int i) { return (e >> i) & 1; }
// v times -i (forward) or +i (inverse) where on is set
template <bool INV> __device__ __forceinline__ double2 rot_if(double2 v, bool on) {
  const double x = on ? v.y : v.x, y = on ? v.x : v.y;
  return INV ? mk(neg_if(x, on), y) : mk(x, neg_if(y, on));
}
// The products of the register transforms by h = sqrt(1/2) are fused into the sums that take them;
// here a value that still lacks its h goes through the butterfly, which multiplies.
constexpr double kSqrtHalf = 0.7071067811865475244008444;
// v W_8^1, or W_8^3 (three), without the factor h
template <bool INV> __device__ __forceinline__ double2 turn8(double2 v, bool three) {
  const double x = neg_if(v.x, three), y = neg_if(v.y, three);
  return INV ? mk(x - v.y, v.x + y) : mk(x + v.y, y - v.x);
}
// sum in the lane whose bit is clear, difference in the lane whose bit is set; odd: the value of
// the lane whose bit is set lacks its factor h
__device__ __forceinline__ double2 butterfly(double2 v, int mask, bool hi, bool odd = false) {
  const double2 w = mk(__shfl_xor_sync(0xffffffffu, v.x, mask), __shfl_xor_sync(0xffffffffu, v.y, mask));
  const double m = neg_if(odd ? kSqrtHalf : 1.0, hi);
  const double2 p = odd && !hi ? w : v, q = odd && !hi ? v : w;
  return mk(fma(p.x, m, q.x), fma(p.y, m, q.y));
}
// 4-point transform over the bits hi, lo of e; lane bit = bit + SH
template <bool INV, int SH> __device__ __forceinline__ double2 lane4(double2 v, int e, int hi, int lo) {
  v = butterfly(v, 1 << (hi + SH), bit(e, hi));
  v = rot_if<INV>(v, bit(e, hi) && bit(e, lo));
  return butterfly(v, 1 << (lo + SH), bit(e, lo));
}
// the last stage of an 8-point transform: W_8^(n1 k1), then the sum or difference over n1
template <bool INV, int SH> __device__ __forceinline__ double2 last8(double2 v, int lane_bit, bool n1, int k1) {
  v = rot_if<INV>(v, n1 && k1 == 2);
  if (n1 && (k1 & 1)) v = turn8<INV>(v, k1 == 3);
  return butterfly(v, 1 << (lane_bit + SH), n1, k1 & 1);
}
// 8-point transform over three bits of e from hi down
template <bool INV, int SH> __device__ __forceinline__ double2 lane8(double2 v, int e, int hi) {
  v = lane4<INV, SH>(v, e, hi, hi - 1);
  return last8<INV, SH>(v, hi - 2, bit(e, hi - 2), (int)bit(e, hi) + 2 * (int)bit(e, hi - 1));
}

// Transform of L points, one (16, 32) or two (64: points e and e + 32) to a lane.  A lane holds the
// point of index e and gets that of index out(e), the bits of e reversed.  16 points: SH is 1 for
// two transforms side by side in a warp (lane 2 e + c), or 0 (the lanes e and e + 16 do the same).
template <int L> struct Lanes {
  static constexpr int E = L == 64 ? 2 : 1, LB = L == 16 ? 4 : L == 32 ? 5 : 6;
  static __device__ __forceinline__ int out(int e) { return (int)(__brev((unsigned)e) >> (32 - LB)); }
  // the index of point e in the table of twiddles W_L^m between the two factors (32, 64)
  static __device__ __forceinline__ int twiddle(int e) {
    return L == 32 ? (e & 3) * (int)(__brev((unsigned)e >> 2) >> 29) : (e & 7) * (int)(__brev((unsigned)e >> 3) >> 29);
  }
  // tw: the point's twiddle W_L^twiddle(e) (32, 64)
  template <bool INV, int SH = 0> static __device__ __forceinline__ void run(double2* v, int e, const double2* tw) {
    if constexpr (L == 16) {
      double2 a = lane4<INV, SH>(v[0], e, 3, 2);
      const int n1 = e & 3, k1 = (int)bit(e, 3) + 2 * (int)bit(e, 2), m = n1 * k1;  // 0, 1, 2, 3, 4, 6, 9
      a = rot_if<INV>(a, m == 4);
      if (m == 2 || m == 6) a = turn8<INV>(a, m == 6);
      if (m & 1) {
        const double c1 = 0.9238795325112867561281832, s1 = 0.3826834323650897717284600;  // pi / 8
        const double c = neg_if(m == 3 ? s1 : c1, m == 9), s = neg_if(m == 3 ? c1 : s1, m == 9);
        a = INV ? mk(fma(a.x, c, -(a.y * s)), fma(a.y, c, a.x * s)) : mk(fma(a.x, c, a.y * s), fma(a.y, c, -(a.x * s)));
      }
      // over the high bit of n1; points 1 and 3 both lack their h when k1 is 2
      const bool hi = bit(e, 1), both = (n1 & 1) && k1 == 2;
      const double2 w = mk(__shfl_xor_sync(0xffffffffu, a.x, 2 << SH), __shfl_xor_sync(0xffffffffu, a.y, 2 << SH));
      if (both) {  // h (v1 +- v3), as fma(h, v1, +-(h v3))
        const double2 one = hi ? w : a, three = hi ? a : w;
        a = mk(fma(one.x, kSqrtHalf, neg_if(three.x * kSqrtHalf, hi)), fma(one.y, kSqrtHalf, neg_if(three.y * kSqrtHalf, hi)));
      } else {
        const bool odd = n1 % 2 == 0 && (k1 & 1);
        const double f = neg_if(odd ? kSqrtHalf : 1.0, hi);
        const double2 p = odd && !hi ? w : a, q = odd && !hi ? a : w;
        a = mk(fma(p.x, f, q.x), fma(p.y, f, q.y));
      }
      a = rot_if<INV>(a, hi && bit(e, 0));
      v[0] = butterfly(a, 1 << SH, bit(e, 0));
    } else if constexpr (L == 32) {
      double2 a = lane8<INV, 0>(v[0], e, 4);
      if (twiddle(e)) a = INV ? cmulc(a, tw[0]) : cmul(a, tw[0]);
      v[0] = lane4<INV, 0>(a, e, 1, 0);
    } else {
      // the top bit of the index is the point within the lane
      double2 p[2] = {v[0] + v[1], v[0] - v[1]};
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int f = e + 32 * r;
        double2 a = rot_if<INV>(p[r], r == 1 && bit(e, 4));
        a = butterfly(a, 16, bit(e, 4));
        a = last8<INV, 0>(a, 3, bit(e, 3), r + 2 * (int)bit(e, 4));
        if (twiddle(f)) a = INV ? cmulc(a, tw[r]) : cmul(a, tw[r]);
        v[r] = lane8<INV, 0>(a, e, 2);
      }
    }
  }
};

// ---------------------------------------------------------------- x passes
// One CTA of three warps per row pair, a component to a warp; the node-wise step on the nodes of
// both rows.
template <int CIN, int COUT, int NX>
__global__ void __launch_bounds__(96) xpass_kernel(const XArgs<double> a) {
  constexpr int Li = CIN == 2 ? 2 * NX : NX, Lo = COUT == 2 ? 2 * NX : NX;
  typedef Lanes<Li> FI;
  typedef Lanes<Lo> FO;
  __shared__ __align__(16) double2 RS[CIN ? 3 : 1][CIN ? NX : 1];       // real rows of the pair, as complex values
  __shared__ __align__(16) double2 Z[COUT ? 3 : 1][COUT ? Lo : 1];
  after_previous();
  const int done = a.check_done ? a.ctrl->done : 0;  // (looked at once the input is on its way)
  const UpdateArgs<double> up = update_args(a);
  const int t = threadIdx.x, lane = t & 31, q = t >> 5;
  const int ny = a.g.ny, nz = a.g.nz;
  const long long N = a.g.N;
  const int hp = (a.use_box ? a.by1 - a.by0 : ny) >> 1;
  const int zb = blockIdx.x / hp;
  const int z = (a.use_box ? a.bz0 : 0) + zb, ya = (a.use_box ? a.by0 : 0) + 2 * ((int)blockIdx.x - zb * hp);
  const size_t na0 = ((size_t)z * ny + ya) * NX;
  double part = 0.0;
  const int eo = lane & (Lo - 1);
  double2 two[FO::E], vo[FO::E];
#pragma unroll
  for (int r = 0; r < FO::E; ++r) {
    two[r] = vo[r] = mk(0.0, 0.0);
    if (COUT && Lo > 16) two[r] = a.tw_out[FO::twiddle(eo + 32 * r)];
  }
  if constexpr (CIN > 0) {
    const double2* ra = a.spec_in + ((size_t)(q * nz + z) * a.in_rows + ya) * a.in_sx;
    const double2* rb = ra + a.in_sx;
    const int e = lane & (Li - 1);
    double2 v[FI::E], tw[FI::E], A[FI::E], B[FI::E];
#pragma unroll
    for (int r = 0; r < FI::E; ++r) {
      const int k = e + 32 * r, kk = k <= Li / 2 ? k : Li - k;
      A[r] = ra[kk];
      B[r] = rb[kk];
      tw[r] = mk(0.0, 0.0);
      if (Li > 16) tw[r] = a.tw_in[FI::twiddle(k)];
    }
    if (done) return;
#pragma unroll
    for (int r = 0; r < FI::E; ++r) {
      // Z[k] = A[k] + i B[k], Z[L-k] = conj(A[k]) + i conj(B[k]); only the real parts of DC and
      // Nyquist are read
      const int k = e + 32 * r;
      if (k == 0 || k == Li / 2) { A[r].y = 0; B[r].y = 0; }
      v[r] = k <= Li / 2 ? mk(A[r].x - B[r].y, A[r].y + B[r].x) : mk(A[r].x + B[r].y, B[r].x - A[r].y);
    }
    FI::template run<true>(v, e, tw);
#pragma unroll
    for (int r = 0; r < FI::E; ++r) {
      const int x = FI::out(e + 32 * r);
      if (x < NX && lane < Li) RS[q][x] = v[r];
    }
    __syncthreads();
#pragma unroll 1
    for (int i = t; i < 2 * NX; i += 96) {
      const int r = i / NX, x = i - r * NX;
      double* p[3];
      double w[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        p[c] = &RS[c][x].x + r;
        w[c] = *p[c];
      }
      part += node_step<double>(a, up, na0 + i, w);
      if (COUT > 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) *p[c] = w[c];
      }
    }
    if constexpr (COUT > 0) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < FO::E; ++r)
        if (eo + 32 * r < NX) vo[r] = RS[q][eo + 32 * r];
    }
  } else {
#pragma unroll
    for (int r = 0; r < FO::E; ++r) {
      if (eo + 32 * r < NX) {
        const size_t na = na0 + eo + 32 * r, nb = na + NX, o = (size_t)q * N;
        const double* src = a.src_t ? a.src_t : a.src_f64;
        double va = src[o + na], vb = src[o + nb];
        if (a.mode == X_ADJ_PAD) {  // (1 - chi)
          if (a.mask[na]) va = 0;
          if (a.mask[nb]) vb = 0;
        }
        if (a.mode == X_ADJ_IN) {  // chi
          if (!a.mask[na]) va = 0;
          if (!a.mask[nb]) vb = 0;
        }
        vo[r] = mk(va, vb);
      }
    }
    if (done) return;
  }
  if constexpr (COUT > 0) {
    FO::template run<false>(vo, eo, two);
#pragma unroll
    for (int r = 0; r < FO::E; ++r)
      if (lane < Lo) Z[q][FO::out(eo + 32 * r)] = vo[r];
    __syncwarp();
    // the two rows' spectra, one of both to a thread: A = (Z[k] + conj Z[Lo-k])/2, B = (Z[k] - conj Z[Lo-k])/(2i)
    constexpr int H = Lo / 2 + 1;
    double2* ra = a.spec_out + ((size_t)(q * nz + z) * a.out_rows + ya) * a.out_sx;
    for (int i = lane; i < 2 * H; i += 32) {
      const bool second = i >= H;
      const int k = second ? i - H : i;
      const double2 Zk = Z[q][k], Zm = Z[q][(Lo - k) % Lo];
      ra[(second ? a.out_sx : 0) + k] =
          second ? mk((Zk.y + Zm.y) * 0.5, (Zm.x - Zk.x) * 0.5) : mk((Zk.x + Zm.x) * 0.5, (Zk.y - Zm.y) * 0.5);
    }
  }
  if (CIN == 2 && a.mode == X_UPDATE) residual_finish<96>(a, part, up.it);
  if (CIN == 1 && a.mode == X_ASSEMBLE && blockIdx.x == 0 && t == 0) begin_loop(a);
}

// ---------------------------------------------------------------- 64 points, 8 to a thread
// 8-point transforms over n2 (n = n1 + 8 n2) and their twiddles, into T[k2 8 + n1]
template <bool INV, bool HALF>
__device__ __forceinline__ void stage_a(double2* v, int n1, const double2* tw, double2* T, int ts) {
  dft_maybe_half<8, INV, HALF>(v);
#pragma unroll
  for (int k2 = 0; k2 < 8; ++k2) {
    double2 w = v[k2];
    if (k2 > 0 && n1 > 0) w = INV ? cmulc(w, tw[n1 * k2]) : cmul(w, tw[n1 * k2]);
    T[(k2 * 8 + n1) * ts] = w;
  }
}
// 8-point transforms over n1: the points k2 + 8 k1, k1 < 8, into w
template <bool INV> __device__ __forceinline__ void stage_b(double2* w, int k2, const double2* T, int ts) {
#pragma unroll
  for (int m = 0; m < 8; ++m) w[m] = T[(k2 * 8 + m) * ts];
  DFT<8, INV, double2>::run(w);
}

// ---------------------------------------------------------------- y passes
struct YArgs {
  double2* base;
  int rows, sx, HX, nzs, planes;
  const double2* tw;
  const Ctrl* ctrl;
  int check_done;
  // planes from zoff; rows outside [ylo, yhi): the forward pass reads them as zero, the inverse
  // pass need not write them
  int zoff, ylo, yhi;
};
// 16 and 32 points: one warp a CTA, two or one columns (component, plane, kx).
template <int L, bool INV, bool PAD> __global__ void __launch_bounds__(32) ypass_lanes_kernel(const YArgs a) {
  constexpr int C = 32 / L, SH = C == 2 ? 1 : 0;
  after_previous();
  const int done = a.check_done ? a.ctrl->done : 0;
  const int c = threadIdx.x % C, row = threadIdx.x / C;
  const int i = blockIdx.x * C + c;
  const bool ok = i < 3 * a.planes * a.HX;
  const int pl = ok ? i / a.HX : 0, kx = ok ? i - pl * a.HX : 0;
  const int q = pl / a.planes, z = a.zoff + pl - q * a.planes;
  double2* col = a.base + ((size_t)(q * a.nzs + z) * a.rows) * a.sx + kx;
  double2 v = mk(0.0, 0.0), tw = mk(0.0, 0.0);
  if (!(PAD && !INV && row >= L / 2) && ok && (INV || (row >= a.ylo && row < a.yhi))) v = col[(size_t)row * a.sx];
  if (L > 16) tw = a.tw[Lanes<L>::twiddle(row)];
  if (done) return;
  Lanes<L>::template run<INV, SH>(&v, row, &tw);
  const int o = Lanes<L>::out(row);
  if (ok && (!INV || (o >= a.ylo && o < a.yhi && (!PAD || o < L / 2)))) col[(size_t)o * a.sx] = v;
}
// 64 points: 32-thread CTAs, 8 threads a column and 8 points a thread.
template <bool INV, bool PAD> __global__ void __launch_bounds__(32) ypass64_kernel(const YArgs a) {
  constexpr int L = 64, TC = 4;
  constexpr bool HALF = PAD && !INV;
  __shared__ __align__(16) double2 tw[L], T[L * TC];
  after_previous();
  if (a.check_done && a.ctrl->done) return;
  const int t = threadIdx.x, c = t % TC, n1 = t / TC;
  const int e = blockIdx.x * TC + c;
  const bool ok = e < 3 * a.planes * a.HX;
  const int pl = ok ? e / a.HX : 0, kx = ok ? e - pl * a.HX : 0;
  const int q = pl / a.planes, z = a.zoff + pl - q * a.planes;
  double2* col = a.base + ((size_t)(q * a.nzs + z) * a.rows) * a.sx + kx;
  double2 v[8];
#pragma unroll
  for (int n2 = 0; n2 < 8; ++n2) {
    const int row = n1 + 8 * n2;
    v[n2] = (!(HALF && n2 >= 4) && ok && (INV || (row >= a.ylo && row < a.yhi))) ? col[(size_t)row * a.sx]
                                                                                 : mk(0.0, 0.0);
  }
  for (int i = t; i < L; i += 32) tw[i] = a.tw[i];
  __syncwarp();
  stage_a<INV, HALF>(v, n1, tw, T + c, TC);
  __syncwarp();
  stage_b<INV>(v, n1, T + c, TC);
  if (ok) {
#pragma unroll
    for (int k1 = 0; k1 < (PAD && INV ? 4 : 8); ++k1) col[(size_t)(n1 + 8 * k1) * a.sx] = v[k1];
  }
}

// ---------------------------------------------------------------- z passes
struct ZArgs {
  double2* base;
  int rows, sx, HX, nzs;
  const double2* tw;
  const double *kt0, *kt1, *kt2, *st0, *st1, *st2;  // curl
  double scale;
  const double* kap;  // kernel
  int nx, ny, nz;
  const Ctrl* ctrl;
  int check_done;
  int ilo, ihi, olo, ohi;  // planes outside [ilo, ihi) read as zero, planes outside [olo, ohi) need not be written
};
// 16 and 32 points: one CTA of three warps, a component to a warp, for two or one columns (kx, y);
// the three spectra meet in shared memory, where each thread takes the product of its own component.
template <int L, int KIND> __global__ void __launch_bounds__(96) zpass_lanes_kernel(const ZArgs a) {
  constexpr int C = 32 / L, SH = C == 2 ? 1 : 0;
  constexpr bool PR = KIND == 1;
  __shared__ __align__(16) double2 F[3][32];
  after_previous();
  const int done = a.check_done ? a.ctrl->done : 0;
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int c = lane % C, l = lane / C;
  const int i = blockIdx.x * C + c;
  const bool ok = i < a.rows * a.HX;
  const int y = ok ? i / a.HX : 0, kx = ok ? i - y * a.HX : 0;
  const size_t zstride = (size_t)a.rows * a.sx;
  double2* col = a.base + (size_t)q * a.nzs * zstride + (size_t)y * a.sx + kx;
  double2 v = mk(0.0, 0.0), tw = mk(0.0, 0.0);
  if (!(PR && l >= L / 2) && ok && l >= a.ilo && l < a.ihi) v = col[l * zstride];
  if (L > 16) tw = a.tw[Lanes<L>::twiddle(l)];
  // the factors of the product i s (k x F): the two that this component takes
  const int qb = q == 2 ? 0 : q + 1, qc = q == 0 ? 2 : q - 1;
  double k[3], s = 1.0;
  if (!PR) {
    k[0] = a.kt0[kx]; k[1] = a.kt1[y]; k[2] = a.kt2[l];
    s = a.st0[kx] * a.st1[y] * a.st2[l] * a.scale;
  } else {
    const int fy = (y <= a.ny) ? y : 2 * a.ny - y;
    const int fz = (l <= a.nz) ? l : 2 * a.nz - l;
    const size_t oct = (size_t)(a.nz + 1) * (a.ny + 1) * (a.nx + 1);
    const size_t off = ((size_t)fz * (a.ny + 1) + fy) * (a.nx + 1) + kx;
    k[0] = a.kap[off];
    k[1] = neg_if(a.kap[oct + off], y > a.ny);
    k[2] = neg_if(a.kap[2 * oct + off], l > a.nz);
  }
  if (done) return;
  Lanes<L>::template run<false, SH>(&v, l, &tw);
  const int o = Lanes<L>::out(l);
  F[q][o * C + c] = v;
  __syncthreads();
  const double kb = qb == 0 ? k[0] : qb == 1 ? k[1] : k[2], kc = qc == 0 ? k[0] : qc == 1 ? k[1] : k[2];
  const double2 Fb = F[qb][lane], Fc = F[qc][lane];
  const double2 x = mk(kb * Fc.x - kc * Fb.x, kb * Fc.y - kc * Fb.y);
  v = PR ? mk(-x.y, x.x) : mk(-s * x.y, s * x.x);
  Lanes<L>::template run<true, SH>(&v, l, &tw);
  if (ok && o >= a.olo && o < a.ohi && (!PR || o < L / 2)) col[o * zstride] = v;
}
// 64 points (always the padded pass): four columns (kx, y) a CTA, its threads over (component,
// residue, column), 8 points a thread; the product over the spectra in shared memory.
__global__ void __launch_bounds__(96) zpass64_kernel(const ZArgs a) {
  constexpr int L = 64, TC = 4, NT = 96;
  __shared__ __align__(16) double2 tw[L], T[3][L * TC], F[3][L * TC];
  after_previous();
  if (a.check_done && a.ctrl->done) return;
  const int t = threadIdx.x, c = t % TC, n1 = (t / TC) % 8, q = t / (TC * 8);
  const int ncol = a.rows * a.HX;
  auto column = [&](int i, int& y, int& kx) {
    const int e = blockIdx.x * TC + i;
    const bool ok = e < ncol;
    y = ok ? e / a.HX : 0;
    kx = ok ? e - y * a.HX : 0;
    return ok;
  };
  int y, kx;
  const bool ok = column(c, y, kx);
  const size_t zstride = (size_t)a.rows * a.sx;
  double2* col = a.base + (size_t)q * a.nzs * zstride + (size_t)y * a.sx + kx;
  double2 v[8];
#pragma unroll
  for (int n2 = 0; n2 < 8; ++n2) {
    const int l = n1 + 8 * n2;
    v[n2] = (n2 < 4 && ok && l >= a.ilo && l < a.ihi) ? col[l * zstride] : mk(0.0, 0.0);
  }
  for (int i = t; i < L; i += NT) tw[i] = a.tw[i];
  __syncthreads();
  stage_a<false, true>(v, n1, tw, T[q] + c, TC);
  __syncthreads();
  stage_b<false>(v, n1, T[q] + c, TC);
#pragma unroll
  for (int k1 = 0; k1 < 8; ++k1) F[q][(n1 + 8 * k1) * TC + c] = v[k1];
  __syncthreads();
#pragma unroll 1
  for (int i = t; i < L * TC; i += NT) {
    const int l = i / TC;
    int py, pk;
    if (!column(i - l * TC, py, pk)) continue;
    const double2 F0 = F[0][i], F1 = F[1][i], F2 = F[2][i];
    const int fy = (py <= a.ny) ? py : 2 * a.ny - py;
    const int fz = (l <= a.nz) ? l : 2 * a.nz - l;
    const size_t oct = (size_t)(a.nz + 1) * (a.ny + 1) * (a.nx + 1);
    const size_t off = ((size_t)fz * (a.ny + 1) + fy) * (a.nx + 1) + pk;
    const double ax = a.kap[off], ay = neg_if(a.kap[oct + off], py > a.ny),
                 az = neg_if(a.kap[2 * oct + off], l > a.nz);
    // G = i (K^ x F)
    F[0][i] = mk(-(ay * F2.y - az * F1.y), ay * F2.x - az * F1.x);
    F[1][i] = mk(-(az * F0.y - ax * F2.y), az * F0.x - ax * F2.x);
    F[2][i] = mk(-(ax * F1.y - ay * F0.y), ax * F1.x - ay * F0.x);
  }
  __syncthreads();
#pragma unroll
  for (int n2 = 0; n2 < 8; ++n2) v[n2] = F[q][(n1 + 8 * n2) * TC + c];
  stage_a<true, false>(v, n1, tw, T[q] + c, TC);
  __syncthreads();
  stage_b<true>(v, n1, T[q] + c, TC);
  if (ok) {
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) col[(n1 + 8 * k1) * zstride] = v[k1];
  }
}

}  // namespace small
}  // namespace scfft
