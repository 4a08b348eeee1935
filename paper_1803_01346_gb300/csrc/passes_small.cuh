// passes_small.cuh - the FP64 passes of small grids (every axis at most 32: transforms of 16, 32
// and 64 points), in native FP64.
//
// These passes are bound by latency: an FP64 instruction of a warp takes 64 clocks whatever its
// lanes do, and the fixed point of passes_fx.cuh is about as slow here through its longer code
// (16^3, us, these | fixed point: Eq. 5 update 18 | 22, mask and pad 16 | 18, kernel z 16 | 15, curl z 22 | 14;
// 18 to 27 before, with one shared-memory kernel for every length).  Their operations are those of
// that kernel in the same order: a small grid's step sequence depends on the last bits of its error
// estimates, and stays what it was.  The three components run side by side (in the lanes of a
// warp in the x passes, in thread groups in the z passes) instead of one after another, work is
// cut into many one- to three-warp CTAs, and a length is one or two register stages: 16 = one
// 16-point transform, 32 = 8 x 4, 64 = 8 x 8 (first factor first).
#pragma once
#include "passes_wide.cuh"

namespace scfft {
namespace small {

// Stage A: R2-point transforms over n = n1 + R1 n2, stage B: R1-point transforms.
template <int L> struct Split;
template <> struct Split<16> { static constexpr int R1 = 1, R2 = 16; };
template <> struct Split<32> { static constexpr int R1 = 4, R2 = 8; };
template <> struct Split<64> { static constexpr int R1 = 8, R2 = 8; };

// Stage A of one pencil's residue n1 on v (its R2 points), into T[k2 R1 + n1].
template <int L, bool INV, bool HALF>
__device__ __forceinline__ void stage_a(double2* v, int n1, const double2* tw, double2* T, int ts) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2;
  dft_maybe_half<R2, INV, HALF>(v);
#pragma unroll
  for (int k2 = 0; k2 < R2; ++k2) {
    double2 w = v[k2];
    if (R1 > 1 && k2 > 0 && n1 > 0) w = INV ? cmulc(w, tw[n1 * k2]) : cmul(w, tw[n1 * k2]);
    T[(k2 * R1 + n1) * ts] = w;
  }
}
// Stage B: the pencil's points k2 + R2 k1, k1 < R1, into w.
template <int L, bool INV> __device__ __forceinline__ void stage_b(double2* w, int k2, const double2* T, int ts) {
  constexpr int R1 = Split<L>::R1;
#pragma unroll
  for (int m = 0; m < R1; ++m) w[m] = T[(k2 * R1 + m) * ts];
  if constexpr (R1 > 1) DFT<R1, INV, double2>::run(w);
}

// ---------------------------------------------------------------- x passes
// One warp per row pair, the lanes over (component, residue) in the transforms and over the nodes
// of both rows in the node-wise step.
template <int CIN, int COUT, int NX>
__global__ void __launch_bounds__(32) xpass_kernel(const XArgs<double> a) {
  constexpr int Li = CIN == 2 ? 2 * NX : NX, Lo = COUT == 2 ? 2 * NX : NX;
  constexpr int A1 = Split<Li>::R1, A2 = Split<Li>::R2, B1 = Split<Lo>::R1, B2 = Split<Lo>::R2;
  constexpr int LM = Li > Lo ? Li : Lo;
  __shared__ __align__(16) double2 RS[3][NX];  // real rows of the pair, as complex values
  __shared__ __align__(16) double2 T[3][LM], Z[COUT ? 3 : 1][COUT ? Lo : 1];
  __shared__ __align__(16) double2 twi[Li], two[Lo];
  if (a.check_done && a.ctrl->done) return;
  const int lane = threadIdx.x;
  const int ny = a.g.ny, nz = a.g.nz;
  const long long N = a.g.N;
  const int hp = (a.use_box ? a.by1 - a.by0 : ny) >> 1;
  const int zb = blockIdx.x / hp;
  const int z = (a.use_box ? a.bz0 : 0) + zb, ya = (a.use_box ? a.by0 : 0) + 2 * ((int)blockIdx.x - zb * hp);
  const size_t na0 = ((size_t)z * ny + ya) * NX;
  double part = 0.0;
  if (CIN && A1 > 1)
    for (int i = lane; i < Li; i += 32) twi[i] = a.tw_in[i];
  if (COUT && B1 > 1)
    for (int i = lane; i < Lo; i += 32) two[i] = a.tw_out[i];
  if constexpr (CIN > 0) {
    __syncwarp();
    if (lane < 3 * A1) {
      const int q = lane / A1, n1 = lane - q * A1;
      const double2* ra = a.spec_in + ((size_t)(q * nz + z) * a.in_rows + ya) * a.in_sx;
      const double2* rb = ra + a.in_sx;
      double2 v[A2];
#pragma unroll
      for (int n2 = 0; n2 < A2; ++n2) {
        // Z[k] = A[k] + i B[k], Z[L-k] = conj(A[k]) + i conj(B[k]); only the real parts of DC and
        // Nyquist are read
        const int k = n1 + A1 * n2;
        const bool lo = k <= Li / 2;
        const int kk = lo ? k : Li - k;
        double2 A = ra[kk], B = rb[kk];
        if (kk == 0 || kk == Li / 2) { A.y = 0; B.y = 0; }
        v[n2] = lo ? mk(A.x - B.y, A.y + B.x) : mk(A.x + B.y, B.x - A.y);
      }
      stage_a<Li, true, false>(v, n1, twi, T[q], 1);
    }
    __syncwarp();
    for (int i = lane; i < 3 * A2; i += 32) {
      const int q = i / A2, k2 = i - q * A2;
      double2 w[A1];
      stage_b<Li, true>(w, k2, T[q], 1);
#pragma unroll
      for (int k1 = 0; k1 < A1; ++k1)
        if (k2 + A2 * k1 < NX) RS[q][k2 + A2 * k1] = w[k1];
    }
    __syncwarp();
#pragma unroll 1
    for (int i = lane; i < 2 * NX; i += 32) {
      const int r = i / NX, x = i - r * NX;
      double* p[3];
      double v[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        p[q] = &RS[q][x].x + r;
        v[q] = *p[q];
      }
      part += node_step<double>(a, na0 + i, v);
      if (COUT > 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q) *p[q] = v[q];
      }
    }
  } else {
#pragma unroll
    for (int i = lane; i < 3 * NX; i += 32) {
      const int q = i / NX, x = i - q * NX;
      const size_t na = na0 + x, nb = na + NX, o = (size_t)q * N;
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
      RS[q][x] = mk(va, vb);
    }
  }
  __syncwarp();
  if constexpr (COUT > 0) {
    if (lane < 3 * B1) {
      const int q = lane / B1, n1 = lane - q * B1;
      double2 v[B2];
#pragma unroll
      for (int n2 = 0; n2 < B2; ++n2)
        v[n2] = (COUT == 2 && n2 >= B2 / 2) ? mk(0.0, 0.0) : RS[q][n1 + B1 * n2];
      stage_a<Lo, false, COUT == 2>(v, n1, two, T[q], 1);
    }
    __syncwarp();
    for (int i = lane; i < 3 * B2; i += 32) {
      const int q = i / B2, k2 = i - q * B2;
      double2 w[B1];
      stage_b<Lo, false>(w, k2, T[q], 1);
#pragma unroll
      for (int k1 = 0; k1 < B1; ++k1) Z[q][k2 + B2 * k1] = w[k1];
    }
    __syncwarp();
    constexpr int H = Lo / 2 + 1;
    for (int i = lane; i < 3 * H; i += 32) {
      const int q = i / H, k = i - q * H;
      const double2 Zk = Z[q][k], Zm = Z[q][(Lo - k) % Lo];
      double2* ra = a.spec_out + ((size_t)(q * nz + z) * a.out_rows + ya) * a.out_sx;
      ra[k] = mk((Zk.x + Zm.x) * 0.5, (Zk.y - Zm.y) * 0.5);
      ra[a.out_sx + k] = mk((Zk.y + Zm.y) * 0.5, (Zm.x - Zk.x) * 0.5);
    }
  }
  if (CIN == 2 && a.mode == X_UPDATE) residual_finish<32>(a, part);
  if (CIN == 1 && a.mode == X_ASSEMBLE && blockIdx.x == 0 && lane == 0) reset_ctrl(a.ctrl);
}

// ---------------------------------------------------------------- y passes
// 32-thread CTAs over the columns (component, plane, kx), R1 threads a column.
struct YArgs {
  double2* base;
  int rows, sx, HX, nzs, planes;
  const double2* tw;
  const Ctrl* ctrl;
  int check_done;
  int zoff, ylo, yhi;  // planes from zoff; input rows outside [ylo, yhi) read as zero (forward)
};
template <int L, bool INV, bool PAD> __global__ void __launch_bounds__(32) ypass_kernel(const YArgs a) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2, TC = 32 / R1;
  constexpr bool HALF = PAD && !INV;
  __shared__ __align__(16) double2 tw[L], T[R1 > 1 ? L * TC : 1];
  if (a.check_done && a.ctrl->done) return;
  const int t = threadIdx.x, c = t % TC, n1 = t / TC;
  const int e = blockIdx.x * TC + c;
  const bool ok = e < 3 * a.planes * a.HX;
  const int pl = ok ? e / a.HX : 0, kx = ok ? e - pl * a.HX : 0;
  const int q = pl / a.planes, z = a.zoff + pl - q * a.planes;
  double2* col = a.base + ((size_t)(q * a.nzs + z) * a.rows) * a.sx + kx;
  double2 v[R2];
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) {
    const int row = n1 + R1 * n2;
    v[n2] = (!(HALF && n2 >= R2 / 2) && ok && (INV || (row >= a.ylo && row < a.yhi))) ? col[(size_t)row * a.sx]
                                                                                   : mk(0.0, 0.0);
  }
  if constexpr (R1 > 1) {
    for (int i = t; i < L; i += 32) tw[i] = a.tw[i];
    __syncwarp();
    stage_a<L, INV, HALF>(v, n1, tw, T + c, TC);
    __syncwarp();
    for (int k2 = n1; k2 < R2; k2 += R1) {
      double2 w[R1];
      stage_b<L, INV>(w, k2, T + c, TC);
      if (ok) {
#pragma unroll
        for (int k1 = 0; k1 < (PAD && INV ? R1 / 2 : R1); ++k1) col[(size_t)(k2 + R2 * k1) * a.sx] = w[k1];
      }
    }
  } else {
    DFT<R2, INV, double2>::run(v);
    if (ok) {
#pragma unroll
      for (int k = 0; k < R2; ++k) col[(size_t)k * a.sx] = v[k];
    }
  }
}

// ---------------------------------------------------------------- z passes
// TC columns (kx, y) a CTA, its threads over (component, residue, column); the product over the
// spectra in shared memory.
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
  int zlo, zhi;  // the padded pass's input planes outside [zlo, zhi) read as zero
};
template <int L> struct ZT {
  static constexpr int R1 = Split<L>::R1, TC = R1 == 1 ? 8 : 4, NT = 3 * R1 * TC;
};
template <int L, int KIND> __global__ void __launch_bounds__(96) zpass_kernel(const ZArgs a) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2, TC = ZT<L>::TC, NT = ZT<L>::NT;
  constexpr bool PR = KIND == 1;
  __shared__ __align__(16) double2 tw[L], T[3][L * TC], F[3][L * TC];
  if (a.check_done && a.ctrl->done) return;
  const int t = threadIdx.x, c = t % TC, n1 = (t / TC) % R1, q = t / (TC * R1);
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
  double2 v[R2];
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) {
    const int l = n1 + R1 * n2;
    v[n2] = (!(PR && n2 >= R2 / 2) && ok && (!PR || (l >= a.zlo && l < a.zhi))) ? col[l * zstride] : mk(0.0, 0.0);
  }
  if (R1 > 1)
    for (int i = t; i < L; i += NT) tw[i] = a.tw[i];
  __syncthreads();
  stage_a<L, false, PR>(v, n1, tw, (R1 > 1 ? T[q] : F[q]) + c, TC);
  __syncthreads();
  if (R1 > 1) {
    for (int k2 = n1; k2 < R2; k2 += R1) {
      double2 w[R1];
      stage_b<L, false>(w, k2, T[q] + c, TC);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) F[q][(k2 + R2 * k1) * TC + c] = w[k1];
    }
    __syncthreads();
  }
#pragma unroll 1
  for (int i = t; i < L * TC; i += NT) {
    const int l = i / TC;
    int py, pk;
    if (!column(i - l * TC, py, pk)) continue;
    const double2 F0 = F[0][i], F1 = F[1][i], F2 = F[2][i];
    double ax, ay, az, s;
    if (!PR) {
      ax = a.kt0[pk]; ay = a.kt1[py]; az = a.kt2[l];
      s = a.st0[pk] * a.st1[py] * a.st2[l] * a.scale;
    } else {
      const int fy = (py <= a.ny) ? py : 2 * a.ny - py;
      const int fz = (l <= a.nz) ? l : 2 * a.nz - l;
      const double sy = (py <= a.ny) ? 1.0 : -1.0, sz = (l <= a.nz) ? 1.0 : -1.0;
      const size_t oct = (size_t)(a.nz + 1) * (a.ny + 1) * (a.nx + 1);
      const size_t off = ((size_t)fz * (a.ny + 1) + fy) * (a.nx + 1) + pk;
      ax = a.kap[off]; ay = sy * a.kap[oct + off]; az = sz * a.kap[2 * oct + off];
      s = 1.0;
    }
    // G = i s (a x F)
    const double2 cx = mk(ay * F2.x - az * F1.x, ay * F2.y - az * F1.y);
    const double2 cy = mk(az * F0.x - ax * F2.x, az * F0.y - ax * F2.y);
    const double2 cz = mk(ax * F1.x - ay * F0.x, ax * F1.y - ay * F0.y);
    F[0][i] = mk(-s * cx.y, s * cx.x);
    F[1][i] = mk(-s * cy.y, s * cy.x);
    F[2][i] = mk(-s * cz.y, s * cz.x);
  }
  __syncthreads();
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) v[n2] = F[q][(n1 + R1 * n2) * TC + c];
  if (R1 > 1) {
    stage_a<L, true, false>(v, n1, tw, T[q] + c, TC);
    __syncthreads();
    for (int k2 = n1; k2 < R2; k2 += R1) {
      double2 w[R1];
      stage_b<L, true>(w, k2, T[q] + c, TC);
      if (ok) {
#pragma unroll
        for (int k1 = 0; k1 < (PR ? R1 / 2 : R1); ++k1) col[(k2 + R2 * k1) * zstride] = w[k1];
      }
    }
  } else {
    DFT<R2, true, double2>::run(v);
    if (ok) {
#pragma unroll
      for (int k = 0; k < (PR ? R2 / 2 : R2); ++k) col[k * zstride] = v[k];
    }
  }
}

}  // namespace small
}  // namespace scfft
