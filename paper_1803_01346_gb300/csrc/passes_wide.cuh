// passes_wide.cuh - what the FFT passes of the FP64 path and the FP32 reverse mode share: arguments
// and node-wise steps of the x passes, the x pass template (instantiated for the FP32 reverse
// mode), and the launchers that choose a pass's kernel.
//
// Every 3D transform is split into three batched 1D passes along x, y and z on
// the layouts [comp][z][y][x] (real) and [comp][z][y][kx] (half spectrum,
// row stride sx).  Pointwise work is fused into the passes:
//   x passes  : C2R of a half-spectrum row, the node-wise step (power law of
//               Eq. 1 / Omega_out Ohm law, dh^0 assembly, mask + zero pad, the
//               Eq. 5 update and its residual), then R2C of the result.
//   z passes  : forward z FFT, the spectral curl multiply i S(k) k x F, or the
//               kernel-spectrum cross product K^ x F of Eq. 7, inverse z FFT.
//   y passes  : plain y FFTs, pruned to the nonzero input / needed output rows
//               on the zero-padded grid.
// Two real rows of one component travel as the real and imaginary parts of one
// complex pencil in the x passes (two real transforms for one complex one).
#pragma once
#include <math.h>
#include <stdio.h>

#include <type_traits>

#include "scfft_internal.cuh"

namespace scfft {

template <typename V> __device__ __forceinline__ V vzero();
template <> __device__ __forceinline__ float2 vzero<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double2 vzero<double2>() { return make_double2(0.0, 0.0); }

// Euclidean norm of the change of one node's iterate (the Eq. 5 residual's summand), in FP64
template <typename T> __device__ __forceinline__ double dnorm3(T v0, T o0, T v1, T o1, T v2, T o2) {
  const double d0 = (double)v0 - (double)o0, d1 = (double)v1 - (double)o1, d2 = (double)v2 - (double)o2;
  return sqrt(d0 * d0 + d1 * d1 + d2 * d2);
}

// Power law of Eq. 1: returns rho(|j|) for |j| = jn.  FP32 evaluates
// |j/jc|^(n-1) as 2^((n-1) log2(|j|/jc)) so that large n cannot overflow an
// intermediate power; FP64 uses pow directly.
__device__ __forceinline__ float rho_power(float jn, float jcv, float n, float e0) {
  if (jn == 0.f) return (n == 1.f) ? e0 / jcv : 0.f;
  return (e0 / jcv) * exp2f((n - 1.f) * log2f(jn / jcv));
}
__device__ __forceinline__ double rho_power(double jn, double jcv, double n, double e0) {
  if (jn == 0.0) return (n == 1.0) ? e0 / jcv : 0.0;
  return (e0 / jcv) * pow(jn / jcv, n - 1.0);
}

namespace wide {

__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }

template <typename V> __device__ __forceinline__ V shfl_v(V v, int src);
template <> __device__ __forceinline__ float2 shfl_v(float2 v, int s) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, s), __shfl_sync(0xffffffffu, v.y, s));
}
template <> __device__ __forceinline__ double2 shfl_v(double2 v, int s) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, s), __shfl_sync(0xffffffffu, v.y, s));
}
// CTAs of a kernel resident at once on the whole GPU (the grid of a persistent launch)
template <typename K> int resident_ctas(K k, int threads, size_t smem) {
  int per_sm = 0, dev = 0, sms = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem);
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return per_sm > 0 && sms > 0 ? per_sm * sms : 1024;
}

}  // namespace wide

// ---------------------------------------------------------------- x passes
template <typename T>
struct XArgs {
  typedef typename cplx_of<T>::type V;
  Geo g;
  int mode;
  const V* spec_in;
  int in_rows, in_sx;
  V* spec_out;
  int out_rows, out_sx;
  const V* tw_in;
  const V* tw_out;
  const double* src_f64;
  const T* src_t;     // real input rows in the pass's own type (instead of src_f64), or nullptr
  double* dst_f64;
  const double* warm;
  const uint8_t* mask;
  const T* jc;
  T* hbuf[2];       // both iterate buffers: the update pass picks by the device's iteration count
  PointParams pp;
  PointParams* ppd; // device copy of pp (written by the assemble pass, read by the update pass)
  Ctrl* ctrl;
  double* partials;
  int check_done;
  // mask/pad pass of an Eq. 5 iteration, and the passes of the transposed one that multiply by chi:
  // only the rows of Omega's box (y in [by0, by1), z in [bz0, bz1)); the source vanishes outside,
  // and nothing downstream reads the rows left out
  int use_box, by0, by1, bz0, bz1;
  // those passes: each work item is one component of a tile.  The box holds few tiles (64 x 64 x 96 shield: 293
  // of four row pairs, two CTAs of 64 threads an SM): FP64 mask/pad 47 -> 25 us there
  int comp_split;
};

// What the update pass takes from the device, so that a captured launch serves every iteration:
// its iteration index, the iterate buffers and dh_e/dt.
template <typename T> struct UpdateArgs {
  int it = 0;
  const T* hold = nullptr;
  T* hnew = nullptr;
  T hedot[3];
};
template <typename T> __device__ __forceinline__ UpdateArgs<T> update_args(const XArgs<T>& a) {
  UpdateArgs<T> u;
  if (a.mode == X_UPDATE) {
    u.it = *reinterpret_cast<volatile const int*>(&a.ctrl->iters);  // (residual_finish writes it at the end)
    u.hold = (u.it & 1) ? a.hbuf[1] : a.hbuf[0];
    u.hnew = (u.it & 1) ? a.hbuf[0] : a.hbuf[1];
    for (int q = 0; q < 3; ++q) u.hedot[q] = (T)a.ppd->hedot[q];
  }
  return u;
}

// The node-wise step of an x pass on one node's three real values v (in and out); returns the
// node's summand of the Eq. 5 residual (the update modes, 0 otherwise).
template <typename T>
__device__ __forceinline__ double node_step(const XArgs<T>& a, const UpdateArgs<T>& up, size_t node, T v[3]) {
  typedef T A;
  const PointParams& pp = a.pp;
  const long long N = a.g.N;
  switch (a.mode) {
    case X_POWERLAW: {
      A w0 = v[0], w1 = v[1], w2 = v[2];
      A rho;
      if (a.mask[node]) {
        A jcv = a.jc ? a.jc[node] : (A)pp.jc;
        if (pp.law) {
          // e(j, h): jc(h) = jc / (1 + |h| / h0) (Kim), e = rho(|A j|) A^2 j
          if (pp.kim_h0 > 0) {
            const A h0 = (A)a.src_f64[node], h1 = (A)a.src_f64[N + node], h2 = (A)a.src_f64[2 * N + node];
            jcv = jcv / ((A)1 + sqrt(h0 * h0 + h1 * h1 + h2 * h2) / (A)pp.kim_h0);
          }
          const A ax = (A)pp.aniso[0], ay = (A)pp.aniso[1], az = (A)pp.aniso[2];
          const A u0 = ax * w0, u1 = ay * w1, u2 = az * w2;
          rho = rho_power(sqrt(u0 * u0 + u1 * u1 + u2 * u2), jcv, (A)pp.n, (A)pp.e0);
          w0 *= rho * ax * ax; w1 *= rho * ay * ay; w2 *= rho * az * az;
        } else {
          const A jn = sqrt(w0 * w0 + w1 * w1 + w2 * w2);
          rho = rho_power(jn, jcv, (A)pp.n, (A)pp.e0);
          w0 *= rho; w1 *= rho; w2 *= rho;
        }
      } else {
        rho = (A)pp.rho_out;
        w0 *= rho; w1 *= rho; w2 *= rho;
      }
      v[0] = w0; v[1] = w1; v[2] = w2;
      return 0.0;
    }
    case X_ASSEMBLE:
      if (a.mask[node]) {
        const T s = -(T)pp.inv_mu0;
        v[0] *= s; v[1] *= s; v[2] *= s;
      } else {
        v[0] = (T)a.warm[node]; v[1] = (T)a.warm[N + node]; v[2] = (T)a.warm[2 * N + node];
      }
      a.hbuf[0][node] = v[0]; a.hbuf[0][N + node] = v[1]; a.hbuf[0][2 * N + node] = v[2];
      return 0.0;
    case X_MASKPAD:
    case X_ADJ_CROP:
      if (!a.mask[node]) { v[0] = 0; v[1] = 0; v[2] = 0; }
      return 0.0;
    case X_UPDATE: {
      const T o0 = up.hold[node], o1 = up.hold[N + node], o2 = up.hold[2 * N + node];
      double d = 0.0;
      if (a.mask[node]) {
        v[0] = o0; v[1] = o1; v[2] = o2;
      } else {
        v[0] = up.hedot[0] + v[0]; v[1] = up.hedot[1] + v[1]; v[2] = up.hedot[2] + v[2];
        d = dnorm3(v[0], o0, v[1], o1, v[2], o2);
      }
      up.hnew[node] = v[0]; up.hnew[N + node] = v[1]; up.hnew[2 * N + node] = v[2];
      return d;
    }
    case X_TO_F64:
    case X_CROP_F64:
      a.dst_f64[node] = (double)v[0]; a.dst_f64[N + node] = (double)v[1]; a.dst_f64[2 * N + node] = (double)v[2];
      return 0.0;
    case X_ADJ_COMBINE: {
      const bool in = a.mask[node];
      a.dst_f64[node] = (double)v[0] + (in ? a.src_f64[node] : 0.0);
      a.dst_f64[N + node] = (double)v[1] + (in ? a.src_f64[N + node] : 0.0);
      a.dst_f64[2 * N + node] = (double)v[2] + (in ? a.src_f64[2 * N + node] : 0.0);
      return 0.0;
    }
    case X_ADJ_POWERLAW: {
      // lam_e = -(curl lam_u)/mu0; lam_j = J_e^T lam_e; J_e = rho (I + (n-1) jhat jhat^T) in Omega
      const A s = -(A)pp.inv_mu0;
      const A l0 = s * v[0], l1 = s * v[1], l2 = s * v[2];
      A w0, w1, w2;
      if (a.mask[node]) {
        const A j0 = (A)a.src_f64[node], j1 = (A)a.src_f64[N + node], j2 = (A)a.src_f64[2 * N + node];
        const A jcv = a.jc ? a.jc[node] : (A)pp.jc;
        const A jn = sqrt(j0 * j0 + j1 * j1 + j2 * j2);
        const A rho = rho_power(jn, jcv, (A)pp.n, (A)pp.e0);
        const A jl = j0 * l0 + j1 * l1 + j2 * l2;
        const A f = jn > 0 ? ((A)pp.n - 1) * jl / (jn * jn) : (A)0;
        w0 = rho * (l0 + f * j0); w1 = rho * (l1 + f * j1); w2 = rho * (l2 + f * j2);
        if (a.dst_f64) a.dst_f64[node] = (double)(-(A)pp.n * rho / jcv * jl);
      } else {
        const A r = (A)pp.rho_out;
        w0 = r * l0; w1 = r * l1; w2 = r * l2;
        if (a.dst_f64) a.dst_f64[node] = 0.0;
      }
      v[0] = w0; v[1] = w1; v[2] = w2;
      return 0.0;
    }
  }
  return 0.0;
}

// The end of an Eq. 5 update pass: the deterministic two-level reduction of the residual's
// summands, the stop flag and the iterate's bookkeeping (written by the last CTA).
template <int NT, typename T> __device__ void residual_finish(const XArgs<T>& a, double part, int it) {
  __shared__ double red[NT / 32];
  __shared__ int am_last;
  const int tid = threadIdx.x;
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((tid & 31) == 0) red[tid >> 5] = part;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int i = 0; i < NT / 32; ++i) s += red[i];
    a.partials[blockIdx.x] = s;
    __threadfence();
    const unsigned prev = atomicAdd(&a.ctrl->counter, 1u);
    am_last = (prev == gridDim.x - 1);
  }
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  double s = 0.0;
  for (int i = tid; i < (int)gridDim.x; i += NT) s += __ldcg(&a.partials[i]);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __syncthreads();
  if ((tid & 31) == 0) red[tid >> 5] = s;
  __syncthreads();
  if (tid == 0) {
    double tot = 0.0;
    for (int i = 0; i < NT / 32; ++i) tot += red[i];
    const double res = tot * a.ppd->inv_nout;
    Ctrl* c = a.ctrl;
    c->residual = res;
    c->iters = it + 1;
    c->iter_total += 1;
    c->cur = (it + 1) & 1;
    const bool finite = isfinite(res);
    if (!finite) c->status = 6;  // SCFFT_ENONFINITE
    c->done = (!finite || res < a.ppd->tol) ? 1 : 0;
    c->counter = 0;
  }
}
template <typename T> __device__ __forceinline__ void begin_loop(const XArgs<T>& a) {
  *a.ppd = a.pp;
  Ctrl* c = a.ctrl;
  c->trips = 0;
  c->done = 0;
  c->iters = 0;
  c->cur = 0;
  c->counter = 0;
  c->residual = 0.0;
}

// An x pass as CIN (its input: 0 real rows, 1 half spectra of length nx, 2 of length 2nx kept to
// x < nx) and COUT (0 real rows, 1 half spectra of length nx, 2 of length 2nx of the zero-padded
// rows); the node-wise step between them is chosen at run time (node_step).  Splits: the C2R is
// R1i R2i, the R2C R1o R2o with R1o = R2i.  TP lanes of one warp hold a row pair.
template <int CIN, int COUT, int R1i, int R2i, int R2o> struct WX {
  static constexpr int R1o = R2i;
  static constexpr int Li = R1i * R2i;
  static constexpr int Lo = R1o * R2o;
  static constexpr int XL = CIN ? (CIN == 2 ? Li / 2 : Li) : (COUT == 2 ? Lo / 2 : Lo);  // nx
  static constexpr int TP0 = wide::cmax(wide::cmax(CIN ? R1i : 1, R2i), COUT ? R2o : 1);
  static constexpr int TP = TP0 <= 4 ? 4 : TP0 <= 8 ? 8 : 16;
  static constexpr int P = 64 / TP;  // row pairs per CTA
  static constexpr int NT = 64;
  static constexpr int KX = CIN == 2 ? R1i / 2 : R1i;
  static constexpr int TT = wide::cmax(CIN ? R2i * (R1i + 1) : 1, COUT ? R2o * (R1o + 1) : 1);
  static constexpr int TWI = CIN ? Li : 0, TWO = COUT ? Lo : 0;
  // whether the node-wise step may be the product by chi (mask/pad, its transposed counterpart), which
  // leaves the components independent
  static constexpr bool MASKS = (CIN == 1 && COUT == 2) || (CIN == 2 && COUT == 1);
  static constexpr int SM = TWI + TWO + 3 * P * XL + P * TT;  // complex values of shared memory
};

// SPLIT: each work item is one component of a tile (the passes that multiply by chi).
template <typename T, int CIN, int COUT, int R1i, int R2i, int R2o, bool SPLIT>
__global__ void __launch_bounds__(64) xwide_kernel(const XArgs<T> a) {
  typedef typename cplx_of<T>::type V;
  typedef WX<CIN, COUT, R1i, R2i, R2o> S;
  constexpr int TP = S::TP, P = S::P, NT = S::NT, XL = S::XL, TT = S::TT, Li = S::Li, Lo = S::Lo, R1o = S::R1o;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  if (a.check_done && a.ctrl->done) return;
  const UpdateArgs<T> up = update_args(a);
  V* twi = reinterpret_cast<V*>(smem_raw);  // [k2][n1]: the lanes of a pair read consecutive words
  V* two = twi + S::TWI;
  V* RS = two + S::TWO;  // [3][P][XL] real rows of the pairs, as complex values
  V* Tb = RS + 3 * P * XL;
  const int tid = threadIdx.x;
  const int p = tid / TP, r = tid % TP;
  for (int i = tid; i < S::TWI; i += NT) twi[i] = a.tw_in[(i % R1i) * (i / R1i)];
  for (int i = tid; i < S::TWO; i += NT) two[i] = a.tw_out[(i % R1o) * (i / R1o)];
  const int ny = a.g.ny, nz = a.g.nz;
  const long long N = a.g.N;
  const int hp = (a.use_box ? a.by1 - a.by0 : ny) >> 1;
  const int npairs = (a.use_box ? a.bz1 - a.bz0 : nz) * hp;
  const int ntiles = (npairs + P - 1) / P;
  V* Tp = Tb + p * TT;
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
        if (r < R1i) {
          const V* ra = a.spec_in + ((size_t)(q * nz + z) * a.in_rows + ya) * a.in_sx;
          const V* rb = ra + a.in_sx;
          V v[R2i];
#pragma unroll
          for (int n2 = 0; n2 < R2i; ++n2) {
            // Z[k] = A[k] + i B[k], Z[L-k] = conj(A[k]) + i conj(B[k]); only the real parts of
            // DC and Nyquist are read
            const int k = r + R1i * n2;
            const bool lo = k <= Li / 2;
            const int kk = lo ? k : Li - k;
            V A = vzero<V>(), B = vzero<V>();
            if (pok) { A = ra[kk]; B = rb[kk]; }
            if (kk == 0 || kk == Li / 2) { A.y = 0; B.y = 0; }
            v[n2] = lo ? mk(A.x - B.y, A.y + B.x) : mk(A.x + B.y, B.x - A.y);
          }
          DFT<R2i, true, V>::run(v);
#pragma unroll
          for (int k2 = 0; k2 < R2i; ++k2) Tp[k2 * (R1i + 1) + r] = k2 == 0 ? v[0] : cmulc(v[k2], twi[k2 * R1i + r]);
        }
        __syncwarp();
        if (r < R2i) {
          V w[R1i];
#pragma unroll
          for (int m = 0; m < R1i; ++m) w[m] = Tp[r * (R1i + 1) + m];
          DFT<R1i, true, V>::run(w);
#pragma unroll
          for (int k1 = 0; k1 < S::KX; ++k1) RS[(q * P + p) * XL + r + R2i * k1] = w[k1];
        }
        __syncwarp();
      }
      // the node-wise step on the nodes x = r + TP j of both rows of the lane's pair
      if constexpr (SPLIT) {
        if (pok) {
          for (int x = r; x < XL; x += TP) {
            V* w = RS + (q0 * P + p) * XL + x;
            if (!a.mask[na0 + x]) w->x = 0;
            if (!a.mask[na0 + XL + x]) w->y = 0;
          }
        }
      } else {
#pragma unroll 1
        for (int x = r; x < XL; x += TP) {
          if (!pok) continue;
          V u[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) u[q] = RS[(q * P + p) * XL + x];
          T va[3] = {u[0].x, u[1].x, u[2].x}, vb[3] = {u[0].y, u[1].y, u[2].y};
          part += node_step<T>(a, up, na0 + x, va);
          part += node_step<T>(a, up, na0 + XL + x, vb);
          if (COUT > 0) {
#pragma unroll
            for (int q = 0; q < 3; ++q) RS[(q * P + p) * XL + x] = mk(va[q], vb[q]);
          }
        }
      }
      __syncwarp();
    } else {
#pragma unroll 1
      for (int q = 0; q < 3; ++q) {
        constexpr int J = XL / TP;
        V u[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const size_t na = na0 + r + TP * j, nb = na + XL;
          T va = 0, vb = 0;
          if (pok) {
            const size_t o = (size_t)q * N;
            va = a.src_t ? a.src_t[o + na] : (T)a.src_f64[o + na];
            vb = a.src_t ? a.src_t[o + nb] : (T)a.src_f64[o + nb];
            if (a.mode == X_ADJ_PAD) {  // (1 - chi)
              if (a.mask[na]) va = 0;
              if (a.mask[nb]) vb = 0;
            }
            if (a.mode == X_ADJ_IN) {  // chi
              if (!a.mask[na]) va = 0;
              if (!a.mask[nb]) vb = 0;
            }
          }
          u[j] = mk(va, vb);
        }
#pragma unroll
        for (int j = 0; j < J; ++j) RS[(q * P + p) * XL + r + TP * j] = u[j];
      }
      __syncwarp();
    }
    if constexpr (COUT > 0) {
#pragma unroll 1
      for (int q = q0; q < q1; ++q) {
        if (r < R1o) {
          V u[R2o];
#pragma unroll
          for (int n2 = 0; n2 < R2o; ++n2)
            u[n2] = (COUT == 2 && n2 >= R2o / 2) ? vzero<V>() : RS[(q * P + p) * XL + r + R1o * n2];
          dft_maybe_half<R2o, false, COUT == 2>(u);
#pragma unroll
          for (int k2 = 0; k2 < R2o; ++k2) Tp[k2 * (R1o + 1) + r] = k2 == 0 ? u[0] : cmul(u[k2], two[k2 * R1o + r]);
        }
        __syncwarp();
        const int k2 = r;
        V Zr[R1o];
#pragma unroll
        for (int m = 0; m < R1o; ++m) Zr[m] = vzero<V>();
        if (k2 < R2o) {
#pragma unroll
          for (int m = 0; m < R1o; ++m) Zr[m] = Tp[k2 * (R1o + 1) + m];
          DFT<R1o, false, V>::run(Zr);
        }
        // separate the two rows: A = (Z[k] + conj Z[Lo-k])/2, B = (Z[k] - conj Z[Lo-k])/(2i).
        // Thread k2 holds Z[k2 + R2o k1]; the mirror Lo - k lives in thread R2o - k2 at register
        // R1o - 1 - k1 (k2 > 0) or in this thread at (R1o - k1) mod R1o (k2 = 0).
        const int lane = tid & 31;
        const int src = lane - k2 + (k2 == 0 ? 0 : (k2 < R2o ? R2o - k2 : k2));
        V* ra = a.spec_out + ((size_t)(q * nz + z) * a.out_rows + ya) * a.out_sx;
        V* rb = ra + a.out_sx;
        const T half = (T)0.5;
#pragma unroll
        for (int k1 = 0; k1 <= R1o / 2; ++k1) {
          const V sh = wide::shfl_v(Zr[R1o - 1 - k1], src);
          const V Zk = Zr[k1];
          const V Zm = k2 == 0 ? Zr[(R1o - k1) % R1o] : sh;
          const int k = k2 + R2o * k1;
          if (k2 < R2o && pok && k <= Lo / 2) {
            ra[k] = mk((Zk.x + Zm.x) * half, (Zk.y - Zm.y) * half);
            rb[k] = mk((Zk.y + Zm.y) * half, (Zm.x - Zk.x) * half);
          }
        }
        __syncwarp();  // the next component's first stage overwrites Tp
      }
    }
    __syncwarp();  // the pair's rows are reused by the next tile
  }

  if (CIN == 2 && a.mode == X_UPDATE) residual_finish<NT>(a, part, up.it);
  if (CIN == 1 && a.mode == X_ASSEMBLE && blockIdx.x == 0 && tid == 0) begin_loop(a);
}

// ---------------------------------------------------------------- launchers
namespace wide {

template <typename T, int CIN, int COUT, int R1i, int R2i, int R2o, bool SPLIT = false>
cudaError_t go_x(const XArgs<T>& a, cudaStream_t st) {
  typedef WX<CIN, COUT, R1i, R2i, R2o> S;
  if constexpr (S::MASKS && !SPLIT)
    if (a.comp_split) return go_x<T, CIN, COUT, R1i, R2i, R2o, true>(a, st);
  constexpr auto k = xwide_kernel<T, CIN, COUT, R1i, R2i, R2o, SPLIT>;
  const size_t smem = sizeof(typename cplx_of<T>::type) * S::SM;
  allow_smem<k>();
  static const int resident = resident_ctas(k, S::NT, smem);
  const int hp = (a.use_box ? a.by1 - a.by0 : a.g.ny) / 2;
  const int ntiles = ((a.use_box ? a.bz1 - a.bz0 : a.g.nz) * hp + S::P - 1) / S::P * (SPLIT ? 3 : 1);
  const int grid = ntiles < resident ? ntiles : resident;
  launch_chained(k, dim3(grid), S::NT, smem, st, a);
  return checked_launch("xwide_kernel", dim3(grid), S::NT, smem);
}

// Splits per nx: C2R(nx) = A B, C2R(2nx) = C D; the R2C's first factor is the C2R's second.
template <typename T, int CIN, int COUT> cudaError_t go_x_n(const XArgs<T>& a, cudaStream_t st) {
#define XN(NN, A_, B_, C_, D_)                                                                                  \
  case NN:                                                                                                      \
    if constexpr (CIN == 0) return go_x<T, CIN, COUT, 1, B_, COUT == 2 ? 2 * A_ : A_>(a, st);                   \
    else if constexpr (CIN == 1) return go_x<T, CIN, COUT, A_, B_, COUT == 2 ? 2 * A_ : COUT == 1 ? A_ : 1>(a, st); \
    else return go_x<T, CIN, COUT, C_, D_, COUT == 1 ? C_ / 2 : 1>(a, st);
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

// Lengths and their (R1, R2) splits, R1 >= R2: unpadded axes 16..128, padded ones 32..256.
#define WIDE_UNPADDED(X) X(16, 4, 4) X(32, 8, 4) X(48, 12, 4) X(64, 8, 8) X(96, 12, 8) X(128, 16, 8)
#define WIDE_PADDED(X) X(32, 8, 4) X(64, 8, 8) X(96, 12, 8) X(128, 16, 8) X(192, 16, 12) X(256, 16, 16)

}  // namespace wide

// the FP64 passes in 64-bit fixed point (passes_fx.cuh)
namespace fx {
template <int CIN, int COUT> cudaError_t go_x_n(const Launch<double>& L, const XArgs<double>& a);
cudaError_t launch_y(const Launch<double>& L, bool padded, bool inverse, bool check_done);
cudaError_t launch_z(const Launch<double>& L, bool padded, bool check_done, double scale);
}  // namespace fx
// the same on small grids: native FP64 (passes_small.cuh)
namespace small {
cudaError_t launch_x(const XArgs<double>& a, int cin, int cout, cudaStream_t st);
cudaError_t launch_y(const Launch<double>& L, bool padded, bool inverse, bool check_done);
cudaError_t launch_z(const Launch<double>& L, bool padded, bool check_done, double scale);
}  // namespace small

template <typename T, int CIN, int COUT> static cudaError_t go_x_any(const Launch<T>& L, const XArgs<T>& a) {
  if constexpr (std::is_same<T, double>::value)
    return fixed_point_grid(L.g) ? fx::go_x_n<CIN, COUT>(L, a) : small::launch_x(a, CIN, COUT, L.st);
  else return wide::go_x_n<T, CIN, COUT>(a, L.st);
}

template <typename T>
static cudaError_t launch_x_impl(const Launch<T>& L, XMode mode, const PointParams& pp, const double* src_f64,
                                 const T* src_t, double* dst_f64, const double* warm, int in_buf, int out_buf,
                                 bool check_done) {
  if (mode == X_POWERLAW_H) mode = X_POWERLAW;
  const bool fd = mode == X_UPDATE_FD;  // the stencil curl reads the iterate as is: no R2C
  if (fd) mode = X_UPDATE;
  XArgs<T> a{};
  const Geo& g = L.g;
  a.g = g;
  a.mode = mode;
  const bool pin = (mode == X_UPDATE || mode == X_CROP_F64 || mode == X_ADJ_CROP);
  const bool pout = (mode == X_MASKPAD || mode == X_PAD_F64 || mode == X_ADJ_PAD);
  a.spec_in = pin ? L.w->Pd : L.w->U;
  a.in_rows = pin ? 2 * g.ny : g.ny;
  a.in_sx = pin ? g.sxp : g.sxu;
  a.spec_out = pout ? L.w->Pd : L.w->U;
  a.out_rows = pout ? 2 * g.ny : g.ny;
  a.out_sx = pout ? g.sxp : g.sxu;
  a.tw_in = pin ? L.w->twp[0] : L.w->twu[0];
  a.tw_out = pout ? L.w->twp[0] : L.w->twu[0];
  a.src_f64 = src_f64;
  a.src_t = src_t;
  a.dst_f64 = dst_f64;
  a.warm = warm;
  a.mask = L.mask;
  a.jc = L.w->jc;
  a.hbuf[0] = L.w->Hd[0];
  a.hbuf[1] = L.w->Hd[1];
  a.pp = pp;
  a.ppd = L.ppd;
  a.ctrl = L.ctrl;
  a.partials = L.partials;
  a.check_done = check_done ? 1 : 0;
  a.use_box = (L.use_box && mode == X_MASKPAD) || (L.use_tbox && (mode == X_ADJ_CROP || mode == X_ADJ_IN));
  a.comp_split = a.use_box && (mode == X_MASKPAD || mode == X_ADJ_CROP);
  a.by0 = L.by0;
  a.by1 = L.by1;
  a.bz0 = L.bz0;
  a.bz1 = L.bz1;
  switch (mode) {
    case X_ADJ_IN: return go_x_any<T, 0, 1>(L, a);
    case X_ADJ_PAD: return go_x_any<T, 0, 2>(L, a);
    case X_ADJ_COMBINE: return go_x_any<T, 1, 0>(L, a);
    case X_ADJ_POWERLAW: return go_x_any<T, 1, 1>(L, a);
    case X_ADJ_CROP: return go_x_any<T, 2, 1>(L, a);
    default: break;
  }
  if constexpr (sizeof(T) == 8) {  // (FP32 forward passes: passes_reg.cu)
    switch (mode) {
      case X_FWD_F64: return go_x_any<T, 0, 1>(L, a);
      case X_PAD_F64: return go_x_any<T, 0, 2>(L, a);
      case X_TO_F64: return go_x_any<T, 1, 0>(L, a);
      case X_POWERLAW:
      case X_ASSEMBLE: return go_x_any<T, 1, 1>(L, a);
      case X_MASKPAD: return go_x_any<T, 1, 2>(L, a);
      case X_UPDATE: return fd ? go_x_any<T, 2, 0>(L, a) : go_x_any<T, 2, 1>(L, a);
      case X_CROP_F64: return go_x_any<T, 2, 0>(L, a);
      default: break;
    }
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_x(const Launch<T>& L, XMode mode, const PointParams& pp, const double* src_f64, double* dst_f64,
                     const double* warm, int in_buf, int out_buf, bool check_done) {
  // the FP32 forward passes have their own kernels; the transposed (reverse-mode) passes are
  // these templates in every precision
  if constexpr (sizeof(T) == 4)
    if (mode < X_ADJ_PAD || mode == X_POWERLAW_H || mode == X_UPDATE_FD)
      return launch_x_reg(L, mode, pp, src_f64, dst_f64, warm, in_buf, out_buf, check_done);
  return launch_x_impl<T>(L, mode, pp, src_f64, nullptr, dst_f64, warm, in_buf, out_buf, check_done);
}

template <typename T>
cudaError_t launch_x_pad_rows(const Launch<T>& L, const PointParams& pp, const T* rows, bool check_done) {
  return launch_x_impl<T>(L, X_PAD_F64, pp, nullptr, rows, nullptr, nullptr, 0, 0, check_done);
}

template <typename T>
cudaError_t launch_y(const Launch<T>& L, bool padded, bool inverse, bool check_done) {
  if constexpr (sizeof(T) == 4) return launch_y_reg(L, padded, inverse, check_done);
  else if (fixed_point_grid(L.g)) return fx::launch_y(L, padded, inverse, check_done);
  else return small::launch_y(L, padded, inverse, check_done);
}

template <typename T>
static cudaError_t launch_z(const Launch<T>& L, bool padded, bool check_done, double scale) {
  if constexpr (sizeof(T) == 4) return launch_z_reg(L, padded, check_done, scale);
  else if (fixed_point_grid(L.g)) return fx::launch_z(L, padded, check_done, scale);
  else return small::launch_z(L, padded, check_done, scale);
}

template <typename T> cudaError_t launch_z_curl(const Launch<T>& L, bool check_done, double scale) {
  return launch_z<T>(L, false, check_done, scale);
}
template <typename T> cudaError_t launch_z_kernel(const Launch<T>& L, bool check_done) {
  return launch_z<T>(L, true, check_done, 1.0);
}

#define INST_PASSES_X(T)                                                                                       \
  template cudaError_t launch_x<T>(const Launch<T>&, XMode, const PointParams&, const double*, double*,        \
                                   const double*, int, int, bool);                                             \
  template cudaError_t launch_x_pad_rows<T>(const Launch<T>&, const PointParams&, const T*, bool);
#define INST_PASSES_YZ(T)                                                                                      \
  template cudaError_t launch_y<T>(const Launch<T>&, bool, bool, bool);                                        \
  template cudaError_t launch_z_curl<T>(const Launch<T>&, bool, double);                                       \
  template cudaError_t launch_z_kernel<T>(const Launch<T>&, bool);

}  // namespace scfft
