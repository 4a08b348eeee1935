"""The FP64 passes' fixed-point building blocks on the CPU, from their own source text: the column maximum
runs in an emulated CTA that knows which lanes exist, and one pencil's transform, put together as the
passes do it, is compared with long double."""

import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1803_01346_gb300", "csrc")

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")


def text(name):
    return open(os.path.join(CSRC, name)).read()


# what fx64.cuh and fft_core.cuh take from CUDA, for a host compiler
CUDA_RUNTIME = r"""
#pragma once
#include <math.h>
#include <stdint.h>
#define __host__
#define __device__
#define __forceinline__ inline
#define __align__(n) alignas(n)
struct int2 { int x, y; };
struct alignas(16) int4 { int x, y, z, w; };
struct float2 { float x, y; };
struct alignas(16) double2 { double x, y; };
inline int2 make_int2(int x, int y) { return {x, y}; }
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
inline float2 make_float2(float x, float y) { return {x, y}; }
inline double2 make_double2(double x, double y) { return {x, y}; }
inline float2 __fadd2_rn(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
inline float2 __ffma2_rn(float2 a, float2 b, float2 c) { return {fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)}; }
"""


def run_cpp(tmp_path, source, *args):
    (tmp_path / "cuda_runtime.h").write_text(CUDA_RUNTIME)
    src = tmp_path / "host.cpp"
    src.write_text(source)
    exe = tmp_path / "host"
    r = subprocess.run(["g++", "-std=c++20", "-O2", "-fwrapv", "-ffp-contract=off", "-pthread", "-I", str(tmp_path), "-I", CSRC, str(src),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe), *map(str, args)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


# A thread per CUDA thread.  A shuffle of a lane that does not exist gives a value no maximum survives.
CTA = r"""
#include <barrier>
#include <climits>
#include <cstdio>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
struct Idx { unsigned x; };
static thread_local Idx threadIdx;
struct Warp { std::unique_ptr<std::barrier<>> bar; int lanes, v[32]; };
static std::vector<Warp> warps;
static std::mutex mu;
static int absent = 0;
static int __shfl_xor_sync(unsigned, int v, int o) {
  Warp& w = warps[threadIdx.x / 32];
  const int lane = threadIdx.x % 32;
  w.v[lane] = v;
  w.bar->arrive_and_wait();
  int r = INT_MAX;
  if ((lane ^ o) < w.lanes) r = w.v[lane ^ o];
  else { std::lock_guard<std::mutex> l(mu); ++absent; }
  w.bar->arrive_and_wait();
  return r;
}
static int atomicMax(int* p, int v) {
  std::lock_guard<std::mutex> l(mu);
  const int o = *p;
  if (v > o) *p = v;
  return o;
}
@FUNCTION@
template <int TC, int R1> int check() {
  constexpr int NT = TC * R1;
  (void)NT;
  int bad = 0;
  for (int top = 0; top < NT; ++top) {  // each thread in turn holds its column's largest value
    warps.clear();
    for (int w = 0; w < (NT + 31) / 32; ++w) {
      const int lanes = NT - 32 * w < 32 ? NT - 32 * w : 32;
      warps.push_back(Warp{std::make_unique<std::barrier<>>(lanes), lanes, {}});
    }
    int unit[TC], want[TC];
    for (int c = 0; c < TC; ++c) unit[c] = want[c] = INT_MIN;
    std::vector<std::thread> ts;
    for (int t = 0; t < NT; ++t) {
      const int p = t == top ? 1000 : (t * 37) % 101 - 50;
      if (p > want[t % TC]) want[t % TC] = p;
      ts.emplace_back([&unit, t, p] { threadIdx.x = t; @CALL@(unit, p); });
    }
    for (auto& t : ts) t.join();
    for (int c = 0; c < TC; ++c) bad += unit[c] != want[c];
  }
  if (bad || absent) printf("TC %d R1 %d: %d wrong, %d reads of absent lanes\n", TC, R1, bad, absent);
  return bad + absent;
}
int main() { return (@CHECKS@) ? 1 : 0; }
"""


def test_column_max_reads_no_absent_lane(tmp_path):
    passes, wide, yz = text("passes_fx.cuh"), text("passes_wide.cuh"), text("passes_yz_f64.cu")
    fn = re.search(r"template <[^>]*> __device__ __forceinline__ void column_max\(.*?\n}\n", passes, re.S).group(0)
    call = set(re.findall(r"column_max<[^>]*>(?=\()", passes))
    assert len(call) == 1 and passes.count("L = R1 * R2, NT = TC * R1;") == 2
    assert set(re.findall(r"constexpr int TC = (.*?);", yz)) == {"R1 >= 8 ? 4 : 8"}
    r1 = {int(m) for m in re.findall(r"X\(\d+, (\d+), \d+\)", wide)}
    assert {4, 8, 12, 16} == r1
    checks = " + ".join(f"check<{4 if r >= 8 else 8}, {r}>()" for r in sorted(r1))
    run_cpp(tmp_path, CTA.replace("@FUNCTION@", fn).replace("@CALL@", call.pop()).replace("@CHECKS@", checks))


# One pencil of R1 R2 points in fixed point, stage by stage as the passes do it, and in FP64 with the same
# two stages; relative 2-norm errors against long double.
PENCIL = r"""
#include <climits>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "fx64.cuh"
using namespace scfft;
typedef std::complex<long double> C;
static const long double PI = acosl(-1.0L);
static long long bits(double d) { long long b; memcpy(&b, &d, 8); return b; }
static int hi(double d) { return (int)(bits(d) >> 32); }
static double dbl(long long v, int u) {
  const unsigned long long b = fx_plain(u) ? fx_to_bits<true>(v, u) : fx_to_bits<false>(v, u);
  double d;
  memcpy(&d, &b, 8);
  return d;
}
template <int HEAD> static fxc fx_of(double2 d, int et) {
  return mk(fx_from_double<HEAD>(hi(d.x), (unsigned)bits(d.x), et), fx_from_double<HEAD>(hi(d.y), (unsigned)bits(d.y), et));
}
template <int R1, int R2, bool INV> void fixed(const double2* x, double2* y) {
  constexpr int L = R1 * R2;
  fxc v[R1][R2];
  int u[R1], U = INT_MIN;
  for (int n1 = 0; n1 < R1; ++n1) {
    int m = 0;
    for (int n2 = 0; n2 < R2; ++n2) m = fx_top(fx_top(m, hi(x[n1 + R1 * n2].x)), hi(x[n1 + R1 * n2].y));
    const int et = fx_exp_of(m);
    for (int n2 = 0; n2 < R2; ++n2) v[n1][n2] = fx_of<fx_head(R2)>(x[n1 + R1 * n2], et);
    DFT<R2, INV, fxc>::run(v[n1]);
    u[n1] = fx_unit_of(et, fx_head(R2)) + 2;
    m = 0;
    for (int k = 0; k < R2; ++k) {
      const long double a = 2 * PI * (n1 * k) / L;
      const long long c = llrintl(ldexpl(cosl(a), 62)) | 1, s = llrintl(ldexpl(sinl(a), 62)) | 1;
      v[n1][k] = k == 0 ? fx_quarter(v[n1][0]) : fx_twiddle<INV>(v[n1][k], make_int4(fx_hi(c), fx_lo(c), fx_hi(s), fx_lo(s)));
      m = fx_or(fx_or(m, v[n1][k].x), v[n1][k].y);
    }
    const int w = u[n1] + fx_bits(m) - fx_head(R1), p = w > u[n1] ? w : u[n1];
    if (p > U) U = p;
  }
  for (int k2 = 0; k2 < R2; ++k2) {
    fxc w[R1];
    for (int i = 0; i < R1; ++i) {
      const int k = U - u[i] < 63 ? U - u[i] : 63;
      w[i] = k > 0 ? mk(fx_shr(v[i][k2].x, k), fx_shr(v[i][k2].y, k)) : v[i][k2];
    }
    DFT<R1, INV, fxc>::run(w);
    for (int k1 = 0; k1 < R1; ++k1) y[k2 + R2 * k1] = make_double2(dbl(w[k1].x, U), dbl(w[k1].y, U));
  }
}
template <int R1, int R2, bool INV> void plain(const double2* x, double2* y) {
  constexpr int L = R1 * R2;
  double2 v[R1][R2];
  for (int n1 = 0; n1 < R1; ++n1) {
    for (int n2 = 0; n2 < R2; ++n2) v[n1][n2] = x[n1 + R1 * n2];
    DFT<R2, INV, double2>::run(v[n1]);
    for (int k = 1; n1 && k < R2; ++k) {
      const long double a = 2 * PI * (n1 * k) / L;
      const double2 w = make_double2((double)cosl(a), (double)-sinl(a));
      v[n1][k] = INV ? cmulc(v[n1][k], w) : cmul(v[n1][k], w);
    }
  }
  for (int k2 = 0; k2 < R2; ++k2) {
    double2 w[R1];
    for (int i = 0; i < R1; ++i) w[i] = v[i][k2];
    DFT<R1, INV, double2>::run(w);
    for (int k1 = 0; k1 < R1; ++k1) y[k2 + R2 * k1] = w[k1];
  }
}
static double normal() { double s = 0; for (int i = 0; i < 12; ++i) s += rand() / (RAND_MAX + 1.0); return s - 6; }
static double weight(int kind, int i, int L, int rep) {
  const int k = i < L / 2 ? i : L - i;
  switch (kind) {
    case 1: return pow(1e-8, (double)i / L);      // decaying over eight decades
    case 2: return 1.0 / (1 + k * k);             // a smooth field's spectrum
    case 3: return i == rep % L ? 1 : 1e-6;       // a spike
    case 4: return i < L / 2 ? 1 : 1e-6;          // a step of 120 dB
    case 5: return i < L / 2;                     // zero-padded
  }
  return 1;                                       // white
}
template <int R1, int R2, bool INV> void go(int kind, int scale) {
  constexpr int L = R1 * R2;
  long double e[2] = {0, 0}, n = 0;
  C root[L];
  for (int i = 0; i < L; ++i) root[i] = C(cosl(2 * PI * i / L), (INV ? 1 : -1) * sinl(2 * PI * i / L));
  for (int rep = 0; rep < 40; ++rep) {
    double2 x[L], y[2][L];
    for (int i = 0; i < L; ++i) {
      const double a = weight(kind, i, L, rep);
      x[i] = make_double2(ldexp(normal() * a, scale), ldexp(normal() * a, scale));
    }
    fixed<R1, R2, INV>(x, y[0]);
    plain<R1, R2, INV>(x, y[1]);
    for (int k = 0; k < L; ++k) {
      C s = 0;
      for (int i = 0; i < L; ++i) s += C(x[i].x, x[i].y) * root[i * k % L];
      n += std::norm(s * ldexpl(1, -scale));
      for (int q = 0; q < 2; ++q) e[q] += std::norm((C(y[q][k].x, y[q][k].y) - s) * ldexpl(1, -scale));
    }
  }
  printf("%d %d %d %d %.4Le %.4Le\n", L, (int)INV, kind, scale, sqrtl(e[0] / n), sqrtl(e[1] / n));
}
template <int R1, int R2> void all(int kinds, int scale) {
  for (int k = 0; k < kinds; ++k) { go<R1, R2, false>(k, scale); go<R1, R2, true>(k, scale); }
}
int main(int argc, char** argv) {
  const int kinds = atoi(argv[1]);
  for (int i = 2; i < argc; ++i) {
    const int s = atoi(argv[i]);
    @SPLITS@
  }
}
"""


def pencils(tmp_path, kinds, scales):
    """(length, inverse, kind, scale, fixed-point error, FP64 error) over every split of the passes."""
    splits = re.findall(r"X\(\d+, (\d+), (\d+)\)", text("passes_wide.cuh"))
    calls = " ".join(f"all<{a}, {b}>(kinds, s);" for a, b in sorted(set(splits)))
    out = run_cpp(tmp_path, PENCIL.replace("@SPLITS@", calls), kinds, *scales)
    rows = [tuple(float(v) for v in line.split()) for line in out.splitlines()]
    assert len(rows) == 2 * kinds * len(scales) * len(set(splits))
    return rows


def test_pencils_of_any_exponent_keep_their_accuracy(tmp_path):
    """The error does not depend on the exponent down to where the results themselves become subnormal: the
    rounding of two stages at 2^-57 of the largest value and of the result to a double stay below 2^-53."""
    for L, inv, _, scale, fx, _ in pencils(tmp_path, 1, (0, 900, -900, -960, -980, -1000, -1010)):
        assert fx < 2.0 ** -53, (L, inv, scale, fx)


def test_pencils_are_nearer_to_exact_than_in_fp64(tmp_path):
    """The rounding of a pencil's largest value at 2^-57 in two stages adds less than the rounding of each
    value at 2^-53 in every butterfly does, whatever the spectrum."""
    for L, inv, kind, _, fx, fp64 in pencils(tmp_path, 6, (0,)):
        assert fx < fp64, (L, inv, kind, fx, fp64)
