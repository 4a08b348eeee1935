"""The FP64 passes' fixed-point building blocks on the CPU, from their own source text: the column maximum
runs in an emulated CTA that knows which lanes exist."""

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


def run_cpp(tmp_path, source, *args):
    src = tmp_path / "host.cpp"
    src.write_text(source)
    exe = tmp_path / "host"
    r = subprocess.run(["g++", "-std=c++20", "-O2", "-fwrapv", "-pthread", "-I", str(tmp_path), "-I", CSRC, str(src),
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
    assert len(call) == 1 and passes.count("__launch_bounds__(TC * R1)") == 2
    assert set(re.findall(r"constexpr int TC = (.*?);", yz)) == {"R1 >= 8 ? 4 : 8"}
    r1 = {int(m) for m in re.findall(r"X\(\d+, (\d+), \d+\)", wide)}
    assert {4, 8, 12, 16} == r1
    checks = " + ".join(f"check<{4 if r >= 8 else 8}, {r}>()" for r in sorted(r1))
    run_cpp(tmp_path, CTA.replace("@FUNCTION@", fn).replace("@CALL@", call.pop()).replace("@CHECKS@", checks))
