"""Launch plans of the CTA-pair kernels (fw_pair_plan.h, plain C++): asked for by several host threads at once, for other layers each,
as callers of different layers may do."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include "fw_pair_plan.h"
using namespace fw;
static std::vector<PairSpec> list_of(int k, bool second, int layers) {
  std::vector<PairSpec> v(layers);
  for (int i = 0; i < layers; ++i) {
    PairSpec& p = v[i];
    p.M = 1024 + 16 * ((7 * k + 5 * i) % 200); p.rows = p.M; p.bf16 = false; p.full = true; p.colsums = false;
    p.sym_out = second; p.fix = second ? 0 : 1; p.split_cap = 1;
  }
  return v;
}
static long plan(int k, bool second, int layers) {
  std::vector<PairSpec> v = list_of(k, second, layers);
  const int panel = pair_choose_panel(v, 74);
  for (PairSpec& p : v) { p.panel = panel; pair_tiles(p.M, true, panel, p.sym_out, p.tiles); }
  pair_choose_splits(v, 74, 0, false);
  long sum = panel;
  for (const PairSpec& p : v) sum = sum * 31 + p.splits * 1000 + p.per;
  return sum;
}
static int threads() {
  const int T = 8, N = 80;
  std::vector<std::vector<long>> got(T, std::vector<long>(N));
  std::vector<std::thread> th;
  for (int t = 0; t < T; ++t)
    th.emplace_back([&, t] { for (int k = 0; k < N; ++k) got[t][k] = plan(N * t / 2 + k, k & 1, 2); });
  for (std::thread& t : th) t.join();
  for (int t = 0; t < T; ++t)
    for (int k = 0; k < N; ++k)
      if (got[t][k] != plan(N * t / 2 + k, k & 1, 2)) return 1;
  return 0;
}
// microseconds of choosing the width of both products' tiles, the first time and at best later
static int repeated() {
  const std::vector<PairSpec> a = list_of(3, false, 16), b = list_of(3, true, 16);
  double first = 0, later = 1e300;
  for (int i = 0; i < 20; ++i) {
    const auto t0 = std::chrono::steady_clock::now();
    pair_choose_panel(a, 74);
    pair_choose_panel(b, 74);
    const double us = std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count();
    if (i == 0) first = us;
    else later = std::min(later, us);
  }
  std::printf("%.1f %.1f\n", first, later);
  return 0;
}
int main(int argc, char**) { return argc > 1 ? repeated() : threads(); }
"""


def compiled(tmp_path, flags):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "plan.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "plan")
    r = subprocess.run([gxx, "-std=c++17", "-pthread", "-I" + os.path.join(ROOT, "paper_2010_01546_b200", "csrc"), str(src), "-o", exe]
                       + flags, capture_output=True, text=True)
    if r.returncode != 0 and "tsan" in r.stderr:
        pytest.skip("no thread sanitizer")
    assert r.returncode == 0, r.stderr
    return exe


def test_plans_of_several_threads(tmp_path):
    r = subprocess.run([compiled(tmp_path, ["-O1", "-g", "-fsanitize=thread"])], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]


def test_a_step_does_not_search_again(tmp_path):
    """A re-sync asks for the tiles of its first product, then for those of its second, every step."""
    r = subprocess.run([compiled(tmp_path, ["-O2"]), "repeated"], capture_output=True, text=True, timeout=300)
    first, later = map(float, r.stdout.split())
    assert 10 * later < first, (first, later)
