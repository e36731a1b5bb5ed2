"""The host's split of a launch into ranges (csrc/hist_plan.h) against its
definition, for inputs of all sizes and orders: every CTA's range, the inputs
that start in it and the ranges the groups of warps take."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1011_0235_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <stdlib.h>
#include <random>
#include <vector>
#include "hist_plan.h"
using namespace histlib;
typedef unsigned long long u64;
int main() {
  std::mt19937_64 r(11);
  const u64 small_max = 256u << 10;
  for (int it = 0; it < 4000; ++it) {
    const uint32_t count = 1 + r() % (it % 4 ? 40 : 1024), grid = 1 + r() % kPlanCtas;
    const u64 top[] = {1, 100, 70000, 300000, 5000000, 1ull << 32}, fixed = 1 + r() % (256u << 10);
    std::vector<u64> n(count), c(count), pos(1, 0);
    for (uint32_t i = 0; i < count; ++i) {
      n[i] = it % 5 ? r() % top[r() % 6] : 1 + r() % 70000;
      c[i] = n[i] + fixed + (i + 2 >= count ? 131072 : 0);
      pos.push_back(pos[i] + c[i]);
    }
    const u64 W = pos[count], range = W / grid;
    auto size = [&](uint32_t i) { return n[i]; };
    auto small = [&](uint32_t i) { return n[i] && n[i] <= small_max && n[i] * 4 <= range; };
    static PlanCosts<1024> pc;
    static RangePlan p;
    plan_costs(&pc, count, size, [&](uint32_t i) { return c[i]; });
    plan_ranges(&p, pc, count, grid, small_max, size);
    auto check = [&](bool ok, const char* what) {
      if (!ok) {
        printf("%s, plan %d\n", what, it);
        exit(1);
      }
    };
    u64 small_cost = 0, bytes = 0;
    for (uint32_t i = 0; i < count; ++i) {
      if (small(i)) small_cost += c[i];
      bytes += n[i];
    }
    check(p.range == range && pc.bytes == bytes, "totals");
    check(p.group_max == (2 * small_cost >= W ? small_max : 0), "group_max");
    for (uint32_t b = 0; b <= grid; ++b) {
      const u64 lo = W * b / grid;
      uint32_t s = 0, j = 0;
      while (s < count && pos[s] < lo) ++s;
      check(p.lo[b] == lo && p.s[b] == s, "range");
      if (b == grid) break;
      while (j + 1 < count && pos[j + 1] <= lo) ++j;
      check(p.j[b] == j && p.pre[b] == pos[j], "first input");
    }
    for (uint32_t b = 0; b < grid; ++b) {
      bool only = p.group_max != 0;
      for (uint32_t k = p.j[b]; k < p.s[b] && only; ++k) only = n[k] * 4 <= range;
      for (uint32_t k = p.s[b]; k < p.s[b + 1] && only; ++k) only = small(k);
      check(only == (p.groups[b >> 5] >> (b & 31) & 1), "groups");
    }
  }
  return 0;
}
"""


def test_ranges_by_definition(tmp_path):
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    src = tmp_path / "plan.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "plan")
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-I", CSRC, "-I", cuda, str(src), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
