"""The kernels' division by launch-time numbers (csrc/fast_div.cuh), compiled for the host, against the
division operator: every divisor and dividend of a small range, and the edges of the whole one."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "fast_div.cuh"
#include <cstdio>
#include <random>
int main() {
  const int top = 0x7fffffff;
  auto same = [](int n, int d) { return spiffy::FastDiv::by(d).div(n) == n / d; };
  for (int d = 1; d <= 700; ++d)
    for (int n = 0; n <= 3000; ++n)
      if (!same(n, d)) return printf("%d / %d\n", n, d), 1;
  std::mt19937 g(1);
  std::uniform_int_distribution<int> any(1, top);
  for (int i = 0; i < 2000000; ++i) {
    const int d = any(g) >> (g() % 31), n = any(g) >> (g() % 31);
    if (d == 0) continue;
    const long long k = (long long)(n / d) * d;  // a multiple of d and its neighbours
    for (long long m : {(long long)n, k, k - 1, k + d - 1, (long long)top, (long long)top - d})
      if (m >= 0 && m <= top && !same((int)m, d)) return printf("%lld / %d\n", m, d), 1;
  }
  for (int s = 0; s < 31; ++s)
    for (long long d : {(1LL << s) - 1, 1LL << s, (1LL << s) + 1})
      for (int n : {0, 1, top - 1, top})
        if (d >= 1 && d <= top && !same(n, (int)d)) return printf("%d / %lld\n", n, d), 1;
  return 0;
}
"""


def test_equals_division(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_2509_18085_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout
