"""The split of a search into work units tries one unit count per unit size; it
picks what trying every count picks, and its time does not grow with the
number of simplices."""
import os
import subprocess

from paper_2007_09884_gb300 import build as B

MAIN = r"""
#include <chrono>
#include <cstdio>
#include "split.h"
using namespace opmm;

static int every_count(int n, int S, const SplitShape& s, int blocks) {
  const int least = (S + s.G - 1) / s.G;
  double best = 1e300;
  int pick = least;
  for (int ng = least; ng <= S; ++ng) {
    const double turns = std::max(1.0, (double)(((long long)n * ng + blocks - 1) / blocks));
    const double t = turns * unit_step(s, (S + ng - 1) / ng);
    if (t < best * 0.999) { best = t; pick = ng; }
  }
  return pick == least && (S % s.G == 0 || least > 8) ? 0 : pick;
}

int main() {
  const SplitShape shapes[] = {{32, 2, 22}, {16, 2, 22}, {64, 2, 22}, {64, 4, 22}, {72, 3, 22}, {54, 2, 13}, {108, 4, 13}};
  long long cases = 0;
  for (const SplitShape& s : shapes)
    for (int blocks : {152, 304, 456})
      for (int n : {1, 2, 3, 5, 17, 75, 151, 152, 153, 400, 1024, 2500, 40000})
        for (int S = 1; S < 6000; S += S < 700 ? 1 : 37) {
          ++cases;
          const int a = split_units(n, S, s, blocks), b = every_count(n, S, s, blocks);
          if (a != b) {
            printf("n %d S %d G %d blocks %d: %d, every count %d\n", n, S, s.G, blocks, a, b);
            return 1;
          }
        }
  const auto t0 = std::chrono::steady_clock::now();
  int sum = 0;
  for (int i = 0; i < 1000; ++i) sum += split_units(1 + i % 3, 90000000 + i, shapes[i % 7], 152);
  const double s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  printf("%lld cases, 1000 splits of 9e7 simplices %.4f s (%d)\n", cases, s, sum);
  return s < 1.0 ? 0 : 2;   // one of them took 0.4 s when every count was tried
}
"""


def test_one_count_per_unit_size_picks_the_same(tmp_path):
    src, exe = tmp_path / "split.cpp", str(tmp_path / "split")
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", B.CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
