"""The limiter tables fit the kernels' fixed-point sums (csrc/tables.cpp: sums_fit), and the check
looks at the sums: tables whose every entry fits but whose sum does not are refused."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cmath>
#include <cstdio>
#include "tables.h"
using namespace dgt;
int main() {
  for (int parent = 0; parent < 2; ++parent)
    for (int N = 1; N <= 3; ++N) {
      Tabs t;
      if (build_tables(N, &t, parent)) return 1;
      // the sums as the kernels form them, largest terms: |X| < 2^62, P < 2^62, with their rounding terms
      for (int g = 0; g < t.NG; ++g) {
        long double T[2] = {0, 0}, S[2] = {0, 0};
        for (int i = 0; i <= N; ++i) {
          const int k = i == weno_neg(N, g, parent);
          S[k] += ldexpl(t.wh[g][i], 61);
          for (int j = 0; j < N; ++j) T[k] += ldexpl(fabsl((long double)t.wc[g][i][j]), 60) + 1;
        }
        for (int k = 0; k < 2; ++k)
          if (!(T[k] < 0x1p63L) || !(S[k] < 0x1p63L)) return 2;
        std::printf("%d %d %d: |wc| %.3f %.3f  wh %.3f %.3f\n", parent, N, g, (double)ldexpl(T[0], -60),
                    (double)ldexpl(T[1], -60), (double)ldexpl(S[0], -61), (double)ldexpl(S[1], -61));
      }
      Tabs u = t;
      for (int i = 0; i <= N; ++i)
        for (int j = 0; j < N; ++j) u.wc[0][i][j] = (j & 1 ? -1 : 1) * 7.5 / (N * (N + 1));
      const bool each = 7.5 / (N * (N + 1)) < 2.0;
      if (sums_fit(u, parent) != each) return 3;
      if (N > 1) {  // entries below 2, sums of 8 and above, and of 4
        for (int i = 0; i <= N; ++i)
          for (int j = 0; j < N; ++j) u.wc[0][i][j] = (j & 1 ? -1 : 1) * 8.2 / (N * (N + 1));
        if (sums_fit(u, parent)) return 4;
        u = t;
        for (int i = 0; i <= N; ++i) u.wh[0][i] = 1.4;
        if (sums_fit(u, parent)) return 5;
      }
    }
  return 0;
}
"""


def test_sums_fit(tmp_path):
    csrc = os.path.join(ROOT, "paper_1904_11147_gb300", "csrc")
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", csrc, str(tmp_path / "t.cpp"), os.path.join(csrc, "tables.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    print(r.stdout)
    assert r.returncode == 0
