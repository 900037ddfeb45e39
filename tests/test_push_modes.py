"""The fused pass's split of a line's modes over component groups (csrc/push_modes.h), on the
host: for every elements-per-thread and group count the passes use, each mode is updated once
with its own coefficients, and no coefficient outside the line's row of L/2 + 1 entries is
read, also by groups that have no mode (FP64: 6 groups of 4 elements per thread)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1608_05739_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include <vector>
#include "push_modes.h"
template <int EPT> int check(int T) {
  const int L = EPT * T;
  for (int G = 1; G <= 6; ++G)
    for (int t = 0; t < T; ++t) {
      std::vector<int> seen(EPT, 0);
      bool ok = true;
      for (int grp = 0; grp < G; ++grp)
        psatd::push_mode_pairs<EPT>(
            grp, G,
            [&](int m) {
              const int e = psatd::coef_entry(t + T * m, L);
              ok = ok && m >= 0 && m < EPT && e >= 0 && e <= L / 2;
              return m;
            },
            [&](int m, int q) {
              ok = ok && m == q && m % G == grp;
              if (m >= 0 && m < EPT) ++seen[m];
            });
      for (int n : seen) ok = ok && n == 1;
      if (!ok) {
        std::printf("ept %d T %d G %d t %d\n", EPT, T, G, t);
        return 1;
      }
    }
  return 0;
}
int main() {
  int bad = 0;
  for (int T : {1, 2, 4, 8, 16, 32, 64, 128, 256})
    bad += check<4>(T) + check<8>(T) + check<12>(T) + check<16>(T) + check<20>(T);
  return bad != 0;
}
"""


def test_every_mode_once_and_no_entry_outside_the_row(tmp_path):
    src, exe = tmp_path / "modes.cpp", tmp_path / "modes"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
