"""Split of the far fields by triangle pairs (csrc/pair_split.h), compiled with the host C++ compiler: its groups tile the
surface, its tasks stay within four times those aimed at (few surfaces: at least one), and no accepted tuning takes
more partial rows than the memory estimate of a solve counts."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_21713_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "pair_split.h"
using namespace pbfb;
int main() {
  int bad = 0;
  auto look = [&](int nt, bool f64, int bps) {
    const int want = pair_want(f64, bps);
    const PairSplit s = pair_split(nt, want, f64);
    const int limit = s.nsub * s.K > 1 ? (f64 ? 24000 : 8192) : 4 * want;
    if (s.nT != (nt + 31) / 32 || (s.G - 1) * s.tpg >= s.nT || s.G * s.tpg < s.nT || 32 % s.K || s.ntask < 1 ||
        s.ntask > limit || s.ntask != s.G * (s.G + 1) / 2 * s.K * s.nsub || s.rows > pair_rows_max(nt)) {
      if (bad++ < 5)
        std::printf("nt %d f64 %d bps %d: G %d tpg %d tasks %d rows %zu of %zu\n", nt, f64, bps, s.G, s.tpg, s.ntask,
                    s.rows, pair_rows_max(nt));
    }
  };
  for (int nt = 1; nt <= 60000; nt += nt < 3000 ? 1 : 17) {
    look(nt, true, 0);
    for (int bps = 0; bps <= 64; bps += nt < 3000 && nt % 50 ? 16 : 1) look(nt, false, bps);
  }
  for (int nt : {12543, 12544, 12575, 12576, 12577, 12607, 12608, 12609, 25184, 25216, 200000, 1000000})
    for (int bps = 0; bps <= 64; ++bps) look(nt, false, bps);
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


def test_splits(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "driver.cpp"), "-o", str(tmp_path / "driver")],
                   check=True)
    subprocess.run([str(tmp_path / "driver")], check=True)
