"""HostRanges (csrc/host_ranges.h), compiled with the host C++ compiler: the passes of one object see the same ranges
even where the processor count changes between them (mesh creation keeps one pass's buffers by range for the next),
the ranges tile [0, n), and an exception of a range reaches the caller after all have ended."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_21713_gb300", "csrc")

DRIVER = r"""
#include <atomic>
#include <cstdio>
#include <stdexcept>
#include "host_ranges.h"
static int g_procs = 8;
extern "C" int get_nprocs() noexcept { return g_procs; }  // what std::thread::hardware_concurrency() reads
struct Pass { int64_t lo[pbfb::HOST_THREADS], hi[pbfb::HOST_THREADS]; };
static Pass pass(const pbfb::HostRanges& r) {
  Pass p;
  for (int k = 0; k < pbfb::HOST_THREADS; ++k) p.lo[k] = p.hi[k] = -1;
  r.run([&](int k, int64_t i0, int64_t i1) { p.lo[k] = i0; p.hi[k] = i1; });
  return p;
}
int main() {
  if (std::thread::hardware_concurrency() != 8u) return 77;  // the count cannot be set here
  int bad = 0;
  for (int64_t n : {0, 1, 7, 31, 32, 100, 1000, 100000})
    for (int64_t grain : {1, 32, 4096}) {
      g_procs = 8;
      const pbfb::HostRanges r(n, grain);
      const Pass a = pass(r);
      for (int procs : {3, 64, 1}) {
        g_procs = procs;
        const Pass b = pass(r);
        for (int k = 0; k < pbfb::HOST_THREADS; ++k) bad += a.lo[k] != b.lo[k] || a.hi[k] != b.hi[k];
      }
      int64_t at = 0;
      for (int k = 0; k < pbfb::HOST_THREADS && a.lo[k] >= 0; ++k) {
        bad += a.lo[k] != at || a.hi[k] < a.lo[k];
        at = a.hi[k];
      }
      bad += at != n;
    }
  g_procs = 8;
  std::atomic<int> ended{0};
  bool caught = false;
  try {
    pbfb::HostRanges(8, 1).run([&](int k, int64_t, int64_t) {
      if (k == 3) throw std::runtime_error("range");
      ++ended;
    });
  } catch (const std::runtime_error&) {
    caught = true;
  }
  bad += !caught || ended != 7;
  std::printf("%d\n", bad);
  return bad ? 1 : 0;
}
"""


def test_passes_share_a_partition(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "driver.cpp"), "-o",
                    str(tmp_path / "driver")], check=True)
    code = subprocess.run([str(tmp_path / "driver")]).returncode
    if code == 77:
        pytest.skip("the processor count cannot be set")
    assert code == 0


def test_mesh_creation_has_no_other_partition():
    src = open(os.path.join(CSRC, "mesh_setup.cu")).read()
    assert src.count("hardware_concurrency") <= 1  # the winding numbers' single pass
    assert "HostRanges" in src
