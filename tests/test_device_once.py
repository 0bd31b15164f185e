"""Per-device set-up (constant tables, kernel attributes): DeviceOnce (csrc/device_once.h) runs a function once for each
device that asks for it, again after a failure, and one caller at a time; compiled with the host C++ compiler.
No once-per-process flag stands before device state, and every such function of mesh creation goes through it."""
import glob
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_21713_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.h"
int main() {
  pbfb::DeviceOnce once;
  int count[80] = {};
  bool fail = true;
  auto ask = [&](int dev) { return once.run(dev, [&] { ++count[dev]; return 0; }); };
  int bad = 0;
  for (int dev : {0, 1, 0, 63, 1, 63, 0}) bad += ask(dev) != 0;
  bad += count[0] != 1 || count[1] != 1 || count[63] != 1 || count[2] != 0;
  // a failure is reported and not remembered
  auto failing = [&](int dev) { return once.run(dev, [&] { ++count[dev]; return fail ? 7 : 0; }); };
  bad += failing(2) != 7 || failing(2) != 7 || count[2] != 2;
  fail = false;
  bad += failing(2) != 0 || failing(2) != 0 || count[2] != 3;
  // past the mask: each time
  ask(64);
  ask(64);
  bad += count[64] != 2;
  std::vector<std::thread> th;
  for (int k = 0; k < 8; ++k) th.emplace_back([&] { ask(5); });
  for (auto& t : th) t.join();
  bad += count[5] != 1;
  std::printf("%d\n", bad);
  return bad;
}
"""


def test_once_per_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "driver.cpp"), "-o",
                    str(tmp_path / "driver")], check=True)
    subprocess.run([str(tmp_path / "driver")], check=True)


def body(name):
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        m = re.search(r"^int " + name + r"\(\) \{\n(.*?)^\}", open(path).read(), re.S | re.M)
        if m:
            return m.group(1)
    raise AssertionError(name)


@pytest.mark.parametrize("name", ["init_quadrature", "init_pair_attributes", "init_dense_attributes"])
def test_set_up_is_per_device(name):
    b = body(name)
    assert "DeviceOnce" in b and "cudaGetDevice" in b


def test_no_flag_per_process():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        assert not re.search(r"static\s+(?:std::atomic<)?bool>?\s+\w+\s*(?:=|;|\{)", open(path).read()), path


def test_symbol_copies_are_waited_for():
    """The tables are copied on the legacy stream from pageable memory, so that a copy may still be on its way when
    the call returns; meshes run on non-blocking streams, which wait for no other."""
    b = body("init_quadrature")
    last = max(b.index("init_correction_rules"), b.rindex("cudaMemcpyToSymbol"))
    assert "cudaStreamSynchronize(cudaStreamLegacy)" in b[last:]
