"""The triangles' solid angles behind both inside checks (csrc/solid_angle.h), compiled with the host C++ compiler:
float64 accuracy against long double, the surface test, and closed surfaces' sums; both checks call this function."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_21713_gb300", "csrc")

# Tolerance: det and den are sums of a few products of at most s3 = |a||b||c| each, the lengths within two roundings: 16
# u s3 of error in either, which turns the angle by 16 u s3 / hypot(det, den); atan2 itself and the result a few u of pi.
DRIVER = r"""
#include <cstdio>
#include <random>
#include "solid_angle.h"
typedef long double L;
int main() {
  const double u = 0x1p-53;
  std::mt19937_64 g(7);
  std::normal_distribution<double> nd;
  int bad = 0;
  for (int n = 0; n < 200000; ++n) {
    double v[3][3];
    const double size = std::exp(2.0 * nd(g));  // from slivers seen from afar to triangles around the point
    double c[3] = {nd(g), nd(g), nd(g)};
    for (auto& p : v)
      for (int d = 0; d < 3; ++d) p[d] = c[d] + size * nd(g);
    double l[3];
    L ll[3], w[3][3];
    for (int k = 0; k < 3; ++k) {
      for (int d = 0; d < 3; ++d) w[k][d] = v[k][d];
      l[k] = std::sqrt(v[k][0] * v[k][0] + v[k][1] * v[k][1] + v[k][2] * v[k][2]);
      ll[k] = sqrtl(w[k][0] * w[k][0] + w[k][1] * w[k][1] + w[k][2] * w[k][2]);
    }
    auto dot = [&](int i, int j) { return w[i][0] * w[j][0] + w[i][1] * w[j][1] + w[i][2] * w[j][2]; };
    const L det = w[0][0] * (w[1][1] * w[2][2] - w[1][2] * w[2][1]) - w[0][1] * (w[1][0] * w[2][2] - w[1][2] * w[2][0]) +
                  w[0][2] * (w[1][0] * w[2][1] - w[1][1] * w[2][0]);
    const L s3 = ll[0] * ll[1] * ll[2], den = s3 + dot(0, 1) * ll[2] + dot(1, 2) * ll[0] + dot(2, 0) * ll[1];
    bool on = false;
    const double h = pbfb::half_solid_angle(v[0][0], v[0][1], v[0][2], v[1][0], v[1][1], v[1][2], v[2][0], v[2][1],
                                            v[2][2], l[0], l[1], l[2], &on);
    const L tol = u * (8 + 16 * s3 / hypotl(det, den));
    bad += on || !(fabsl(h - atan2l(det, den)) <= tol);
  }
  // a corner, a point within and points beside a triangle in its plane
  auto on_at = [](double x, double y) {
    const double P[3][2] = {{0, 0}, {4, 0}, {0, 4}};
    double a[3][3], l[3];
    for (int k = 0; k < 3; ++k) {
      a[k][0] = P[k][0] - x, a[k][1] = P[k][1] - y, a[k][2] = 0.0;
      l[k] = std::sqrt(a[k][0] * a[k][0] + a[k][1] * a[k][1]);
    }
    bool on = false;
    pbfb::half_solid_angle(a[0][0], a[0][1], a[0][2], a[1][0], a[1][1], a[1][2], a[2][0], a[2][1], a[2][2], l[0], l[1],
                           l[2], &on);
    return on;
  };
  bad += !on_at(0, 0) + !on_at(1, 1) + !on_at(0.5, 3) + on_at(5, 5) + on_at(-1, 2);
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


def test_solid_angles_in_float64(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "driver.cpp"), "-o", str(tmp_path / "driver")],
                   check=True)
    subprocess.run([str(tmp_path / "driver")], check=True)


@pytest.mark.parametrize("path,name", [("bem_kernels.cu", "k_winding"), ("mesh_setup.cu", "winding_numbers")])
def test_both_checks_use_them(path, name):
    src = open(os.path.join(CSRC, path)).read()
    body = re.search(name + r"\(.*?\n\}", src, re.S).group(0)
    assert "half_solid_angle(" in body and "atan2" not in body and "float" not in body.replace("<float", "")
