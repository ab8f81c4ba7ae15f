"""Scalar functions of the kernels, compiled for the host: their rounding errors against the textbook
forms, both from a wider type."""
import os
import subprocess

import pytest

from paper_1709_09347_gb300 import build

PRELUDE = r"""
#include <cstdio>
#include <random>
typedef long double W;
struct Errors {
  double top = 0, sum = 0;
  long n = 0;
  void add(double e) { if (e > top) top = e; sum += e * e; ++n; }
  void print() const { printf("%.6g %.6g\n", top, sqrt(sum / n)); }
};
"""

ROTATION = r"""
#include "rotation.cuh"
""" + PRELUDE + r"""
int main() {
  std::mt19937_64 g(3);
  std::normal_distribution<double> nd;
  Errors own, book;
  for (int i = 0; i < 400000; ++i) {
    const double al = exp(3 * nd(g)), be = exp(3 * nd(g)), m = 0.9 * sqrt(al * be) * exp2(-(double)(g() % 45)), ph = 9 * nd(g);
    const double gx = m * cos(ph), gy = m * sin(ph);
    W ag = hypotl(gx, gy), z = ((W)be - al) / (2 * ag), t = (z >= 0 ? 1 : -1) / (fabsl(z) + sqrtl(1 + z * z));
    W s = t / sqrtl(1 + t * t), x = s * gx / ag, y = s * gy / ag;
    double c;
    double2 sp;
    if (!cbs::pair_rotation(al, be, gx, gy, 1e-16, c, sp)) return 1;
    own.add((double)(hypotl(sp.x - x, sp.y - y) / fabsl(s)));
    const double bg = hypot(gx, gy), bz = (be - al) / (2 * bg), bt = (bz >= 0 ? 1 : -1) / (fabs(bz) + sqrt(1 + bz * bz));
    const double bs = bt / sqrt(1 + bt * bt);
    book.add((double)(hypotl(bs * gx / bg - x, bs * gy / bg - y) / fabsl(s)));
  }
  own.print();
  book.print();
  return 0;
}
"""


def _errors(tmp_path, source):
    """(largest, root mean square) relative error of the kernels' form and of the textbook's."""
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    cu, exe = str(tmp_path / "t.cu"), str(tmp_path / "t")
    with open(cu, "w") as f:
        f.write(source)
    subprocess.run([nvcc, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", build.INCLUDE, cu, "-o", exe],
                   check=True, capture_output=True, env=dict(os.environ))
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    return [tuple(float(v) for v in out[k:k + 2]) for k in (0, 2)]


def test_jacobi_rotation(tmp_path):
    """The sine of the rotation, over 90 orders of 2 of the columns' angle, no less accurate than
    t = 1 / (|zeta| + sqrt(1 + zeta^2)) in divisions and square roots."""
    own, book = _errors(tmp_path, ROTATION)
    assert own[0] <= book[0] and own[1] <= book[1], (own, book)
