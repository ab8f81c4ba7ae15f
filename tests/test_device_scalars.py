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

QUOTIENT = r"""
#include "common.cuh"
""" + PRELUDE + r"""
static double2 smith(double2 a, double2 b) {
  if (fabs(b.x) >= fabs(b.y)) {
    const double r = b.y / b.x, d = fma(b.y, r, b.x);
    return make_double2(fma(a.y, r, a.x) / d, fma(-a.x, r, a.y) / d);
  }
  const double r = b.x / b.y, d = fma(b.x, r, b.y);
  return make_double2(fma(a.x, r, a.y) / d, fma(a.y, r, -a.x) / d);
}
int main() {
  std::mt19937_64 g(5);
  std::normal_distribution<double> nd;
  Errors own, book;
  for (int i = 0; i < 400000; ++i) {
    const double s = exp2((int)(g() % 40) - 20), t = exp2((int)(g() % 600) - 300), u = exp2((int)(g() % 400) - 200);
    const double2 a = make_double2(nd(g) * t, nd(g) * t), b = make_double2(nd(g) * u, nd(g) * u * (i & 1 ? s : 1));
    const W p = b.x, q = b.y, n = p * p + q * q;
    const W x = ((W)a.x * p + (W)a.y * q) / n, y = ((W)a.y * p - (W)a.x * q) / n, m = hypotl(x, y);
    const double2 o = cbs::cdiv(a, b), k = smith(a, b);
    own.add((double)(hypotl(o.x - x, o.y - y) / m));
    book.add((double)(hypotl(k.x - x, k.y - y) / m));
  }
  own.print();
  book.print();
  // ends of the range: the results stay finite and right
  const double e[6][4] = {{1e250, 1e250, 1e90, 0}, {1e-250, 0, 1e-90, 1e-90}, {0, 0, 3, 4}, {1e-300, 0, 1e-120, 0},
                          {1e300, 0, 1e120, 0}, {3e-160, 4e-160, 1e-99, 0}};
  for (const auto &v : e) {
    const double2 q = cbs::cdiv(make_double2(v[0], v[1]), make_double2(v[2], v[3]));
    const W n = (W)v[2] * v[2] + (W)v[3] * v[3], x = ((W)v[0] * v[2] + (W)v[1] * v[3]) / n, y = ((W)v[1] * v[2] - (W)v[0] * v[3]) / n;
    if (!(hypotl(q.x - x, q.y - y) <= 1e-15 * hypotl(x, y))) return 2;
  }
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


def test_complex_quotient(tmp_path):
    """Relative to the modulus, no less accurate than Smith's algorithm."""
    own, book = _errors(tmp_path, QUOTIENT)
    assert own[0] <= book[0] and own[1] <= book[1], (own, book)
