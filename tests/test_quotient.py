"""The coarsest level's factorisation forms its multipliers, and the columns of
its inverse their entries, as quotients: the product with a rounded reciprocal
has a second rounding, and a pivot below 2^-1024 has no finite reciprocal."""
import os
import subprocess

from test_pdl_sources import CSRC, body_of, sources

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "dp_quotient.h"
int main() {
  std::mt19937_64 g(1);
  auto value = [&](int kind) {
    uint64_t b = g();
    if (kind == 0) b = (b & 0x800fffffffffffffull) | ((uint64_t)(1023 + (int)(g() % 7) - 3) << 52);
    if (kind == 2) b |= 0x000fffff00000000ull >> (g() % 20);
    double v;
    memcpy(&v, &b, 8);
    return v;
  };
  long off = 0, product = 0, n = 0;
  auto same = [](double x, double y) { return x == y ? std::signbit(x) == std::signbit(y) : x != x && y != y; };
  for (int i = 0; i < 6000000; ++i) {
    double a = value(i % 3), d = value((i / 3) % 3);
    if (d == 0.0) continue;
    double r = 1.0 / d;
    off += !same(dp::quotient(a, d, r), a / d);
    product += !same(a * r, a / d);
    ++n;
  }
  const double s[] = {0.0, -0.0, 1.0, -3.0, INFINITY, -INFINITY, NAN, 4.9e-324, 2e-309, 2e-308, 1e-200,
                      1e200, 1.7e308};
  for (double a : s)
    for (double d : s) {
      if (d == 0.0) off += dp::quotient(a, d, 0.0) != 0.0;
      else off += !same(dp::quotient(a, d, 1.0 / d), a / d);
    }
  std::printf("%ld %ld %ld\n", n, off, product);
}
"""


def test_quotients_are_those_of_the_division(tmp_path):
    """Six million pairs over a few binades and over the whole range, and the
    special values: bit for bit the division (the product alone is not)."""
    src, exe = tmp_path / "quotient.cpp", tmp_path / "quotient"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)
    n, off, product = map(int, subprocess.run([str(exe)], capture_output=True, text=True,
                                              check=True).stdout.split())
    assert n > 5_900_000 and off == 0 and product > n // 20


def test_the_dense_factorisation_forms_quotients():
    text = sources()
    for kernel in ("k_dense_factor", "k_dense_cols"):
        body = body_of(text, kernel, "__global__")
        assert "quotient(" in body and "] * r;" not in body and "* rd[" not in body, kernel
