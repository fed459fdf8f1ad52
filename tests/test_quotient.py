"""The coarsest level's factorisation and its inverse's columns divide by a
pivot through its reciprocal, which a pivot below 2^-1024 does not have: 0
times it would be NaN."""
import os
import subprocess

from test_pdl_sources import CSRC, body_of, sources

MAIN = r"""
#include <cmath>
#include <initializer_list>
#include <cstdio>
#include "dp_quotient.h"
int main() {
  int off = 0;
  auto recip = [](double d) { return d != 0.0 ? 1.0 / d : 0.0; };
  const double tiny[] = {ldexp(1.0, -1030), -ldexp(3.0, -1040), 4.9e-324, ldexp(1.0, 1022),
                         -ldexp(1.5, 1023)};
  for (double d : tiny)   // no normal reciprocal: the division
    for (double f : {0.0, 1.0, -0.5, 0.25, 1.0 / 3.0}) {
      double a = f * d, q = dp::quotient(a, d, recip(d));
      off += !(q == a / d) || !std::isfinite(q);
    }
  for (double d : {1.0, -3.0, 7e-200, 1e300, ldexp(1.0, -1022)})   // the product
    for (double a : {0.0, 1.0, -2.5, 1e-3, 4e5}) {
      double q = dp::quotient(a * d, d, recip(d)), e = (a * d) * (1.0 / d);
      off += !(q == e || (q != q && e != e));
    }
  for (double a : {0.0, 1.0, -2.0}) off += dp::quotient(a, 0.0, recip(0.0)) != 0.0;
  std::printf("%d\n", off);
}
"""


def test_quotients_by_extreme_pivots(tmp_path):
    src, exe = tmp_path / "quotient.cpp", tmp_path / "quotient"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout == "0\n"


def test_the_dense_factorisation_divides_by_quotient():
    text = sources()
    for kernel in ("k_dense_factor", "k_dense_cols"):
        body = body_of(text, kernel, "__global__")
        assert "quotient(" in body and "] * r;" not in body and "* rd[" not in body, kernel
