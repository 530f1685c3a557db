"""Characters exp(2 pi i n / d) of the sectors' tables (csrc/character.h), compiled for the host,
against 80-bit arithmetic (x86) or better."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_05028_gb300", "csrc")

SRC = r"""
#include "character.h"
#include <cstdio>
int main() {
  const long double pi = 3.14159265358979323846264338327950288L;
  double worst = 0, plain = 0;
  bool exact = true;
  for (int d = 1; d <= 400; d++)
    for (int n = -d; n <= 2 * d; n++) {
      double c, s;
      ed_character(n, d, &c, &s);
      const long double a = 2 * pi * n / d, ec = std::cos(a), es = std::sin(a);
      worst = std::fmax(worst, (double)std::fmax(std::fabs(c - ec), std::fabs(s - es)));
      const double b = 2.0 * M_PI * (double)n / (double)d;
      if (n >= 0 && n < d) plain = std::fmax(plain, (double)std::fmax(std::fabs(std::cos(b) - ec), std::fabs(std::sin(b) - es)));
      if (4 * n % d == 0) {   // multiples of a quarter turn
        const int q = ((4 * n / d) % 4 + 4) % 4;
        exact = exact && c == (q == 0) - (q == 2) && s == (q == 1) - (q == 3);
      }
    }
  printf("%.3g %.3g %d", worst, plain, exact);
}
"""


def test_characters(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    worst, plain, exact = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    # half an ulp of cos or sin and half an ulp of the correction's sum, both below 1
    assert float(worst) <= 1.2e-16 and exact == "1"
    assert float(plain) > 3e-16      # what the rounded angle costs
