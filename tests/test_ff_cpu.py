"""The float-float sums of the frequency-batched chi0's recombination (csrc/ff.h) on
the host: sums of products against extended precision, and against the textbook
step that renormalises the pair after every term.

A term's rounding errors are those of the error pair (2^-24 of a number at 2^-24 of
the sum): 2^-48 of the sum each, of random sign.  The tests' sums of n terms of random
sign stay at sqrt(n) terms, so the error over the sum of magnitudes is a few 2^-48 /
sqrt(n) times sqrt(n) steps / n: below 2^-48 whatever n.  (4000 sums per figure: it is good to 2 %, so 5 % more than the
textbook step's is allowed.)"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cmath>
#include <random>
#include "ff.h"
typedef long double ld;
static void textbook(float& h, float& l, float kx, float ky, float x0, float x1) {
  const float p = kx * x0;
  const float t = fmaf(kx, x0, -p) + fmaf(kx, x1, ky * x0);
  const float s = h + p, bb = s - h, e = (h - (s - bb)) + (p - bb);
  const float q = e + t + l;
  h = s + q;
  l = q - (h - s);
}
int main() {
  std::mt19937 r(7);
  std::normal_distribution<double> g;
  for (int n : {6, 30, 150, 600}) {
    double a = 0, b = 0, c2 = 0, worst = 0;
    const int T = 4000;
    for (int t = 0; t < T; ++t) {
      float h = 0, l = 0, h2 = 0, l2 = 0, h3 = 0, l3 = 0, pk[4] = {0, 0, 0, 0};
      ld ex = 0, mag = 0;
      for (int i = 0; i < n; ++i) {
        const double c = g(r) * ldexp(1.0, -(i % 5)), x = g(r);
        const float kx = c, ky = c - (double)kx, x0 = x, x1 = x - (double)x0;
        ex += ((ld)kx + ky) * ((ld)x0 + x1);
        mag += fabsl((ld)kx * x0);
        rpa::ff_fma(h, l, kx, ky, x0, x1);
        textbook(h2, l2, kx, ky, x0, x1);
        if (i % 2) {
          rpa::ff_fma2(h3, l3, pk[0], pk[1], pk[2], pk[3], kx, ky, x0, x1);
          if (fabsf(l3) > ldexpf(fabsf(h3), -24)) worst = 1;
        }
        pk[0] = kx, pk[1] = ky, pk[2] = x0, pk[3] = x1;
        if (fabsf(l) > ldexpf(fabsf(h), -24)) worst = 1;
      }
      const double u = (double)(((ld)h + l - ex) / mag), v = (double)(((ld)h2 + l2 - ex) / mag),
                   w = (double)(((ld)h3 + l3 - ex) / mag);
      a += u * u;
      b += v * v;
      c2 += w * w;
    }
    printf("%d %.6e %.6e %.6e %g\n", n, sqrt(a / T), sqrt(b / T), sqrt(c2 / T), worst);
  }
}
"""


def test_sums_keep_the_textbook_precision(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2505_06021_gb300", "csrc"), str(tmp_path / "t.cpp"), "-o", exe], check=True)
    rows = [[float(x) for x in ln.split()] for ln in subprocess.run([exe], check=True, capture_output=True,
                                                                    text=True).stdout.splitlines()]
    assert len(rows) == 4
    for n, ours, ref, pairs, loose in rows:
        assert loose == 0  # the pair is renormalised
        assert ours <= 2.0 ** -48 and ours <= 1.05 * ref and pairs <= 1.05 * ref, (n, ours, pairs, ref)
