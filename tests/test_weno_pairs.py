"""The WENO5 face value in pairs of FP32 numbers (csrc/vof_df.cuh, compiled for
the host) against the same weights in long double, on smooth and random stencils
and with temperature jumps at every place.

Bound: the weights and the products take chains of at most ~40 pair operations
of 2^-46 each, and what they scale are the candidates by their own weights, so
the correction is within 2^-40 of sum_k (w_k / W) |terms of r_k| / 6, and the sum
with the donor value rounds once (2^-53 of each operand).  A jump counts by the
weight of the candidate that crosses it: 1e-12 or less."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2001_03477_gb300", "csrc")

PROGRAM = r"""
#include "vof_df.cuh"
#include <cstdio>
#include <cstdlib>
#include <random>
using namespace vofgb;
typedef long double L;
static L ab(L x) { return x < 0 ? -x : x; }
int main(int argc, char** argv) {
  const int fam = atoi(argv[1]);
  std::mt19937_64 r(11 + fam);
  std::uniform_real_distribution<double> u(-1, 1), p(0, 1);
  double worst = 0;
  for (int i = 0; i < 100000; ++i) {
    double v[5];
    const double s = u(r), q = u(r);
    for (int j = 0; j < 5; ++j) {
      if (fam < 4) v[j] = j <= fam ? 0.0 : 1.0 + 1e-3 * u(r);            // cold donor side
      else if (fam < 8) v[j] = j <= fam - 4 ? 1.0 + 1e-3 * u(r) : 0.0;   // hot donor side
      else if (fam == 8) v[j] = 373.15 + 5 * s * j + q * j * j + 0.01 * u(r);
      else if (fam == 9) v[j] = u(r);
      else if (fam == 10) v[j] = u(r) * exp2(-30 * p(r));
      else if (fam == 11) v[j] = (r() & 1) ? 0.0 : 1.0 + 0.01 * u(r);
      else v[j] = j <= (int)(r() % 4) ? 373.15 : 383.0 + u(r);
    }
    const double D[4] = {v[1] - v[0], v[2] - v[1], v[3] - v[2], v[4] - v[3]};
    const double f = weno5_add6(v[2], weno5_corr6_df(D[0], D[1], D[2], D[3]));
    const L D0 = D[0], D1 = D[1], D2 = D[2], D3 = D[3], e = 1e-6L;
    const L d0 = D1 - D0, d1 = D2 - D1, d2 = D3 - D2;
    const L b0 = 13.0L / 12 * d0 * d0 + 0.25L * (3 * D1 - D0) * (3 * D1 - D0),
            b1 = 13.0L / 12 * d1 * d1 + 0.25L * (D1 + D2) * (D1 + D2),
            b2 = 13.0L / 12 * d2 * d2 + 0.25L * (D3 - 3 * D2) * (D3 - 3 * D2);
    const L w0 = 1 / ((e + b0) * (e + b0)), w1 = 6 / ((e + b1) * (e + b1)), w2 = 3 / ((e + b2) * (e + b2)), W = w0 + w1 + w2;
    const L corr = (w0 * (5 * D1 - 2 * D0) + w1 * (D1 + 2 * D2) + w2 * (4 * D2 - D3)) / W / 6;
    const L size = (w0 * (5 * ab(D1) + 2 * ab(D0)) + w1 * (ab(D1) + 2 * ab(D2)) + w2 * (4 * ab(D2) + ab(D3))) / W / 6;
    const L bound = exp2l(-40) * size + exp2l(-53) * (ab(v[2]) + ab(corr)) * 2;
    const L err = ab((L)f - ((L)v[2] + corr));
    if (bound > 0 && (double)(err / bound) > worst) worst = (double)(err / bound);
    if (bound == 0 && err != 0) worst = 1e9;
  }
  printf("%.6g\n", worst);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("weno")
    (d / "w.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "w"), str(d / "w.cpp"), "-lm"], check=True)
    return str(d / "w")


@pytest.mark.parametrize("family", range(13))
def test_face_value_keeps_its_accuracy_at_jumps(program, family):
    out = subprocess.run([program, str(family)], check=True, capture_output=True, text=True).stdout
    assert float(out) <= 1.0
