"""Coefficients (2 - delta_k0) J_k(alpha) of a piece of an interval, from the library's own functions compiled for the host,
against the Bessel functions' power series in 60-digit decimals.

One rounding of the values (at most 2) is 2.2e-16; the table's recurrence and the sum of the Taylor series add a few:
1e-15 in the 2-norm over all k."""
import decimal
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1801_04382_gb300", "csrc")
PROG = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "kt_common.h"
int main(int argc, char **argv) {
  const double r = atof(argv[1]), dt = atof(argv[2]);
  const int K = atoi(argv[3]), segs = kt_piece_segments(r * dt);
  std::vector<double> t((size_t)segs * (KT_PIECE_DEG + 1) * K);
  kt_piece_table(segs, K, t.data());
  for (int a = 4; a < argc; ++a)
    for (int k = 0; k < K; ++k) printf("%.17g\n", kt_piece_coef(t.data(), segs, K, k, r, atof(argv[a])));
}
"""


def bessel(alpha, n):
    """2 J_k(alpha) (J_0 for k = 0), k < n, alpha a Decimal"""
    out = []
    h = alpha / 2
    for k in range(n):
        term = decimal.Decimal(1)
        for i in range(1, k + 1):
            term = term * h / i
        tot, m = term, 0
        while abs(term) > decimal.Decimal(10) ** -40 or m < 2 * h:
            m += 1
            term = -term * h * h / (m * (m + k))
            tot += term
        out.append(float(tot * (2 if k else 1)))
    return np.array(out)


@pytest.mark.parametrize("r,dt,K", [(3e-7, 0.1, 4), (7.3, 0.05, 15), (106.3, 0.05, 36), (157.9, 0.025, 19), (61.7, 1.0, 96)])
def test_piece_coefficients(tmp_path, r, dt, K):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    decimal.getcontext().prec = 80
    (tmp_path / "t.cpp").write_text(PROG)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")], check=True)
    rng = random.Random(3)
    times = [0.0, dt, 0.5 * dt, dt * 2.0 ** -40, 1.0 / r if r * dt > 1 else 0.3 * dt] + [rng.uniform(0.0, dt) for _ in range(12)]
    out = subprocess.run([str(tmp_path / "t"), repr(r), repr(dt), str(K), *[repr(s) for s in times]], capture_output=True,
                         text=True, check=True).stdout
    got = np.array([float(x) for x in out.split()]).reshape(len(times), K)
    for s, g in zip(times, got):
        ref = bessel(decimal.Decimal(r) * decimal.Decimal(s), K)
        assert np.linalg.norm(g - ref) <= 1e-15, (s, np.linalg.norm(g - ref))
