"""Whole-number powers and roots of the equation of state (csrc/whole_power.cuh), compiled
for the host, against exact rational arithmetic: no further off than the 1 ulp (2^-52 of the
value at most) a library pow is allowed, where plain squaring is up to 5.  CPU only; needs a
C++ compiler.  Bounds: half an ulp of the last rounding and 1% for what is carried to first
order; the root's first guess leaves (k^2 - 1) / 12 (3e-7)^3 < 6e-19, 0.6% of an ulp."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OUT = os.path.join(ROOT, "paper_2206_14780_gb300", "_build", "whole_power_probe")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "whole_power.cuh"
int main(int argc, char** argv) {
  const int k = atoi(argv[1]);
  double x;
  while (fread(&x, 8, 1, stdin) == 1) {
    const double r[2] = {sph::whole_pow_m1(x, k), x > 0 ? sph::whole_root(x, k) : 0.0};
    fwrite(r, 8, 2, stdout);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def run():
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    os.makedirs(OUT, exist_ok=True)
    src, exe = os.path.join(OUT, "probe.cpp"), os.path.join(OUT, "probe")
    with open(src, "w") as fh:
        fh.write(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-Wall", "-I",
                    os.path.join(ROOT, "paper_2206_14780_gb300", "csrc"), src, "-o", exe], check=True)

    def go(x, k):
        out = subprocess.run([exe, str(k)], input=np.asarray(x, np.float64).tobytes(), capture_output=True, check=True)
        return np.frombuffer(out.stdout, np.float64).reshape(-1, 2)

    return go


def _ulp(v):
    return Fraction(float(np.spacing(np.abs(v))))


@pytest.mark.parametrize("k", [2, 3, 5, 7, 8, 11, 15, 16])
def test_power_minus_one(run, k):
    rng = np.random.default_rng(k)
    x = np.concatenate([1.0 + rng.uniform(-0.1, 0.1, 300), 1.0 + 1e-6 * rng.normal(size=300),
                        np.exp(rng.uniform(-3, 3, 300)), [1.0, 1.0 + 2.0 ** -24, 1.0 - 2.0 ** -24]])
    for v, (got, _) in zip(x, run(x, k)):
        power = Fraction(float(v)) ** k
        exact = power - 1
        # half an ulp of the result, and of the power's carried part
        assert abs(Fraction(float(got)) - exact) <= Fraction(51, 100) * _ulp(float(exact)) + Fraction(2) ** -98 * power


@pytest.mark.parametrize("k", [2, 3, 5, 7, 8, 11, 15, 16])
def test_root(run, k):
    rng = np.random.default_rng(100 + k)
    x = np.concatenate([1.0 + rng.uniform(-0.3, 0.3, 300), np.exp(rng.uniform(-60, 60, 300))])
    for v, (_, got) in zip(x, run(x, k)):
        y, e = Fraction(float(got)), Fraction(52, 100) * _ulp(float(got))
        assert (y - e) ** k <= Fraction(float(v)) <= (y + e) ** k


def test_infinite_and_vanishing_powers(run):
    got = run([1e300, 1e-300, 0.0, np.inf, np.nan], 7)[:, 0]
    assert got[0] == np.inf and got[1] == -1.0 and got[2] == -1.0 and got[3] == np.inf and np.isnan(got[4])
