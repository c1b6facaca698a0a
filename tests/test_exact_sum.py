"""The error-free float32 sums (csrc/exact_sum.cuh), compiled for the host: against exact
rational arithmetic, and never further off than a float64 sum of the same terms (what these
sums replace).  CPU only; needs a C++ compiler.

Bound: n terms x of a three-part sum are off by less than 4 n^2 2^-72 sum |x| (each of the
three levels leaves at most n u of what it sums, u = 2^-24), and the result is rounded to
float64 twice (2^-52 of its size)."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OUT = os.path.join(ROOT, "paper_2206_14780_gb300", "_build", "exact_sum_probe")

# rows of a residual: n terms a (k - x), a and x given as (a hi, a lo, x), one accumulator, or
# `splits` of them taking groups of four terms in turn and put together as the solve does
ROWS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "exact_sum.cuh"
using namespace sph;
int main(int argc, char** argv) {
  const int n = atoi(argv[1]), splits = atoi(argv[2]);
  std::vector<float> row(1 + 3 * n);
  while (fread(row.data(), 4, row.size(), stdin) == row.size()) {
    std::vector<DFAcc> part(splits);
    for (int i = 0; i < n; ++i)
      part[i / 4 % splits].add(row[1 + 3 * i], row[2 + 3 * i], row[0], row[3 + 3 * i], 0.f, 0.f);
    double v;
    if (splits == 1) {
      v = part[0].value();
    } else {
      SplitSum s(part[0]);
      for (int k = 1; k < splits; ++k) s.add(SplitSum(part[k]));
      v = s.value();
    }
    fwrite(&v, 8, 1, stdout);
  }
  return 0;
}
"""

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "exact_sum.cuh"
using namespace sph;
int main(int argc, char** argv) {
  const int kind = atoi(argv[1]), splits = atoi(argv[2]);
  std::vector<float> v;
  float x;
  while (fread(&x, 4, 1, stdin) == 1) v.push_back(x);
  const int n = (int)v.size() / kind;
  std::vector<Sum3> part(splits);
  for (int i = 0; i < n; ++i) {
    Sum3& s = part[i % splits];
    const float* t = &v[(size_t)i * kind];
    if (kind == 1) s.add(t[0]);
    else if (kind == 2) s.add_product(t[0], t[1]);
    else s.add_product(t[0], t[1], t[2]);
  }
  for (int k = 1; k < splits; ++k) part[0].add(part[k]);
  const double r = part[0].value();
  fwrite(&r, 8, 1, stdout);
  return 0;
}
"""


def _compile(name, program):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    os.makedirs(OUT, exist_ok=True)
    src, exe = os.path.join(OUT, name + ".cpp"), os.path.join(OUT, name)
    with open(src, "w") as fh:
        fh.write(program)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-Wall", "-I",
                    os.path.join(ROOT, "paper_2206_14780_gb300", "csrc"), src, "-o", exe], check=True)
    return exe


@pytest.fixture(scope="module")
def run():
    exe = _compile("probe", PROGRAM)

    def go(terms, splits=1):
        terms = np.ascontiguousarray(terms, np.float32)
        kind = 1 if terms.ndim == 1 else terms.shape[1]
        out = subprocess.run([exe, str(kind), str(splits)], input=terms.tobytes(), capture_output=True, check=True)
        return float(np.frombuffer(out.stdout, np.float64)[0])

    return go


def _exact(terms):
    terms = np.asarray(terms, np.float32).reshape(len(terms), -1)
    rows = [np.prod([Fraction(float(x)) for x in row]) for row in terms]
    return sum(rows), sum(abs(r) for r in rows)


def _cancelling(rng, n, factors):
    """Terms whose sum is far below their size: pairs that cancel up to a part in 10^9."""
    a = rng.normal(size=(n, factors)).astype(np.float32)
    b = a.copy()
    b[:, 0] = -b[:, 0]
    small = (1e-9 * rng.normal(size=(n // 4, factors))).astype(np.float32)
    return rng.permutation(np.concatenate([a, b, small]))


@pytest.mark.parametrize("factors", [1, 2, 3])
@pytest.mark.parametrize("splits", [1, 2, 8])
@pytest.mark.parametrize("seed", range(4))
def test_sum_is_no_further_off_than_a_float64_sum(run, factors, splits, seed):
    rng = np.random.default_rng(seed)
    for terms in (_cancelling(rng, 40, factors), rng.normal(size=(80, factors)).astype(np.float32),
                  np.exp(rng.uniform(-30, 30, size=(80, 1)) / factors).astype(np.float32) * np.ones((1, factors), np.float32)):
        exact, size = _exact(terms)
        got = run(terms[:, 0] if factors == 1 else terms, splits)
        n = len(terms) * factors
        off = abs(Fraction(got) - exact)
        assert off <= 4 * n * n * Fraction(2) ** -72 * size + Fraction(2) ** -52 * abs(exact)
        plain = 0.0
        for row in terms.astype(np.float64):
            plain += np.prod(row)
        assert off <= max(abs(Fraction(float(plain)) - exact), 2 * Fraction(2) ** -53 * abs(exact))


@pytest.mark.parametrize("n", [80, 250])
def test_split_rows_are_no_further_off_than_one_accumulator(n):
    """Rows of a residual in every number of splits against float64 longer arithmetic: the
    root mean square error over 2,000 rows, relative to the terms' magnitudes, stays within
    5% (its own scatter is 1/sqrt(4000) = 1.6%) of one float64-combined accumulator's."""
    exe = _compile("rows", ROWS)
    rng = np.random.default_rng(n)
    count = 2000
    a = 5.0 * rng.random((count, n)) ** 3
    hi = a.astype(np.float32)
    lo = (a - hi).astype(np.float32)
    k = rng.normal(size=(count, 1)).astype(np.float32)
    x = (k + 0.1 * rng.normal(size=(count, n))).astype(np.float32)
    rows = np.concatenate([k, np.stack([hi, lo, x], axis=2).reshape(count, 3 * n)], axis=1).astype(np.float32)
    coef = hi.astype(np.longdouble) + lo
    terms = coef * (k.astype(np.longdouble) - x)
    exact, size = terms.sum(axis=1), np.abs(terms).sum(axis=1)
    rms = {}
    for splits in (1, 2, 4, 8):
        out = subprocess.run([exe, str(n), str(splits)], input=rows.tobytes(), capture_output=True, check=True).stdout
        got = np.frombuffer(out, np.float64)
        assert got.size == count
        rms[splits] = float(np.sqrt(np.mean(((got - exact) / size) ** 2)))
    assert rms[1] < 2.0 ** -48
    for splits in (2, 4, 8):
        assert rms[splits] <= 1.05 * rms[1], rms


def test_non_finite_terms_give_what_a_float64_sum_gives(run):
    for terms, want in (([1.0, np.inf, 2.0], np.inf), ([1.0, -np.inf], -np.inf), ([np.inf, -np.inf], np.nan),
                        ([np.nan, 1.0], np.nan), ([], 0.0)):
        for splits in (1, 2):
            got = run(np.array(terms, np.float32), splits)
            assert got == want or (np.isnan(got) and np.isnan(want))
