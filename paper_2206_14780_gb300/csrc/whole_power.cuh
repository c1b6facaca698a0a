// Powers and roots with whole exponents in float64.  Plain C++ under a host compiler too
// (with -ffp-contract=off), so that they are tested without a GPU.
#pragma once

#include <cmath>

#include "exact_sum.cuh"

namespace sph {

// x^k as h + l for k >= 1: powers by squaring, the rounding error of every product
// (Dekker's, through fma) carried along to first order; h + l is off by a few 2^-100
struct TwoDouble {
  double h, l;
};
SPH_HD TwoDouble two_mul(TwoDouble a, TwoDouble b) {
  const double p = mul_rn(a.h, b.h);
  return TwoDouble{p, fma(a.h, b.l, fma(a.l, b.h, fma(a.h, b.h, -p)))};
}
SPH_HD TwoDouble whole_pow(double x, int k) {
  TwoDouble b{x, 0.0}, r{1.0, 0.0};
  bool first = true;
  for (;;) {
    if (k & 1) {
      r = first ? b : two_mul(r, b);
      first = false;
    }
    k >>= 1;
    if (k == 0) return r;
    b = two_mul(b, b);
  }
}
// x^k - 1 (an infinite power as it is)
SPH_HD double whole_pow_m1(double x, int k) {
  const TwoDouble p = whole_pow(x, k);
  if (!std::isfinite(p.h)) return p.h - 1.0;
  const double s = p.h - 1.0, bb = s - p.h;   // TwoSum of p.h and -1
  return s + (((p.h - (s - bb)) + (-1.0 - bb)) + p.l);
}
// v^(1/k) for 1e-30 < v < 1e30: one Halley step from the float32 root y, error
// (k^2 - 1) / 12 of the cube of its ~3e-7, with v - y^k from the exact power
SPH_HD double whole_root(double v, int k) {
  const double y = (double)powf((float)v, 1.f / (float)k);
  const TwoDouble p = whole_pow(y, k);
  return y + y * (2.0 * ((v - p.h) - p.l)) / ((double)(k + 1) * p.h + (double)(k - 1) * v);
}

}  // namespace sph
