// Error-free float32 sums.  Plain C++ under a host compiler too, so that the
// arithmetic is tested without a GPU.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define SPH_HD __host__ __device__ __forceinline__
#else
#define SPH_HD inline
#endif

namespace sph {

// Knuth's TwoSum: s + e == a + b exactly (no branch, any magnitudes)
SPH_HD void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// A running sum in three float32 parts, s + e + f: the rounding errors of s are added
// up in e, those of e in f (the K-fold sum of Ogita, Rump and Oishi, 2005, for K = 3).
// n terms x_i and products are off by a few n^2 2^-72 of sum |x_i|, where a float64
// sum is off by n 2^-53; it is ~13 float32 operations a term, where a float64 addition
// takes a warp 63 cycles.
struct Sum3 {
  float s = 0.f, e = 0.f, f = 0.f;
  SPH_HD void add_low(float x) {   // a term already small against s
    float t, r;
    two_sum(e, x, t, r);
    e = t;
    f += r;
  }
  SPH_HD void add(float x) {
    float t, r;
    two_sum(s, x, t, r);
    s = t;
    add_low(r);
  }
  // a b, exactly: the product and its rounding error
  SPH_HD void add_product(float a, float b) {
    const float p = a * b;
    add(p);
    add_low(fmaf(a, b, -p));
  }
  // a b c, exactly: (p + q) c with p + q = a b
  SPH_HD void add_product(float a, float b, float c) {
    const float p = a * b, q = fmaf(a, b, -p), t = p * c, u = q * c;
    add(t);
    add_low(fmaf(p, c, -t));
    add_low(u);
    f += fmaf(q, c, -u);
  }
  SPH_HD void add(const Sum3& o) {
    add(o.s);
    add_low(o.e);
    f += o.f;
  }
  // an infinite or undefined s keeps its value, as a float64 sum would
  SPH_HD double value() const { return std::isfinite(s) ? (double)s + ((double)e + (double)f) : (double)s; }
};

}  // namespace sph
