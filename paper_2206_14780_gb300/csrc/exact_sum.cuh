// Error-free float32 transformations (Knuth's TwoSum; Dekker's TwoProd through fma) and the
// sums made of them.  Plain C++ under a host compiler too, so that the
// arithmetic is tested without a GPU.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define SPH_HD __host__ __device__ __forceinline__
#else
#define SPH_HD inline
#endif

namespace sph {

// one rounded operation, never merged with another into a multiply-add (a host build of
// this file needs -ffp-contract=off)
#ifdef __CUDA_ARCH__
SPH_HD float add_rn(float a, float b) { return __fadd_rn(a, b); }
SPH_HD float mul_rn(float a, float b) { return __fmul_rn(a, b); }
SPH_HD double mul_rn(double a, double b) { return __dmul_rn(a, b); }
#else
SPH_HD float add_rn(float a, float b) { return a + b; }
SPH_HD float mul_rn(float a, float b) { return a * b; }
SPH_HD double mul_rn(double a, double b) { return a * b; }
#endif

// Knuth's TwoSum: s + e == a + b exactly (no branch, any magnitudes)
SPH_HD void two_sum(float a, float b, float& s, float& e) {
  s = add_rn(a, b);
  const float bb = add_rn(s, -a);
  e = add_rn(add_rn(a, -add_rn(s, -bb)), add_rn(b, -bb));
}

// sum_a a_ba (kap x_b - x_a) for one component with float32 error-free
// transformations: the difference of the hi parts exactly (TwoSum), its product
// with a_hi exactly (Dekker's TwoProd via fma), the running sum exactly
// (TwoSum), and the terms of order 2^-24 (a_hi * diff error, a_lo * diff,
// a_hi * lo-part difference) in plain float32.  Error ~2^-47 of sum |terms|.
struct DFAcc {
  float sh = 0.f, sl = 0.f, c = 0.f;
  SPH_HD void add(float ahi, float alo, float kxbh, float xah, float kxbl, float xal) {
    float d, de;
    two_sum(kxbh, -xah, d, de);
    const float p = mul_rn(ahi, d);
    const float pe = fmaf(ahi, d, -p);
    float t, te;
    two_sum(sh, p, t, te);
    sh = t;
    sl += te;
    c += pe + fmaf(ahi, de, fmaf(alo, d, ahi * (kxbl - xal)));
  }
  SPH_HD double value() const { return (double)sh + ((double)sl + (double)c); }
};

// A row's DFAcc sums over its splits put together in a float32 pair.  The error of the
// combination is below what the shorter sums save: in the root mean square, relative to
// sum |terms|, 2^-49.0 for one DFAcc over 80 terms, 2^-49.3 / 49.5 / 49.4 for 2 / 4 / 8 of
// them combined so (250 terms: 2^-48.6 and 2^-49.1 / 49.5 / 49.7).  A single DFAcc is not put through it
// (2^-48.9): its value() is in float64.
struct SplitSum {
  float hi, lo;
  SPH_HD explicit SplitSum(const DFAcc& a) : hi(a.sh), lo(a.sl + a.c) {}
  SPH_HD SplitSum(float h, float l) : hi(h), lo(l) {}
  SPH_HD void add(const SplitSum& o) {   // the high parts exactly
    float t, e;
    two_sum(hi, o.hi, t, e);
    hi = t;
    lo += o.lo + e;
  }
  SPH_HD double value() const { return (double)hi + (double)lo; }
};

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
    const float p = mul_rn(a, b);
    add(p);
    add_low(fmaf(a, b, -p));
  }
  // a b c, exactly: (p + q) c with p + q = a b
  SPH_HD void add_product(float a, float b, float c) {
    const float p = mul_rn(a, b), q = fmaf(a, b, -p), t = mul_rn(p, c), u = mul_rn(q, c);
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
