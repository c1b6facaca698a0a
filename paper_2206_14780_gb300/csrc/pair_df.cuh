// Pair quantities of A(dt) in double-float arithmetic (dfloat.cuh), shared by the
// two forms the coefficients are stored in (operator.cu, tiles.cu).
#pragma once

#include "dfloat.cuh"
#include "sph_internal.cuh"

namespace sph {

struct OpGeom {
  double L[3];
  double invL[3];
  int periodic[3];
  double h;
  double inv_h;
};

// Geometry of the double-float set-up: periods, 1/h and 1/h^2 as (hi, lo)
struct OpGeomDF {
  dfl L[3];
  float invL[3];
  int periodic[3];
  dfl inv_h, inv_h2;
};

// |r_a - r_b|^2 in double-float: the coordinate differences of the float32
// positions exactly (TwoSum), the minimum image by a whole period, the squared
// norm with exact products
__device__ __forceinline__ dfl pair_r2_df(float4 pa, float4 pb, const OpGeomDF& g) {
  dfl d[3] = {df_exact_sum(pa.x, -pb.x), df_exact_sum(pa.y, -pb.y), df_exact_sum(pa.z, -pb.z)};
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    if (g.periodic[ax]) {
      const float k = rintf(d[ax].hi * g.invL[ax]);
      if (k != 0.f) d[ax] = df_add(d[ax], dfl{-k * g.L[ax].hi, -k * g.L[ax].lo});
    }
  }
  return df_add(df_add(df_mul(d[0], d[0]), df_mul(d[1], d[1])), df_mul(d[2], d[2]));
}
// q = r / h, one Newton step on the root
__device__ __forceinline__ dfl pair_q_df(dfl r2, const OpGeomDF& g) { return df_mul(df_sqrt(r2), g.inv_h); }

// Wendland psi_{3,1} without its constant factor (it cancels in W / S):
// (1 - q/2)^4 (2q + 1), zero for q >= 2
__device__ __forceinline__ dfl wendland_w_df(dfl q) {
  dfl t = df_add(dfl{1.f, 0.f}, dfl{-0.5f * q.hi, -0.5f * q.lo});
  if (t.hi <= 0.f) return dfl{0.f, 0.f};
  const dfl t2 = df_mul(t, t);
  return df_mul(df_mul(t2, t2), df_add(dfl{1.f, 0.f}, dfl{2.f * q.hi, 2.f * q.lo}));
}

// e^{-k / kExpSteps} as (hi, lo), for arguments up to the truncated Gaussian's 9:
// Taylor's series of the step, then powers, in the compiler's float64 arithmetic with
// the powers' rounding errors carried along (TwoProd by Veltkamp's splitting)
constexpr int kExpSteps = 128;
constexpr int kExpEntries = 9 * kExpSteps + 8;
struct alignas(8) ExpEntry {
  float hi, lo;
};
struct ExpTable {
  ExpEntry v[kExpEntries];
  static constexpr double high_half(double a) {
    const double t = 134217729.0 * a;
    return t - (t - a);
  }
  constexpr ExpTable() : v{} {
    // e^{-1/128} = sh + sl: the terms from the smallest up, the leading ones exactly
    double tail = 0.0;
    for (int k = 12; k >= 3; --k) {
      double term = 1.0;
      for (int m = 1; m <= k; ++m) term *= -1.0 / (kExpSteps * m);
      tail += term;
    }
    const double lead = 1.0 - 1.0 / kExpSteps + 0.5 / (kExpSteps * (double)kExpSteps);   // exact
    const double sh = lead + tail, sl = tail - (sh - lead);
    const double s1 = high_half(sh), s2 = sh - s1;
    double h = 1.0, l = 0.0;
    for (int k = 0; k < kExpEntries; ++k) {
      v[k].hi = (float)h;
      v[k].lo = (float)((h - (double)v[k].hi) + l);
      const double h1 = high_half(h), h2 = h - h1, p = h * sh;
      const double e = (((h1 * s1 - p) + h1 * s2 + h2 * s1) + h2 * s2) + (h * sl + l * sh);
      h = p + e;
      l = e - (h - p);
    }
  }
};
static __device__ const ExpTable kExpTable{};

// truncated Gaussian (Sec. 5.2, radius 3h): e^{-x}, x = q^2 in double-float, formed from
// r^2 without a root.  x = k / 128 + r: the table's value times 1 - r + r^2 / 2 - r^3 / 6
// + ..., the cubic and later terms (below 2^-26) in float32.  Relative error of the
// function below 2^-45.5; with that of x (a few 2^-46 times x) the factor of a pair is
// 2^-46.4 off in the root mean square, 2^-43.1 at most, against 2^-44.8 and 2^-41.8 with
// the root, its square and a float64 exp (4 million random pairs).  That exp costs a warp about 20 float64
// instructions of ~63 cycles and set the pace of the Gaussian's set-up: 5.6k rows of ~250
// neighbours 123 us with it, 45 us without.
__device__ __forceinline__ dfl gauss_e_df(dfl x) {
  const float kf = fminf(rintf(x.hi * (float)kExpSteps), (float)(kExpEntries - 1));
  const ExpEntry t = kExpTable.v[(int)kf];
  const dfl r = df_exact_sum(fmaf(kf, -1.f / kExpSteps, x.hi), x.lo);
  const float p = r.hi * r.hi, pe = fmaf(r.hi, r.hi, -p);
  // r^3 / 6 - r^4 / 24 + r^5 / 120 with r = hi + lo to first order
  const float c = p * fmaf(r.hi, fmaf(r.hi, fmaf(r.hi, 1.f / 120.f, -1.f / 24.f), 1.f / 6.f), 0.5f * r.lo);
  const dfl u = df_quick(1.f, -r.hi), w = df_quick(u.hi, 0.5f * p);
  const float lo = (u.lo + w.lo) + (fmaf(r.hi, r.lo, 0.5f * pe) - r.lo - c);
  return df_mul(dfl{t.hi, t.lo}, df_quick(w.hi, lo));
}

// the fluid coefficient's kernel factor: (2 - q)^3 (Wendland) or e^{-q^2} (Gaussian),
// each without the constant of |f| (it is in R_b)
__device__ __forceinline__ dfl fluid_kernel_df(dfl r2, const OpGeomDF& g, int gauss) {
  if (gauss) return gauss_e_df(df_mul(r2, g.inv_h2));
  dfl tq = df_add(dfl{2.f, 0.f}, df_neg(pair_q_df(r2, g)));
  if (tq.hi <= 0.f) tq = dfl{0.f, 0.f};
  return df_mul(df_mul(tq, tq), tq);
}

// the Shepard weight w(q) without its constant: Wendland, or e^{-q^2} - e^{-9}
__device__ __forceinline__ dfl shepard_w_df(dfl r2, const OpGeomDF& g, int gauss, dfl gauss_tail) {
  if (gauss) return df_add(gauss_e_df(df_mul(r2, g.inv_h2)), df_neg(gauss_tail));
  return wendland_w_df(pair_q_df(r2, g));
}

}  // namespace sph
