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

// Geometry of the double-float set-up: periods as (hi, lo), 1/h as (hi, lo)
struct OpGeomDF {
  dfl L[3];
  float invL[3];
  int periodic[3];
  dfl inv_h;
};

// |r_a - r_b| in double-float: the coordinate differences of the float32
// positions exactly (TwoSum), the minimum image by a whole period, the squared
// norm with exact products, one Newton step on the root
__device__ __forceinline__ dfl pair_r_df(float4 pa, float4 pb, const OpGeomDF& g) {
  dfl d[3] = {df_exact_sum(pa.x, -pb.x), df_exact_sum(pa.y, -pb.y), df_exact_sum(pa.z, -pb.z)};
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    if (g.periodic[ax]) {
      const float k = rintf(d[ax].hi * g.invL[ax]);
      if (k != 0.f) d[ax] = df_add(d[ax], dfl{-k * g.L[ax].hi, -k * g.L[ax].lo});
    }
  }
  const dfl r2 = df_add(df_add(df_mul(d[0], d[0]), df_mul(d[1], d[1])), df_mul(d[2], d[2]));
  return df_sqrt(r2);
}

// Wendland psi_{3,1} without its constant factor (it cancels in W / S):
// (1 - q/2)^4 (2q + 1), zero for q >= 2
__device__ __forceinline__ dfl wendland_w_df(dfl q) {
  dfl t = df_add(dfl{1.f, 0.f}, dfl{-0.5f * q.hi, -0.5f * q.lo});
  if (t.hi <= 0.f) return dfl{0.f, 0.f};
  const dfl t2 = df_mul(t, t);
  return df_mul(df_mul(t2, t2), df_add(dfl{1.f, 0.f}, dfl{2.f * q.hi, 2.f * q.lo}));
}

// truncated Gaussian (Sec. 5.2, radius 3h): e^{-q^2} from the double-float q,
// the exponential in float64 once per pair (the set-up runs once per A(dt))
__device__ __forceinline__ dfl gauss_e_df(dfl q) { return df_from_double(exp(-df_to_double(df_mul(q, q)))); }

// the fluid coefficient's kernel factor: (2 - q)^3 (Wendland) or e^{-q^2} (Gaussian),
// each without the constant of |f| (it is in R_b)
__device__ __forceinline__ dfl fluid_kernel_df(dfl q, int gauss) {
  if (gauss) return gauss_e_df(q);
  dfl tq = df_add(dfl{2.f, 0.f}, df_neg(q));
  if (tq.hi <= 0.f) tq = dfl{0.f, 0.f};
  return df_mul(df_mul(tq, tq), tq);
}

// the Shepard weight w(q) without its constant: Wendland, or e^{-q^2} - e^{-9}
__device__ __forceinline__ dfl shepard_w_df(dfl q, int gauss, double gauss_tail) {
  if (gauss) return df_from_double(exp(-df_to_double(df_mul(q, q))) - gauss_tail);
  return wendland_w_df(q);
}

}  // namespace sph
