// A(dt) in the tile form (tiles.cuh): its coefficients, y = A v, the dummy-wall
// closure and the float64-accurate residuals.  Every kernel runs one block of 256
// threads per tile of TS slices; with TS < 8 the S = 8 / TS threads of a row take
// its groups of four entries in turn.
#include <atomic>
#include <cmath>

#include "dfloat.cuh"
#include "pair_df.cuh"
#include "reduce.cuh"
#include "tiles.cuh"

namespace sph {

TileView tile_view(const sph_neighbors* H) {
  return TileView{H->t_idx.p, H->t_istride, H->t_hi.p,   H->t_lo.p,   H->t_off.p,      H->op_cnt.p,       H->op_kind.p,
                  H->invD.p,  H->t_uni.p,   H->t_unum.p, H->t_ustride, (int32_t)H->ntiles, H->nslices};
}

size_t tile_smem(const sph_neighbors* H, int bytes_per_row) {
  return (size_t)(H->tile_umax > 0 ? H->tile_umax : 1) * bytes_per_row;
}

int tile_grid(const sph_neighbors* H, const void* kernel, size_t smem) {
  // the limit of a block once, for the largest union any kernel holds (32 bytes a row)
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (kTileUnion + 1) * 32);
  int occ = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 256, smem);
  const int64_t all = (int64_t)(H->num_sms > 0 ? H->num_sms : 1) * (occ > 0 ? occ : 1);
  const int64_t rounds = (H->ntiles + all - 1) / all;
  return rounds > 0 ? (int)((H->ntiles + rounds - 1) / rounds) : 1;
}

namespace {

// per particle: V = m / rho and 1 / mu as double-float pairs (V hi, V lo, 1/mu hi,
// 1/mu lo)
__global__ void k_tile_aux(const float4* __restrict__ pos, const float* __restrict__ rho, const float* __restrict__ mu,
                           int64_t n_pad, float4* __restrict__ aux) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n_pad; s += (int64_t)gridDim.x * blockDim.x) {
    const dfl v = df_quotient(dfl{pos[s].w, 0.f}, rho[s]), w = df_quotient(dfl{1.f, 0.f}, mu[s]);
    aux[s] = make_float4(v.hi, v.lo, w.hi, w.lo);
  }
}

struct FillArgs {
  const float4* pos;
  const float* rho;
  const float* mu;
  const uint8_t* type;
  const float4* aux;
  const int32_t* nfl;
  int64_t n;
  OpGeomDF g;
  dfl kf;              // 2 dt times the constant of |f| over h^5, divided by 2^kf_exp
  int kf_exp;
  int dummy, arithmetic, gauss;
  dfl gauss_tail;      // e^{-9}
  float* hi;
  float* lo;
  int32_t* op_cnt;
  uint8_t* op_kind;
  float* invD;
  double* D64;
  unsigned long long* nnz;
};

// The coefficients of A(dt), formulas and arithmetic as k_op_fill (operator.cu), in
// the tiles' entry order: the union's positions, volumes and 1/mu are read into
// shared memory once per tile (32 bytes a row), a lane computes four entries per
// step (independent chains of ~170 float32 operations) and stores them with one
// 16-byte store each for hi and lo.
template <int TS>
__global__ void __launch_bounds__(256) k_tile_fill(TileView op, FillArgs A) {
  constexpr int S = 8 / TS, R = 32 * TS;
  extern __shared__ __align__(16) float4 dyn[];
  __shared__ double part[S > 1 ? S * R : 1];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int split = wid / TS, row = (wid % TS) * 32 + lane;
  for (int64_t tile = blockIdx.x; tile < op.ntiles; tile += gridDim.x) {
    const int nu = op.unum[tile];
    const int32_t* __restrict__ ids = op.uni + tile * op.ustride;
    float4* P = dyn;         // x, y, z, 1 on fluid rows
    float4* B = dyn + nu;    // V hi, V lo, 1/mu hi (or mu), 1/mu lo
    for (int i = tid; i < nu; i += 256) {
      const int t = ids[i];
      float4 p = A.pos[t], b = A.aux[t];
      p.w = A.type[t] == SPH_FLUID ? 1.f : 0.f;
      if (A.arithmetic) b.z = A.mu[t];
      P[i] = p;
      B[i] = b;
    }
    const int64_t sl = tile * TS + wid % TS, s = sl * kSlice + lane;
    const bool have = sl < op.nslices;
    uint8_t kd = KIND_IDENTITY;
    int c = 0;
    if (have && s < A.n) {
      const int f = A.nfl[s];
      if (A.type[s] == SPH_FLUID) {
        kd = KIND_FLUID;
        c = f;
      } else if (A.dummy && f > 0) {
        kd = KIND_SHEPARD;
        c = f;
      }
    }
    __syncthreads();
    const uint2* __restrict__ pi = reinterpret_cast<const uint2*>(op.idx + sl * op.istride) + lane;
    const int64_t o0 = have ? op.off[sl] : 0;
    float4* __restrict__ ph = reinterpret_cast<float4*>(A.hi + o0) + lane;
    float4* __restrict__ pl = reinterpret_cast<float4*>(A.lo + o0) + lane;
    const int ng = (c + 3) >> 2;
    const float4 pb = c > 0 ? A.pos[s] : make_float4(0.f, 0.f, 0.f, 0.f);
    dfl sum{0.f, 0.f};
    if (kd == KIND_FLUID) {
      const float mu_b = A.mu[s];
      const float4 ab = A.aux[s];
      const dfl imu_b{ab.z, ab.w};
      const dfl Rb = c > 0 ? df_quotient(A.kf, A.rho[s], A.kf_exp) : dfl{0.f, 0.f};
      for (int g = split; g < ng; g += S) {
        uint32_t o[4];
        tile_unpack(pi[g * 32], o);
        float h4[4], l4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 pa = tile_at(P, o[k]), at = tile_at(B, o[k]);
          const dfl tq3 = fluid_kernel_df(pair_r2_df(pa, pb, A.g), A.g, A.gauss);
          dfl mub{mu_b, 0.f};
          if (pa.w != 0.f) {
            if (A.arithmetic) {
              const dfl m2 = df_exact_sum(at.z, mu_b);
              mub = dfl{0.5f * m2.hi, 0.5f * m2.lo};
            } else {
              const dfl h = df_rcp(df_add(dfl{at.z, at.w}, imu_b));
              mub = dfl{2.f * h.hi, 2.f * h.lo};
            }
          }
          dfl a = df_mul(df_mul(Rb, dfl{at.x, at.y}), df_mul(mub, tq3));
          if (g * 4 + k >= c) a = dfl{0.f, 0.f};
          h4[k] = a.hi;
          l4[k] = a.lo;
          sum = df_add(sum, a);
        }
        ph[g * 32] = make_float4(h4[0], h4[1], h4[2], h4[3]);
        pl[g * 32] = make_float4(l4[0], l4[1], l4[2], l4[3]);
      }
    } else if (kd == KIND_SHEPARD) {
      for (int g = split; g < ng; g += S) {
        uint32_t o[4];
        tile_unpack(pi[g * 32], o);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (g * 4 + k < c)
            sum = df_add(sum, shepard_w_df(pair_r2_df(tile_at(P, o[k]), pb, A.g), A.g, A.gauss, A.gauss_tail));
      }
    }
    double tot = df_to_double(sum);
    if (S > 1) {   // every thread of a row takes the row's sum, in one order
      part[split * R + row] = tot;
      __syncthreads();
      tot = 0.0;
#pragma unroll
      for (int k = 0; k < S; ++k) tot += part[k * R + row];
    }
    if (kd == KIND_SHEPARD) {
      // S rounds to zero only if every fluid neighbour sits at the support's edge to
      // within rounding: zero coefficients then make the row an identity row
      const dfl Sd = df_from_double(tot);
      const dfl invS = Sd.hi > 0.f ? df_rcp(Sd) : dfl{0.f, 0.f};
      for (int g = split; g < ng; g += S) {
        uint32_t o[4];
        tile_unpack(pi[g * 32], o);
        float h4[4], l4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          dfl a = df_mul(shepard_w_df(pair_r2_df(tile_at(P, o[k]), pb, A.g), A.g, A.gauss, A.gauss_tail),
                         invS);
          if (g * 4 + k >= c) a = dfl{0.f, 0.f};
          h4[k] = a.hi;
          l4[k] = a.lo;
        }
        ph[g * 32] = make_float4(h4[0], h4[1], h4[2], h4[3]);
        pl[g * 32] = make_float4(l4[0], l4[1], l4[2], l4[3]);
      }
    }
    if (split == 0 && have) {
      A.op_cnt[s] = c;
      A.op_kind[s] = kd;
      if (kd == KIND_FLUID) {
        const double D = 1.0 + tot;
        A.D64[s] = D;
        A.invD[s] = df_rcp(df_from_double(D)).hi;
      } else {
        A.D64[s] = 1.0;
        A.invD[s] = 1.f;
      }
      int many = c;
      for (int k = 16; k > 0; k >>= 1) many += __shfl_xor_sync(0xffffffffu, many, k);
      if (lane == 0 && many > 0) atomicAdd(A.nnz, (unsigned long long)many);
    }
    __syncthreads();
  }
}

// y = A v.  CALLER: v and y in the caller's order (the union and the rows are read
// and written through perm, so no sorted copy of v or y is made).
template <int TS, bool CALLER>
__global__ void __launch_bounds__(256, kTileBlocks) k_tile_apply(TileView op, const float4* __restrict__ v, float4* __restrict__ y,
                                                    const int32_t* __restrict__ perm, int64_t n) {
  constexpr int S = 8 / TS, R = 32 * TS;
  extern __shared__ __align__(16) float4 u[];
  __shared__ float part[S > 1 ? (S - 1) * R * 3 : 1];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int split = wid / TS, row = (wid % TS) * 32 + lane;
  for (int64_t tile = blockIdx.x; tile < op.ntiles; tile += gridDim.x) {
    if (CALLER) {
      const int32_t* __restrict__ ids = op.uni + tile * op.ustride;
      const int nu = op.unum[tile];
      for (int i = tid; i < nu; i += 256) cp_async16(u + i, v + perm[ids[i]]);
    } else {
      tile_load_union(op, tile, v, u);
    }
    const int64_t sl = tile * TS + wid % TS, s = sl * kSlice + lane;
    const bool have = sl < op.nslices && (!CALLER || s < n);
    int c = 0;
    uint8_t kd = KIND_IDENTITY;
    float4 vb = make_float4(0.f, 0.f, 0.f, 0.f);
    int64_t at = s;
    if (have) {
      c = op.cnt[s];
      kd = op.kind[s];
      if (CALLER) at = perm[s];
      vb = v[at];
    }
    const float kap = kd == KIND_FLUID ? 1.f : 0.f;
    TileStream ts;
    ts.start(op, sl, lane, c, split, S);
    cp_async_wait_all();
    __syncthreads();
    float ax = 0.f, ay = 0.f, az = 0.f;
    ts.sum(u, split, S, kap * vb.x, kap * vb.y, kap * vb.z, ax, ay, az);
    tile_combine<TS>(part, split, row, ax, ay, az);
    if (have && split == 0) y[at] = tile_finish(kd, vb, ax, ay, az, 1.f);
    __syncthreads();
  }
}

// Dummy-wall closure (Eq. dummyvel) in the caller's x0: on a Shepard row x0 = b -
// sum of (W / S) x0 over its fluid neighbours, on the other wall rows x0 = b.  Only
// the tiles that hold a wall row read their union (13% of the box's rows are walls).
template <int TS>
__global__ void __launch_bounds__(256) k_tile_wall_close(TileView op, const uint8_t* __restrict__ type,
                                                         const int32_t* __restrict__ perm, int64_t n,
                                                         const double* __restrict__ b, double* x0) {
  constexpr int S = 8 / TS, R = 32 * TS;
  extern __shared__ __align__(16) float4 u[];
  __shared__ float part[S > 1 ? (S - 1) * R * 3 : 1];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int split = wid / TS, row = (wid % TS) * 32 + lane;
  for (int64_t tile = blockIdx.x; tile < op.ntiles; tile += gridDim.x) {
    const int64_t sl = tile * TS + wid % TS, s = sl * kSlice + lane;
    const bool wall = sl < op.nslices && s < n && type[s] != SPH_FLUID;
    const bool shep = wall && op.kind[s] == KIND_SHEPARD;
    if (__syncthreads_or(wall) == 0) continue;
    if (__syncthreads_or(shep) != 0) {
      const int32_t* __restrict__ ids = op.uni + tile * op.ustride;
      const int nu = op.unum[tile];
      for (int i = tid; i < nu; i += 256) {
        const int t = ids[i];
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (type[t] == SPH_FLUID) {
          const int64_t j = perm[t];
          q = make_float4((float)x0[3 * j], (float)x0[3 * j + 1], (float)x0[3 * j + 2], 0.f);
        }
        u[i] = q;
      }
    }
    __syncthreads();
    float ax = 0.f, ay = 0.f, az = 0.f;
    TileStream ts;
    ts.start(op, sl, lane, shep ? op.cnt[s] : 0, split, S);
    ts.sum(u, split, S, 0.f, 0.f, 0.f, ax, ay, az);
    tile_combine<TS>(part, split, row, ax, ay, az);
    if (wall && split == 0) {
      const int64_t i = perm[s];
      // A x~ on the row, x~ = x0 with its wall rows zero: 0 - (sum of a (0 - x0))
      x0[3 * i] = b[3 * i] - (double)(0.f - ax);
      x0[3 * i + 1] = b[3 * i + 1] - (double)(0.f - ay);
      x0[3 * i + 2] = b[3 * i + 2] - (double)(0.f - az);
    }
    __syncthreads();
  }
}

// X2: r = b - A x on sorted [n_pad][3] arrays, x2 = x in float32 halves (hi, lo
// interleaved); else r -= A d.  Partial sums of r_c^2 go through the grid reduction
// into res_out.  The gathers come from shared memory (32 or 16 bytes a union row),
// so the double-float additions set the pace.
template <int TS, bool X2>
__global__ void __launch_bounds__(256) k_tile_residual(TileView op, const float4* __restrict__ x2,
                                                       const double* __restrict__ x, const double* __restrict__ b,
                                                       double* __restrict__ r, int64_t n, double* __restrict__ partials,
                                                       unsigned int* counter, double* __restrict__ res_out) {
  constexpr int S = 8 / TS, R = 32 * TS;
  extern __shared__ __align__(16) float4 dyn[];
  __shared__ double part[S > 1 ? (S - 1) * R * 3 : 1];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int split = wid / TS, row = (wid % TS) * 32 + lane;
  double acc2[3] = {0.0, 0.0, 0.0};
  for (int64_t tile = blockIdx.x; tile < op.ntiles; tile += gridDim.x) {
    const int nu = op.unum[tile];
    const int32_t* __restrict__ ids = op.uni + tile * op.ustride;
    float4* uh = dyn;
    float4* ul = dyn + nu;
    for (int i = tid; i < nu; i += 256) {
      const int64_t t = ids[i];
      if (X2) {
        cp_async16(uh + i, x2 + 2 * t);
        cp_async16(ul + i, x2 + 2 * t + 1);
      } else {
        cp_async16(uh + i, x2 + t);
      }
    }
    const int64_t sl = tile * TS + wid % TS, s = sl * kSlice + lane;
    const bool have = sl < op.nslices;
    int c = 0;
    uint8_t kd = KIND_IDENTITY;
    float4 bh = make_float4(0.f, 0.f, 0.f, 0.f), bl = bh;
    if (have) {
      c = op.cnt[s];
      kd = op.kind[s];
      bh = X2 ? x2[2 * s] : x2[s];
      if (X2) bl = x2[2 * s + 1];
    }
    const float kap = kd == KIND_FLUID ? 1.f : 0.f;
    cp_async_wait_all();
    __syncthreads();
    DFAcc a0, a1, a2;
    if (c > 0)
      tile_residual_row<X2>(op, uh, ul, sl, lane, c, split, S,
                            make_float4(kap * bh.x, kap * bh.y, kap * bh.z, 0.f),
                            make_float4(kap * bl.x, kap * bl.y, kap * bl.z, 0.f), a0, a1, a2);
    double v0 = a0.value(), v1 = a1.value(), v2 = a2.value();
    if (S > 1) {
      if (split > 0) {
        double* q = part + ((split - 1) * R + row) * 3;
        q[0] = v0;
        q[1] = v1;
        q[2] = v2;
      }
      __syncthreads();
      if (split == 0)
        for (int k = 0; k < S - 1; ++k) {
          const double* q = part + (k * R + row) * 3;
          v0 += q[0];
          v1 += q[1];
          v2 += q[2];
        }
    }
    if (have && split == 0) {
      const double sg = kd == KIND_FLUID ? 1.0 : (kd == KIND_SHEPARD ? -1.0 : 0.0);
      double r0 = 0.0, r1 = 0.0, r2 = 0.0;
      if (s < n) {
        if (X2) {
          r0 = b[3 * s] - (x[3 * s] + sg * v0);
          r1 = b[3 * s + 1] - (x[3 * s + 1] + sg * v1);
          r2 = b[3 * s + 2] - (x[3 * s + 2] + sg * v2);
        } else {
          r0 = r[3 * s] - ((double)bh.x + sg * v0);
          r1 = r[3 * s + 1] - ((double)bh.y + sg * v1);
          r2 = r[3 * s + 2] - ((double)bh.z + sg * v2);
        }
      }
      r[3 * s] = r0;
      r[3 * s + 1] = r1;
      r[3 * s + 2] = r2;
      acc2[0] += r0 * r0;
      acc2[1] += r1 * r1;
      acc2[2] += r2 * r2;
    }
    __syncthreads();
  }
  if (partials == nullptr) return;
  block_partials_f64<3>(acc2, partials + (size_t)blockIdx.x * kMaxDots);
  if (arrive_last(counter)) {
    __shared__ double res[3];
    final_sum<3>(partials, counter, res);
    if (threadIdx.x < 3) res_out[threadIdx.x] = res[threadIdx.x];
  }
}

}  // namespace

sph_status tile_fill(sph_neighbors* H, const sph_visc_params* P, cudaStream_t st) {
  SPH_TRY(H->t_hi.alloc(H->t_entries > 0 ? H->t_entries : 1));
  SPH_TRY(H->t_lo.alloc(H->t_entries > 0 ? H->t_entries : 1));
  SPH_TRY(H->aux_df.alloc(H->n_pad));
  SPH_TRY(H->t_nnz.alloc(1));
  SPH_TRY_CUDA(cudaMemsetAsync(H->t_nnz.p, 0, sizeof(unsigned long long), st));
  auto split = [](double x) {
    const float hi = (float)x;
    return dfl{hi, (float)(x - (double)hi)};
  };
  FillArgs A{};
  for (int ax = 0; ax < 3; ++ax) {
    A.g.L[ax] = split(H->grid.L[ax]);
    A.g.invL[ax] = (float)(1.0 / H->grid.L[ax]);
    A.g.periodic[ax] = H->grid.periodic[ax];
  }
  const double ih = 1.0 / (double)H->h;
  A.g.inv_h = split(ih);
  A.g.inv_h2 = split(ih * ih);
  A.gauss = H->kernel == SPH_KERNEL_GAUSSIAN ? 1 : 0;
  A.kf = split(std::frexp(2.0 * P->dt * (A.gauss ? 2.0 / gauss_norm() : 105.0 / (128.0 * M_PI)) * (ih * ih * ih * ih * ih),
                          &A.kf_exp));
  A.pos = H->pos_s.p;
  A.rho = H->rho_s.p;
  A.mu = H->mu_s.p;
  A.type = H->type_s.p;
  A.aux = H->aux_df.p;
  A.nfl = H->t_nfl.p;
  A.n = H->n;
  A.dummy = P->boundary == SPH_BC_DUMMY ? 1 : 0;
  A.arithmetic = P->mean == SPH_MEAN_ARITHMETIC ? 1 : 0;
  A.gauss_tail = split(std::exp(-kGaussK * kGaussK));
  A.hi = H->t_hi.p;
  A.lo = H->t_lo.p;
  A.op_cnt = H->op_cnt.p;
  A.op_kind = H->op_kind.p;
  A.invD = H->invD.p;
  A.D64 = H->D64.p;
  A.nnz = H->t_nnz.p;
  SPH_LAUNCH(k_tile_aux, grid_for(H, H->n_pad), kBlock, 0, st)(H->pos_s.p, H->rho_s.p, H->mu_s.p, H->n_pad, H->aux_df.p);
  auto kern = SPH_TILE_PICK(H, k_tile_fill);
  const size_t smem = tile_smem(H, 32);
  SPH_LAUNCH(kern, tile_grid(H, (const void*)kern, smem), 256, smem, st)(tile_view(H), A);
  SPH_TRY_CUDA(cudaGetLastError());
  H->op_nnz = -1;
  return SPH_OK;
}

void tile_apply(const sph_neighbors* H, const float4* v, float4* y, bool caller_order, cudaStream_t st) {
  auto kern = caller_order ? SPH_TILE_PICK(H, k_tile_apply, SPH_COMMA true) : SPH_TILE_PICK(H, k_tile_apply, SPH_COMMA false);
  const size_t smem = tile_smem(H, 16);
  SPH_LAUNCH(kern, tile_grid(H, (const void*)kern, smem), 256, smem, st)(tile_view(H), v, y, H->perm.p, H->n);
}

void tile_wall_close(const sph_neighbors* H, double* x0, const double* b, cudaStream_t st) {
  auto kern = SPH_TILE_PICK(H, k_tile_wall_close);
  const size_t smem = tile_smem(H, 16);
  SPH_LAUNCH(kern, tile_grid(H, (const void*)kern, smem), 256, smem, st)(tile_view(H), H->type_s.p, H->perm.p, H->n, b, x0);
}

void tile_residual(const sph_neighbors* H, const float4* x2, const double* x, const double* b, double* r,
                   double* partials, unsigned int* counter, double* res_out, cudaStream_t st) {
  auto kern = SPH_TILE_PICK(H, k_tile_residual, SPH_COMMA true);
  const size_t smem = tile_smem(H, 32);
  const int g = tile_grid(H, (const void*)kern, smem);   // partials hold red_cap blocks
  SPH_LAUNCH(kern, g < H->red_cap ? g : H->red_cap, 256, smem, st)(tile_view(H), x2, x, b, r, H->n, partials, counter, res_out);
}

void tile_residual_update(const sph_neighbors* H, const float4* d, double* r, double* partials,
                          unsigned int* counter, double* res_out, cudaStream_t st) {
  auto kern = SPH_TILE_PICK(H, k_tile_residual, SPH_COMMA false);
  const size_t smem = tile_smem(H, 16);
  const int g = tile_grid(H, (const void*)kern, smem);   // partials hold red_cap blocks
  SPH_LAUNCH(kern, g < H->red_cap ? g : H->red_cap, 256, smem, st)(tile_view(H), d, nullptr, nullptr, r, H->n, partials, counter,
                                                       res_out);
}

}  // namespace sph
