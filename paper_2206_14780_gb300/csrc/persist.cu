// The inner BiCGSTAB and the refinement passes around it as one cooperative kernel,
// for particle sets whose tiles are all resident at once.
//
// Below ~100k rows an iteration of the five-kernel loop (solver.cu) costs 37-50 us of
// which the applies' memory traffic is a few: the rest is five launches and three
// grid reductions whose last block runs alone.  Whole passes (rebuild, start, solve to
// 1e-8) at the tile sizes neighbors.cu picks, five kernels / this one, us: 2.2k rows
// 1386 / 921, 6.8k 2043 / 1584, 16k 2597 / 2153, 30k 3567 / 3062, 51k 5125 / 4268, 59k
// 5337 / 4044, 79k 6779 / 6269, 97k 7437 / 6552, 110k 7735 / 7463; Gaussian 3.1k 1419 / 1034,
// 11.5k 2522 / 1880, 35k 4334 / 3449, 77k 8815 / 6858.  Three 8-slice tiles a block reach
// 116.7k rows; a fourth needs unions below ~1,330 rows, which thin layers have (a slope of
// 8 spacings, 133k rows: 12601 / 9855) and boxes, channels and deep slopes of that size do
// not (1,460-1,560: they run the loop, 117k rows 8705, 155k 10378).
// What is left per iteration (2.2k rows: 17 us) is the three
// exchanges at ~3 us each and the latency of two applies' streams.  Here one block of 512 threads per SM
// keeps, for every distinct neighbour of its tiles, r (or r*), p and A p in shared
// memory (40 bytes with its row number), so that blocks exchange A p and A r* only,
// once each per iteration; the vector updates of the union copies are the operations
// of the rows they copy, bit for bit.  An iteration has three grid barriers, one per
// reduction: every block stores its partial sums with the barrier's number beside
// them, waits until it has seen every other block's and adds them up itself (in the
// same order everywhere), so no block waits for another's result to be published and
// the fence for the exchanged vectors runs beside the block's own float64 sum.
// Float64 is scarce (an addition takes a warp 63 cycles), so the scalars are turned
// into float32 once per block, not by every thread.  After a pass the block adds d to
// x, exchanges d, updates the float64 residual and starts the next pass; the host
// sees one launch per solve.
//
// Waits are bounded; a block that gives up sets `fault` and leaves, and the others
// then give up too (SPH_ERR_TIMEOUT).
#include <algorithm>
#include <cmath>

#include "bicgstab_scalars.cuh"
#include "dfloat.cuh"
#include "persist.cuh"
#include "reduce.cuh"
#include "tiles.cuh"

namespace sph {

namespace {

constexpr int kPT = 512;             // threads per block
constexpr int kPW = kPT / 32;
constexpr int kPTilesMax = 16;       // tiles a block may hold
constexpr int kPSliceMax = 64;       // slices a block may hold
constexpr int kPDepth = 3;           // groups of a row's stream in flight per lane
constexpr size_t kPSmem = 216 * 1024;   // dynamic shared memory of a block beside `Shared`
constexpr long long kPWaitCycles = 4000000000ll;   // ~2 s of SM clock

// a block's partial sum: the two halves of a float64, each beside the barrier's number
struct __align__(16) Slot {
  unsigned long long lo, hi;
};

struct PersistArgs {
  TileView op;
  int ts_shift;                      // log2 of the slices per tile
  int tiles_per_block;               // contiguous tiles of a block, at most
  int splits;                        // threads that share a row in the applies
  int ucap, rcap;                    // union places and rows of a block in shared memory
  int64_t n;
  const double* D64;                 // the preconditioner's diagonal
  double* iD64;                      // its reciprocals, made once per launch
  float4 *r, *rh, *p, *Ap, *As, *d;
  double *x64, *r64;
  double tol;                        // rtol ||b||
  double eps_floor;
  double rr0[3];                     // squared norms of r64 at the start
  int maxit, max_pass;
  Slot* slots;                       // [2][6][grid]
  PersistResult* out;
};

struct Shared {
  SolverScalars S;
  double res[6], own[6], rr[3];
  float wsum[kPW][6];
  double wsumd[kPW][6];
  int64_t soff[kPSliceMax];
  int ubase[kPTilesMax + 1];
  int stop, go;
};

// warp_sum_multi (reduce.cuh) for float32
template <int K>
__device__ __forceinline__ float warp_sum_multi_f(const float (&in)[K], int& index) {
  constexpr int P = K <= 4 ? 4 : 8, LP = P == 4 ? 2 : 3;
  const int lane = threadIdx.x & 31;
  float v[P];
#pragma unroll
  for (int i = 0; i < P; ++i) v[i] = i < K ? in[i] : 0.f;
  int idx = 0;
#pragma unroll
  for (int L = 0; L < LP; ++L) {
    const int o = 16 >> L, c = P >> (L + 1);
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < c; ++i) {
      const float send = hi ? v[i] : v[i + c], keep = hi ? v[i + c] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    if (hi) idx += c;
  }
#pragma unroll
  for (int o = 16 >> LP; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  index = idx;
  return v[0];
}

__device__ __forceinline__ Slot load_slot(const Slot* p) {
  Slot s;
  asm volatile("ld.acquire.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(s.lo), "=l"(s.hi) : "l"(p) : "memory");
  return s;
}

// The barrier and the sum over the blocks: `mine` is the block's value k in warp k
// (k < K; lane 0), every global store of the block before the caller's last
// __syncthreads is visible to the other blocks after it, and res[k] holds the sum.
// The last warp's fence and its stores of the slots make the release, the acquiring
// loads of the slots the other side.  false: the wait gave up.
template <int K>
__device__ __forceinline__ bool exchange(const PersistArgs& A, unsigned& epoch, Shared* sh, double mine) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  ++epoch;
  if (wid < K && lane == 0) sh->own[wid] = mine;
  if (wid == kPW - 1) __threadfence();
  __syncthreads();
  Slot* slots = A.slots + (size_t)(epoch & 1) * 6 * gridDim.x;
  const unsigned long long tag = (unsigned long long)epoch << 32;
  if (wid == kPW - 1 && lane < K) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(sh->own[lane]);
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(slots + (size_t)lane * gridDim.x + blockIdx.x),
                 "l"(tag | (bits & 0xffffffffull)), "l"(tag | (bits >> 32))
                 : "memory");
  }
  double v = 0.0;
  if (wid < K) {
    const Slot* row = slots + (size_t)wid * gridDim.x;
    bool ok = true;
    long long t0 = 0;
    for (;;) {   // all of the lane's slots in flight at once, again until every one is there
      bool all = true;
      v = 0.0;
#pragma unroll 5
      for (int b = lane; b < gridDim.x; b += 32) {
        const Slot s = load_slot(row + b);
        all = all && ((s.lo ^ tag) >> 32) == 0 && ((s.hi ^ tag) >> 32) == 0;
        v += __longlong_as_double((long long)((s.lo & 0xffffffffull) | (s.hi << 32)));
      }
      if (all) break;
      if (t0 == 0) t0 = clock64();
      if (clock64() - t0 > kPWaitCycles) {
        ok = false;
        break;
      }
    }
    if (!ok) {
      sh->stop = 1;
      atomicExch(&A.out->fault, 1);
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  if (wid < K && lane == 0) sh->res[wid] = v;
  __syncthreads();
  return sh->stop == 0;
}

// Per-thread float32 sums of K values over the grid.  busy: the warp has rows.
template <int K>
__device__ __forceinline__ bool grid_sum(const PersistArgs& A, unsigned& epoch, Shared* sh, const float (&acc)[K],
                                         bool busy) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int P = K <= 4 ? 4 : 8;
  int idx = lane / (32 / P);
  float t = 0.f;
  if (busy) t = warp_sum_multi_f<K>(acc, idx);
  if ((lane & (32 / P - 1)) == 0 && idx < K) sh->wsum[wid][idx] = t;
  __syncthreads();
  double v = 0.0;
  if (wid < K) {
    if (lane < kPW) v = (double)sh->wsum[lane][wid];
#pragma unroll
    for (int o = kPW / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return exchange<K>(A, epoch, sh, v);
}

// The same for six float64 sums.
__device__ __forceinline__ bool grid_sum_f64(const PersistArgs& A, unsigned& epoch, Shared* sh, const double (&acc)[6],
                                             bool busy) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int idx = lane / 4;
  double t = 0.0;
  if (busy) t = warp_sum_multi<6>(acc, idx);
  if ((lane & 3) == 0 && idx < 6) sh->wsumd[wid][idx] = t;
  __syncthreads();
  double v = 0.0;
  if (wid < 6) {
    if (lane < kPW) v = sh->wsumd[lane][wid];
#pragma unroll
    for (int o = kPW / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return exchange<6>(A, epoch, sh, v);
}

__global__ void __launch_bounds__(kPT, 1) k_persist(PersistArgs A) {
  extern __shared__ __align__(16) char dyn[];
  __shared__ Shared sh;
  const TileView& op = A.op;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int t0 = blockIdx.x * A.tiles_per_block, t1 = min(t0 + A.tiles_per_block, op.ntiles);
  const int tsh = A.ts_shift;
  const int64_t sl0 = (int64_t)t0 << tsh;
  const int nsl = (int)max((int64_t)0, min((int64_t)t1 << tsh, op.nslices) - sl0);
  const int NR = nsl * 32, SP = A.splits;
  const int64_t row0 = sl0 * kSlice;
  const bool rows_here = wid * 32 < NR;              // the warp has rows in the loops over rows
  float4* P = reinterpret_cast<float4*>(dyn);        // p, A p x
  float4* R = P + A.ucap;                            // r or r*, A p y
  float* Z = reinterpret_cast<float*>(R + A.ucap);   // A p z
  int* ID = reinterpret_cast<int*>(Z + A.ucap);      // the union's rows
  unsigned* info = reinterpret_cast<unsigned*>(ID + A.ucap);   // entries | kind << 16
  float* wD = reinterpret_cast<float*>(info + A.rcap);         // 1/D
  float* part = wD + A.rcap;                         // [SP][NR][3], in the residual [SP][NR][6]
  if (tid == 0) {
    int u = 0;
    for (int t = t0; t < t1; ++t) {
      sh.ubase[t - t0] = u;
      u += op.unum[t];
    }
    sh.ubase[t1 - t0] = u;
    sh.stop = 0;
    for (int c = 0; c < 3; ++c) sh.rr[c] = A.rr0[c];
  }
  for (int i = tid; i < nsl; i += kPT) sh.soff[i] = op.off[sl0 + i];
  for (int r = tid; r < NR; r += kPT) {
    info[r] = (unsigned)op.cnt[row0 + r] | ((unsigned)op.kind[row0 + r] << 16);
    wD[r] = op.invD[row0 + r];
  }
  __syncthreads();
  for (int t = t0; t < t1; ++t) {
    const int b = sh.ubase[t - t0], m = sh.ubase[t - t0 + 1] - b;
    const int32_t* __restrict__ ids = op.uni + (int64_t)t * op.ustride;
    for (int i = tid; i < m; i += kPT) ID[b + i] = ids[i];
  }
  const int U = sh.ubase[t1 - t0];
  unsigned epoch = 0;
  SolverScalars* S = &sh.S;

  // y rows of the apply on the union copies in X; finish(row of the block, v_b, sums)
  auto apply = [&](const float4* X, auto own, auto finish) {
    for (int u = wid; u < nsl * SP; u += kPW) {
      const int i = u % nsl, split = u / nsl, r = i * 32 + lane;
      const unsigned in = info[r];
      TileStreamD<kPDepth> ts;
      ts.start_at(op, sl0 + i, sh.soff[i], lane, (int)(in & 0xffffu), split, SP);
      const float kap = (in >> 16) == KIND_FLUID ? 1.f : 0.f;
      const float4 vb = own(r);
      float ax = 0.f, ay = 0.f, az = 0.f;
      ts.sum(X + sh.ubase[i >> tsh], split, SP, kap * vb.x, kap * vb.y, kap * vb.z, ax, ay, az);
      if (SP == 1) {
        finish(r, vb, ax, ay, az);
      } else {
        float* q = part + ((size_t)split * NR + r) * 3;
        q[0] = ax;
        q[1] = ay;
        q[2] = az;
      }
    }
    if (SP > 1) {
      __syncthreads();
      for (int r = tid; r < NR; r += kPT) {
        const float4 vb = own(r);
        float ax = 0.f, ay = 0.f, az = 0.f;
        for (int k = SP - 1; k >= 0; --k) {
          const float* q = part + ((size_t)k * NR + r) * 3;
          ax += q[0];
          ay += q[1];
          az += q[2];
        }
        finish(r, vb, ax, ay, az);
      }
    }
  };
  // r = r0^ = D^-1 r64 of a row, and its squares
  auto start_row = [&](double (&sums)[6], int64_t s, double r0, double r1, double r2) {
    const double sc = A.iD64[s];
    const float4 v = make_float4((float)(r0 * sc), (float)(r1 * sc), (float)(r2 * sc), 0.f);
    __stcg(A.r + s, v);
    __stcg(A.rh + s, v);
    sums[3] += (double)v.x * v.x;
    sums[4] += (double)v.y * v.y;
    sums[5] += (double)v.z * v.z;
  };

  int passes = 0, iters = 0, last_iter = 0, stuck = 0, stalled = 0;
  {
  double sums[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int r = tid; r < NR; r += kPT) {
    const int64_t s = row0 + r;
    A.iD64[s] = 1.0 / A.D64[s];
    start_row(sums, s, A.r64[3 * s], A.r64[3 * s + 1], A.r64[3 * s + 2]);
  }
  if (!grid_sum_f64(A, epoch, &sh, sums, rows_here)) return;
  }
  for (;;) {
    if (tid == 0) {
      const double q = sh.rr[0] + sh.rr[1] + sh.rr[2], rn = sqrt(q);
      sh.go = isfinite(sh.rr[0]) && isfinite(sh.rr[1]) && isfinite(sh.rr[2]) && rn > A.tol && passes < A.max_pass && iters < A.maxit;
      if (sh.go) {
        const double eps = fmax(A.eps_floor, 0.25 * A.tol / rn);
        scal_init(S, sh.res + 3, eps * eps, A.maxit - iters);
      }
    }
    for (int i = tid; i < U; i += kPT) {
      const float4 v = __ldcg(A.r + ID[i]);
      R[i] = v;
      P[i] = v;
      Z[i] = 0.f;
    }
    for (int r = tid; r < NR; r += kPT) {
      __stcg(A.p + row0 + r, __ldcg(A.r + row0 + r));
      __stcg(A.d + row0 + r, make_float4(0.f, 0.f, 0.f, 0.f));
    }
    __syncthreads();
    if (!sh.go) break;
    while (!S->done) {
      // A p, delta
      float a3[3] = {0.f, 0.f, 0.f};
      apply(P, [&](int r) { return __ldcg(A.p + row0 + r); },
            [&](int r, float4 vb, float ax, float ay, float az) {
              const float4 h = __ldcg(A.rh + row0 + r);
              const float4 o = tile_finish((uint8_t)(info[r] >> 16), vb, ax, ay, az, wD[r]);
              __stcg(A.Ap + row0 + r, o);
              a3[0] = fmaf(h.x, o.x, a3[0]);
              a3[1] = fmaf(h.y, o.y, a3[1]);
              a3[2] = fmaf(h.z, o.z, a3[2]);
            });
      if (!grid_sum<3>(A, epoch, &sh, a3, SP == 1 || rows_here)) return;
      if (wid == 0) scal_after_delta_w(S, sh.res);
      __syncthreads();
      const float al0 = S->alpha_f[0], al1 = S->alpha_f[1], al2 = S->alpha_f[2];
      // r* = r - alpha A p, A r*, omega
#pragma unroll 2
      for (int i = tid; i < U; i += kPT) {
        const float4 q = __ldcg(A.Ap + ID[i]), v = R[i];
        R[i] = make_float4(fmaf(-al0, q.x, v.x), fmaf(-al1, q.y, v.y), fmaf(-al2, q.z, v.z), q.y);
        P[i].w = q.x;
        Z[i] = q.z;
      }
      __syncthreads();
      float a6[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      auto rstar = [&](int r) {
        const float4 v = __ldcg(A.r + row0 + r), q = __ldcg(A.Ap + row0 + r);
        return make_float4(fmaf(-al0, q.x, v.x), fmaf(-al1, q.y, v.y), fmaf(-al2, q.z, v.z), 0.f);
      };
      apply(R, rstar, [&](int r, float4 vb, float ax, float ay, float az) {
        const float4 o = tile_finish((uint8_t)(info[r] >> 16), vb, ax, ay, az, wD[r]);
        __stcg(A.As + row0 + r, o);
        a6[0] = fmaf(vb.x, o.x, a6[0]);
        a6[1] = fmaf(vb.y, o.y, a6[1]);
        a6[2] = fmaf(vb.z, o.z, a6[2]);
        a6[3] = fmaf(o.x, o.x, a6[3]);
        a6[4] = fmaf(o.y, o.y, a6[4]);
        a6[5] = fmaf(o.z, o.z, a6[5]);
      });
      if (!grid_sum<6>(A, epoch, &sh, a6, SP == 1 || rows_here)) return;
      if (wid == 0) scal_after_omega_w(S, sh.res);
      __syncthreads();
      const float w0 = S->omega_f[0], w1 = S->omega_f[1], w2 = S->omega_f[2];
      // r = r* - omega A r*, d, gamma' and r.r
#pragma unroll
      for (int k = 0; k < 6; ++k) a6[k] = 0.f;
      for (int r = tid; r < NR; r += kPT) {
        const int64_t s = row0 + r;
        const float4 rs = rstar(r), as = __ldcg(A.As + s), p = __ldcg(A.p + s), h = __ldcg(A.rh + s);
        float4 d = __ldcg(A.d + s);
        const float4 v = make_float4(fmaf(-w0, as.x, rs.x), fmaf(-w1, as.y, rs.y), fmaf(-w2, as.z, rs.z), 0.f);
        d.x = fmaf(w0, rs.x, fmaf(al0, p.x, d.x));
        d.y = fmaf(w1, rs.y, fmaf(al1, p.y, d.y));
        d.z = fmaf(w2, rs.z, fmaf(al2, p.z, d.z));
        __stcg(A.r + s, v);
        __stcg(A.d + s, d);
        a6[0] = fmaf(h.x, v.x, a6[0]);
        a6[1] = fmaf(h.y, v.y, a6[1]);
        a6[2] = fmaf(h.z, v.z, a6[2]);
        a6[3] = fmaf(v.x, v.x, a6[3]);
        a6[4] = fmaf(v.y, v.y, a6[4]);
        a6[5] = fmaf(v.z, v.z, a6[5]);
      }
#pragma unroll 2
      for (int i = tid; i < U; i += kPT) {
        const float4 q = __ldcg(A.As + ID[i]);
        float4 v = R[i];
        v.x = fmaf(-w0, q.x, v.x);
        v.y = fmaf(-w1, q.y, v.y);
        v.z = fmaf(-w2, q.z, v.z);
        R[i] = v;
      }
      if (!grid_sum<6>(A, epoch, &sh, a6, rows_here)) return;
      if (wid == 0) scal_after_update_w(S, sh.res, sh.res + 3);
      __syncthreads();
      if (S->done) break;
      // p = r + beta p - alpha' A p  (a zero coefficient skips its vector)
      const float c0 = S->alphap_f[0], c1 = S->alphap_f[1], c2 = S->alphap_f[2];
      const float b0 = S->beta_f[0], b1 = S->beta_f[1], b2 = S->beta_f[2];
      const bool useP = (b0 != 0.f) || (b1 != 0.f) || (b2 != 0.f);
      const bool useA = (c0 != 0.f) || (c1 != 0.f) || (c2 != 0.f);
      auto next_p = [&](float4 v, float4 q, float4 a) {
        if (useP) {
          v.x = fmaf(b0, q.x, v.x);
          v.y = fmaf(b1, q.y, v.y);
          v.z = fmaf(b2, q.z, v.z);
        }
        if (useA) {
          v.x = fmaf(-c0, a.x, v.x);
          v.y = fmaf(-c1, a.y, v.y);
          v.z = fmaf(-c2, a.z, v.z);
        }
        v.w = 0.f;
        return v;
      };
      for (int r = tid; r < NR; r += kPT) {
        const int64_t s = row0 + r;
        __stcg(A.p + s, next_p(__ldcg(A.r + s), __ldcg(A.p + s), __ldcg(A.Ap + s)));
      }
      for (int i = tid; i < U; i += kPT) {
        const float4 v = R[i], q = P[i];
        P[i] = next_p(v, q, make_float4(q.w, v.w, Z[i], 0.f));
      }
      __syncthreads();
    }
    ++passes;
    last_iter = S->iter;
    iters += last_iter;
    for (int c = 0; c < 3; ++c) stalled |= S->stalled_any[c] ? 1 << c : 0;
    // x += d
    for (int r = tid; r < NR; r += kPT) {
      const int64_t s = row0 + r;
      const float4 d = __ldcg(A.d + s);
      A.x64[3 * s] += (double)d.x;
      A.x64[3 * s + 1] += (double)d.y;
      A.x64[3 * s + 2] += (double)d.z;
    }
    if (last_iter == 0) {   // nothing progressed: a further pass would repeat it
      stuck = 1;
      break;
    }
    // r64 -= A d (all of d is known since the last reduction), and the next pass's r
    for (int i = tid; i < U; i += kPT) P[i] = __ldcg(A.d + ID[i]);
    __syncthreads();
    double sums[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    auto finish64 = [&](int r, const double (&v)[3]) {
      const int64_t s = row0 + r;
      const unsigned kd = info[r] >> 16;
      const double sg = kd == KIND_FLUID ? 1.0 : (kd == KIND_SHEPARD ? -1.0 : 0.0);
      const float4 db = __ldcg(A.d + s);
      double r0 = 0.0, r1 = 0.0, r2 = 0.0;
      if (s < A.n) {
        r0 = A.r64[3 * s] - ((double)db.x + sg * v[0]);
        r1 = A.r64[3 * s + 1] - ((double)db.y + sg * v[1]);
        r2 = A.r64[3 * s + 2] - ((double)db.z + sg * v[2]);
      }
      A.r64[3 * s] = r0;
      A.r64[3 * s + 1] = r1;
      A.r64[3 * s + 2] = r2;
      sums[0] += r0 * r0;
      sums[1] += r1 * r1;
      sums[2] += r2 * r2;
      start_row(sums, s, r0, r1, r2);
    };
    for (int u = wid; u < nsl * SP; u += kPW) {
      const int i = u % nsl, split = u / nsl, r = i * 32 + lane;
      const unsigned in = info[r];
      const float kap = (in >> 16) == KIND_FLUID ? 1.f : 0.f;
      const float4 db = __ldcg(A.d + row0 + r);
      DFAcc x0, x1, x2;
      const float4* X = P + sh.ubase[i >> tsh];
      if ((in & 0xffffu) != 0)
        tile_residual_row<false>(op, X, X, sl0 + i, lane, (int)(in & 0xffffu), split, SP,
                                 make_float4(kap * db.x, kap * db.y, kap * db.z, 0.f),
                                 make_float4(0.f, 0.f, 0.f, 0.f), x0, x1, x2);
      if (SP == 1) {
        finish64(r, {x0.value(), x1.value(), x2.value()});
      } else {
        const SplitSum v[3] = {SplitSum(x0), SplitSum(x1), SplitSum(x2)};
        float* q = part + ((size_t)split * NR + r) * 6;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          q[2 * k] = v[k].hi;
          q[2 * k + 1] = v[k].lo;
        }
      }
    }
    if (SP > 1) {
      __syncthreads();
      for (int r = tid; r < NR; r += kPT) {
        const float* q = part + (size_t)r * 6;
        SplitSum v[3] = {SplitSum(q[0], q[1]), SplitSum(q[2], q[3]), SplitSum(q[4], q[5])};
        for (int w = 1; w < SP; ++w) {
          q += (size_t)NR * 6;
#pragma unroll
          for (int k = 0; k < 3; ++k) v[k].add(SplitSum(q[2 * k], q[2 * k + 1]));
        }
        finish64(r, {v[0].value(), v[1].value(), v[2].value()});
      }
    }
    // (this barrier also holds the next pass's reset of d back until every block has
    // read it)
    if (!grid_sum_f64(A, epoch, &sh, sums, SP == 1 || rows_here)) return;
    if (tid < 3) sh.rr[tid] = sh.res[tid];
    __syncthreads();
  }
  if (blockIdx.x == 0 && tid == 0) {
    PersistResult* o = A.out;
    o->passes = passes;
    o->iters = iters;
    o->last_iter = last_iter;
    o->stuck = stuck;
    o->stalled = stalled;
    for (int c = 0; c < 3; ++c) {
      o->state[c] = passes > 0 ? S->state[c] : 0;
      o->rr[c] = sh.rr[c];
    }
    __threadfence();
    o->done = 1;
  }
}

}  // namespace

PersistPlan persist_plan(const sph_neighbors* H) {
  PersistPlan p;
  const int sms = H->num_sms > 0 ? H->num_sms : 1;
  if (!H->op_tile_valid || H->ntiles < 1) return p;
  p.tiles_per_block = (int)((H->ntiles + sms - 1) / sms);
  // One-slice tiles: fewer blocks with more tiles each, since an exchange costs the more
  // the more blocks take part.  Whole passes with 1 / 2 / 3 / 4 tiles a block, us: rows of
  // ~80, solves of 2.7k rows 1133 / 1078 / 990 / 1026, 3.2k from host buffers 816 / 749 /
  // 760 / 735, a step of 2.6k 842 / 841 / 812 / 838; rows of ~250, 2.9k rows 1079 / 1103 /
  // 1168 / 1204, 4.7k 1590 / 1430 / 1473 / 1530.
  if (H->tile_ts == 1) {
    const int least = H->maxnb <= 160 ? 3 : (H->ntiles <= 2 * (int64_t)sms / 3 ? 1 : 2);
    p.tiles_per_block = (p.tiles_per_block + least - 1) / least * least;
  }
  const int nsl = p.tiles_per_block * H->tile_ts;
  if (p.tiles_per_block > kPTilesMax || nsl > kPSliceMax) return p;
  p.grid = (int)((H->ntiles + p.tiles_per_block - 1) / p.tiles_per_block);
  p.ucap = (p.tiles_per_block * std::max(H->tile_umax, 1) + 3) & ~3;
  p.rcap = nsl * 32;
  // threads per row: the warps' rounds times the groups of a row each walks (plus the
  // start of a stream, ~3 groups' worth), over the lists' longest row
  const int groups = (H->max_cnt + 3) / 4;
  int best = 0;
  for (int sp = 1; sp <= 8; sp *= 2) {
    const size_t part = sp > 1 ? (size_t)sp * p.rcap * 6 * sizeof(float) : 0;
    const size_t smem = (size_t)p.ucap * 40 + (size_t)p.rcap * 8 + part;
    if (smem > kPSmem) break;
    const int cost = (nsl * sp + kPW - 1) / kPW * ((groups + sp - 1) / sp + 3);
    if (best == 0 || cost < best) {
      best = cost;
      p.splits = sp;
      p.smem = smem;
    }
  }
  p.ok = best > 0;
  return p;
}

sph_status persist_solve(sph_neighbors* H, const PersistPlan& plan, const TileView& view, const double* D64, double tol,
                         double eps_floor, const double rr0[3], int maxit, int max_pass, PersistResult* out,
                         cudaStream_t st) {
  static_assert(sizeof(PersistResult) <= 256 && sizeof(Slot) == 16, "device blocks");
  const size_t nslots = (size_t)2 * 6 * plan.grid;
  SPH_TRY(H->persist_buf.alloc(nslots * 2 + 32 + H->n_pad));   // the slots, the result, the reciprocals
  if (!H->host_persist) SPH_TRY_CUDA(cudaMallocHost(&H->host_persist, 256));
  SPH_TRY_CUDA(cudaMemsetAsync(H->persist_buf.p, 0, (nslots * 2 + 32) * sizeof(double), st));
  PersistArgs A{};
  A.op = view;
  A.ts_shift = H->tile_ts == 8 ? 3 : (H->tile_ts == 4 ? 2 : (H->tile_ts == 2 ? 1 : 0));
  A.tiles_per_block = plan.tiles_per_block;
  A.splits = plan.splits;
  A.ucap = plan.ucap;
  A.rcap = plan.rcap;
  A.n = H->n;
  A.D64 = D64;
  A.r = H->v_r.p;
  A.rh = H->v_rh.p;
  A.p = H->v_p.p;
  A.Ap = H->v_Ap.p;
  A.As = H->v_As.p;
  A.d = H->v_d.p;
  A.x64 = H->x64.p;
  A.r64 = H->r64.p;
  A.tol = tol;
  A.eps_floor = eps_floor;
  for (int c = 0; c < 3; ++c) A.rr0[c] = rr0[c];
  A.maxit = maxit;
  A.max_pass = max_pass;
  A.slots = reinterpret_cast<Slot*>(H->persist_buf.p);
  A.out = reinterpret_cast<PersistResult*>(H->persist_buf.p + nslots * 2);
  A.iD64 = H->persist_buf.p + nslots * 2 + 32;
  SPH_TRY_CUDA(cudaFuncSetAttribute((const void*)k_persist, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPSmem));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)plan.grid);
  cfg.blockDim = dim3(kPT);
  cfg.dynamicSmemBytes = plan.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  note_launch();
  SPH_TRY_CUDA(cudaLaunchKernelEx(&cfg, k_persist, A));
  SPH_TRY_CUDA(cudaMemcpyAsync(H->host_persist, A.out, sizeof(PersistResult), cudaMemcpyDeviceToHost, st));
  SPH_TRY_CUDA(cudaStreamSynchronize(st));
  *out = *static_cast<const PersistResult*>(H->host_persist);
  if (out->fault || !out->done) {
    set_error("sph_visc_solve: a grid barrier of the cooperative solve kernel gave up");
    return SPH_ERR_TIMEOUT;
  }
  return SPH_OK;
}

}  // namespace sph
