// Warm-start network training on the 5th-generation tensor cores (tcgen05): the
// mean-squared-error loss and its gradient with respect to all 9,603 parameters.
//
// Two CTAs of 8 warps per SM walk 128-row tiles (persistent over the tiles), so
// one CTA's epilogues overlap the other's MMAs.  Each row is one particle; warps w
// and w + 4 share the tensor-memory lanes 32 (w % 4) .. 32 (w % 4) + 31 and split
// every 64-column layer into two halves.  Every product of a tile is one tcgen05.mma
// chain issued by one thread:
//
//   forward      Z_l  = A_{l-1} W_l^T               K-major tiles, as in inference
//   data grad    DA   = Delta_{l+1} W_{l+1}         B = the W_{l+1} tile read MN-major
//   weight grad  dW_l += Delta_l^T A_{l-1}          both operands MN-major: the
//                                                   row-by-row tiles read with the
//                                                   tile's 128 rows as the K index
//
// What bounds it: the tensor pipe needs ~1,300 cycles of a tile; the instructions of
// the epilogues and the chain of seven hand-overs between them and the MMAs set the
// time.  Hence:
//   * epilogues read tensor memory as 16 x 256-bit fragments (4 rows x 8 columns per
//     thread, not 1 x 32): a bias column is 12 two-wide additions in the thread and
//     7 shuffles instead of 31, biases are 4 loads instead of 32, and the bf16 tiles
//     are written by stmatrix, one 128-byte core matrix a step;
//   * the arithmetic between the transcendentals is two-wide (f32x2), SiLU'(Z_3) is
//     kept in registers from the forward epilogue;
//   * a thread waits for the MMAs its next loads need and no others: the weight
//     gradients run under the epilogue that follows (their own barrier where that
//     epilogue overwrites their operand), and the last one of a tile is issued with
//     the next tile's first product.  That tile's features are copied (cp.async) into
//     the buffer of this tile's output deltas meanwhile; the two swap roles per tile.
// 262k rows: 49.5 -> 27.0 million warp instructions, 103 -> 74 us against eight hand-overs
// at which every thread waited for every MMA, with one row per thread.
//
// Tensor memory (256 columns per CTA): Z (64) holds the forward's pre-activations in
// turn and, in the backward pass, Z_2 and Z_1 (recomputed by the same MMAs, so SiLU'
// sees the forward's float32 values); DA (64) the output Y and then
// the data gradients; the weight gradients accumulate over all of the CTA's tiles
// and are written once, as the CTA's partial gradient, at the end.  dW_3 and dW_2
// share one 128-row accumulator: the hidden-delta tile keeps two 64-column halves
// per 8-row group, and Delta_3 is written to the first half with the second zeroed,
// Delta_2 to the second with the first zeroed, so the M = 128 MMA over both halves
// adds Delta_3^T A_2 to rows 0..63 and Delta_2^T A_1 to rows 64..127.  dW_1 and
// dW_4^T have 16 columns each; their rows 64..127 read bytes beyond the operand
// (padded tile memory) and are never read back.  Bias gradients are column sums of
// the float32 deltas (one column per lane, kept over the tiles).
//
// Rounding points follow the float64 reference: inputs, weights, hidden activations
// and backpropagated deltas enter products as bf16; accumulation, biases, SiLU' and
// the bias sums are float32.  Each partial gradient is deterministic (fixed tile
// order per CTA), and the partials are summed in block order by the caller.
//
// Waits on the MMA mbarriers are bounded; a thread whose wait gave up sets *err and
// walks on without waiting, so that the CTA frees its tensor memory and returns.
#include <cuda_bf16.h>

#include <cstdint>

#include "f32x2.cuh"
#include "sph_internal.cuh"
#include "tcgen05.cuh"

namespace sph {

struct MlpPack;
const void* mlp_pack_ptr(const sph_mlp* M);
void mlp_pack_layout(size_t* off_w1, size_t* off_w2, size_t* off_w3, size_t* off_w4, size_t* off_b);

namespace {

constexpr int kNP = 9603;
constexpr int OFF_W1 = 0, OFF_B1 = 1024, OFF_W2 = 1088, OFF_B2 = 5184, OFF_W3 = 5248, OFF_B3 = 9344,
              OFF_W4 = 9408, OFF_B4 = 9600;
constexpr int kRows = 128;
constexpr int kThreads = 256;
constexpr uint32_t kTmemCols = 256;
constexpr long long kMmaWaitCycles = 4000000000ll;

// tensor-memory columns
constexpr uint32_t TZ = 0, TDA = 64, TW23 = 128, TW1 = 192, TW4 = 208;

// shared-memory map (bytes from the dynamic base)
constexpr int SM_W1 = 0;                  // 64 x 16  [out][in], SBO 256
constexpr int SM_W2 = SM_W1 + 2048;       // 64 x 64, SBO 1024
constexpr int SM_W3 = SM_W2 + 8192;
constexpr int SM_W4 = SM_W3 + 8192;       // 16 x 64 (rows 3..15 zero)
constexpr int SM_X = SM_W4 + 2048;        // 128 x 16 features, SBO 256
constexpr int SM_A1 = SM_X + 4096;        // 128 x 64 activations, SBO 1024
constexpr int SM_A2 = SM_A1 + 16384;
constexpr int SM_A3 = SM_A2 + 16384;      // + 1 KB read by the M = 128 dW_4^T MMA
constexpr int SM_D4 = SM_A3 + 16384 + 1024;   // 128 x 16 output deltas, SBO 256
constexpr int SM_DL = SM_D4 + 4096;       // 128 x (64 + 64) hidden deltas in two halves, SBO 2048
constexpr int SM_B = SM_DL + 32768;       // biases: 64 + 64 + 64 + 8 float
constexpr int SM_BAR = SM_B + 800;        // two mbarriers (8 B each) + tensor-memory address (4 B)
constexpr int SM_END = SM_BAR + 32;
constexpr int SM_RED = SM_A1;             // after the last tile: 8 warps x 32 x 3 bias partials, 8 x 4, 8
constexpr int kSmemDyn = SM_END;
static_assert(kSmemDyn <= 111 * 1024, "two CTAs per SM need at most 111 KB each");
static_assert((8 * 32 * 3 + 8 * 4 + 8) * 4 <= 16384, "reduction scratch exceeds its alias");
static_assert(SM_X % 1024 == 0 && SM_A1 % 1024 == 0 && SM_A3 % 1024 == 0 && SM_DL % 1024 == 0, "tile alignment");

// 1 / (1 + e^-z) of two values with the hardware exponential and reciprocal (relative
// error ~2e-7, far below the bf16 rounding that follows)
__device__ __forceinline__ f2 sigmoid2(f2 z) {
  float a, b;
  f2_unpack(f2_mul(z, f2_pack(-1.4426950408889634f, -1.4426950408889634f)), a, b);
  asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(a));
  asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(b));
  f2_unpack(f2_add(f2_pack(a, b), f2_pack(1.f, 1.f)), a, b);
  asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(a));
  asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(b));
  return f2_pack(a, b);
}
// SiLU'(z) = s (1 + z (1 - s)) with s = sigmoid(z)
__device__ __forceinline__ f2 dsilu2(f2 z, f2 s) {
  const f2 one = f2_pack(1.f, 1.f), q = f2_fma(s, f2_pack(-1.f, -1.f), one);
  return f2_mul(s, f2_fma(z, q, one));
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&p);
}
__device__ __forceinline__ uint32_t pack2(f2 v) {
  float a, b;
  f2_unpack(v, a, b);
  return pack2(a, b);
}

// A warp's 32 x 32 block of a layer as fragments: frag[8 h + 2 j + g] holds row
// 16 h + 8 g + lane / 4, columns 8 j + 2 (lane % 4) and the next one.
__device__ __forceinline__ void ld_frag_nowait(uint32_t taddr, f2 f[16]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t r[16];
    tc::ld16x256_nowait(taddr + ((uint32_t)(16 * h) << 16), r);
#pragma unroll
    for (int k = 0; k < 8; ++k) f[8 * h + k] = f2_pack(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1]));
  }
}

// column sums of a block over the warp's rows: lane l's result is that of column
// frag_column(l)
__device__ __forceinline__ int frag_column(int lane) { return 8 * (lane >> 3) + 2 * (lane & 3) + ((lane >> 2) & 1); }
__device__ __forceinline__ float frag_column_sum(const f2 f[16], int lane) {
  float v[8];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    f2_unpack(f2_add(f2_add(f[2 * j], f[2 * j + 1]), f2_add(f[8 + 2 * j], f[8 + 2 * j + 1])), v[2 * j], v[2 * j + 1]);
#pragma unroll
  for (int c = 4; c >= 1; c >>= 1) {
    const bool up = (lane & (4 * c)) != 0;
#pragma unroll
    for (int i = 0; i < c; ++i) {
      const float send = up ? v[i] : v[i + c], keep = up ? v[i + c] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * c);
    }
  }
  return v[0];
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
  return v;
}

// a block as bf16 into a row-by-row tile whose 8-row groups are sbo bytes apart: one
// core matrix (8 rows x 16 bytes) per stmatrix step; `at` is this lane's row of the
// first four
__device__ __forceinline__ void stmatrix4(uint32_t at, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}
__device__ __forceinline__ void store_frag(uint32_t at, const f2 f[16], int sbo) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const f2* v = f + 8 * h + 4 * q;
      stmatrix4(at + 2 * h * sbo + 256 * q, pack2(v[0]), pack2(v[1]), pack2(v[2]), pack2(v[3]));
    }
}

__global__ void __launch_bounds__(kThreads, 2)
    k_mlp_grad_tc(const char* __restrict__ pack, int64_t off_w1, int64_t off_w2, int64_t off_w3, int64_t off_w4,
                  int64_t off_b, const __nv_bfloat16* __restrict__ feats, const float4* __restrict__ tgt,
                  const uint8_t* __restrict__ mask, int64_t m, float inv_cnt, float* __restrict__ partial,
                  float* __restrict__ loss_part, int* err) {
  extern __shared__ __align__(1024) char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = 32 * (warp & 3) + lane, half = warp >> 2, c0 = 32 * half;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + SM_BAR);   // [0] the next loads' MMAs, [1] weight gradients
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + SM_BAR + 16);
  float* bias = reinterpret_cast<float*>(smem + SM_B);

  // weights into row-by-row tiles (16-byte chunks of 8 bf16 along the inner index)
  for (int i = tid; i < 64 * 2; i += kThreads) {            // W1 [64][16]
    const int n = i >> 1, c = i & 1;
    *reinterpret_cast<uint4*>(smem + SM_W1 + tc::cm_off(n, 8 * c, 256)) =
        *reinterpret_cast<const uint4*>(pack + off_w1 + (size_t)(n * 16 + 8 * c) * 2);
  }
  for (int i = tid; i < 64 * 8; i += kThreads) {            // W2, W3 [64][64]
    const int n = i >> 3, c = i & 7;
    const int o = tc::cm_off(n, 8 * c, 1024);
    const size_t src = (size_t)(n * 64 + 8 * c) * 2;
    *reinterpret_cast<uint4*>(smem + SM_W2 + o) = *reinterpret_cast<const uint4*>(pack + off_w2 + src);
    *reinterpret_cast<uint4*>(smem + SM_W3 + o) = *reinterpret_cast<const uint4*>(pack + off_w3 + src);
  }
  for (int i = tid; i < 16 * 8; i += kThreads) {            // W4 [16][64], rows >= 3 zero
    const int n = i >> 3, c = i & 7;
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    if (n < 3) w = *reinterpret_cast<const uint4*>(pack + off_w4 + (size_t)(n * 64 + 8 * c) * 2);
    *reinterpret_cast<uint4*>(smem + SM_W4 + tc::cm_off(n, 8 * c, 1024)) = w;
  }
  for (int i = tid; i < 200; i += kThreads) bias[i] = *reinterpret_cast<const float*>(pack + off_b + (size_t)i * 4);
  // the padding behind A3 (read into dW_4^T rows that are never read back) and the
  // hidden-delta tile (its second halves must be zero before the first Delta_3)
  for (int i = tid; i < 64; i += kThreads)
    reinterpret_cast<uint4*>(smem + SM_A3 + 16384)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = tid; i < 32768 / 16; i += kThreads)
    reinterpret_cast<uint4*>(smem + SM_DL)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 1, 1);
    fence_mbarrier_init();
  }
  if (warp == 0) tc::alloc(tslot, kTmemCols);
  // a tile's features, by asynchronous copies (zeros beyond the last row)
  auto load_features = [&](int64_t tile, char* X) {
    const int r = tid >> 1, c = tid & 1;
    const int64_t p = tile * kRows + r;
    const bool in = p < m;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(X + tc::cm_off(r, 8 * c, 256))),
                 "l"(feats + (in ? p : 0) * 16 + 8 * c), "r"(in ? 16 : 0)
                 : "memory");
  };
  load_features(blockIdx.x, smem + SM_X);
  fence_proxy_async();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = *tslot;
  const uint32_t tlane = tbase + ((uint32_t)(32 * (warp & 3)) << 16);

  const uint32_t aA1 = smem_addr(smem + SM_A1), aA2 = smem_addr(smem + SM_A2), aA3 = smem_addr(smem + SM_A3),
                 aDL = smem_addr(smem + SM_DL);
  const uint32_t aW1 = smem_addr(smem + SM_W1), aW2 = smem_addr(smem + SM_W2), aW3 = smem_addr(smem + SM_W3),
                 aW4 = smem_addr(smem + SM_W4);
  constexpr uint32_t id64 = tc::idesc_bf16(128, 64), id16 = tc::idesc_bf16(128, 16);
  constexpr uint32_t idB64 = tc::idesc_bf16(128, 64, false, true);                  // B read MN-major
  constexpr uint32_t idT64 = tc::idesc_bf16(128, 64, true, true), idT16 = tc::idesc_bf16(128, 16, true, true);
  // this lane's row of the first four core matrices of its warp's block, with 8-row
  // groups 1024 (activations) and 2048 (deltas) bytes apart
  const uint32_t st_col = (uint32_t)((c0 >> 3) + (lane >> 4)) * 128 + (uint32_t)(lane & 7) * 16;
  const int st_grp = 4 * (warp & 3) + ((lane >> 3) & 1);
  const uint32_t st1 = (uint32_t)st_grp * 1024 + st_col, st2 = (uint32_t)st_grp * 2048 + st_col;

  float lsum = 0.f, bs1 = 0.f, bs2 = 0.f, bs3 = 0.f, bs4[3] = {0.f, 0.f, 0.f};
  uint32_t phase0 = 0, phase1 = 0;
  bool failed = false;

  // Z = A W^T over K = 64 (four K = 16 steps) for a hidden tile A and weight tile W
  auto mma_forward64 = [&](uint32_t d, uint32_t a, uint32_t w, uint32_t idesc) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      tc::mma(tbase + d, tc::desc_k(a + 256 * k, 1024), tc::desc_k(w + 256 * k, 1024), idesc, k > 0 ? 1u : 0u);
  };
  // DA = Delta W over K = 64 output features: Delta = the half of the delta tile at
  // dl (K-major, SBO 2048), W = a 64 x 64 weight tile read MN-major
  auto mma_data_grad = [&](uint32_t dl, uint32_t w) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      tc::mma(tbase + TDA, tc::desc_k(dl + 256 * k, 2048), tc::desc_mn(w + 2048 * k, 1024), idB64, k > 0 ? 1u : 0u);
  };
  // [dW3 | dW2] += DL^T A over the tile's rows
  auto mma_weight_grad = [&](uint32_t a, uint32_t acc) {
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
      tc::mma(tbase + TW23, tc::desc_mn(aDL + 4096 * kk, 2048), tc::desc_mn(a + 2048 * kk, 1024), idT64,
              kk > 0 ? 1u : acc);
  };
  // dW1 += Delta_1^T X (rows 64..127: the stale second half, never read back)
  auto mma_dw1 = [&](uint32_t x, uint32_t acc) {
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
      tc::mma(tbase + TW1, tc::desc_mn(aDL + 4096 * kk, 2048), tc::desc_mn(x + 512 * kk, 256), idT16,
              kk > 0 ? 1u : acc);
  };

  // one hand-over: operands written by every thread -> one thread issues; then every
  // thread waits for what it is about to read (wait_for)
  auto issue = [&](auto mmas) {
    fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after();
      mmas();
    }
    __syncwarp();
  };
  auto wait_for = [&](int k) {
    uint32_t& ph = k ? phase1 : phase0;
    if (!failed && !mbar_wait(bar + k, ph, kMmaWaitCycles)) {
      failed = true;
      atomicExch(err, 1);
    }
    ph ^= 1u;
    __syncwarp();
    tc::fence_after();
  };
  auto bias2 = [&](int l, int j) {
    const float2 b = *reinterpret_cast<const float2*>(bias + 64 * l + c0 + 8 * j + 2 * (lane & 3));
    return f2_pack(b.x, b.y);
  };

  // hidden layer l (0-based) forward epilogue: A = bf16(SiLU(Z + b)) of this warp's block
  auto epi_hidden = [&](int l, uint32_t A) {
    f2 z[16];
    ld_frag_nowait(tlane + TZ + c0, z);
    tc::wait_ld();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const f2 v = f2_add(z[k], bias2(l, (k & 7) >> 1));
      z[k] = f2_mul(v, sigmoid2(v));
    }
    store_frag(A + st1, z, 1024);
  };
  // Delta (two-wide, in d) -> half `dh` of the delta tile (bf16), the other half zeroed
  // when `zero_other`; returns the float32 column sum over the warp's rows
  auto put_delta = [&](const f2* d, int dh, bool zero_other) -> float {
    store_frag(aDL + 1024 * dh + st2, d, 2048);
    if (zero_other) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        stmatrix4(aDL + 1024 * (1 - dh) + st2 + 4096 * (k >> 1) + 256 * (k & 1), 0u, 0u, 0u, 0u);
    }
    return frag_column_sum(d, lane);
  };
  // backward epilogue of layer l < 2: Delta = DA * SiLU'(Z + b); the delta tile is
  // free once the weight gradient that reads it has completed (barrier 1)
  auto epi_back = [&](int l, int dh, bool zero_other) -> float {
    f2 d[16], z[16];
    ld_frag_nowait(tlane + TDA + c0, d);
    ld_frag_nowait(tlane + TZ + c0, z);
    tc::wait_ld();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const f2 v = f2_add(z[k], bias2(l, (k & 7) >> 1));
      d[k] = f2_mul(d[k], dsilu2(v, sigmoid2(v)));
    }
    wait_for(1);
    return put_delta(d, dh, zero_other);
  };

  const int64_t ntiles = (m + kRows - 1) / kRows;
  int64_t done = 0;        // tiles this CTA has walked
  int xo = SM_X, d4o = SM_D4;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++done) {
    const int64_t p = tile * kRows + row;
    const uint32_t aX = smem_addr(smem + xo), aD4 = smem_addr(smem + d4o);
    asm volatile("cp.async.wait_all;" ::: "memory");
    issue([&] {   // Z = X W1^T, and the last tile's dW1 (its features are where D4 goes)
      tc::mma(tbase + TZ, tc::desc_k(aX, 256), tc::desc_k(aW1, 256), id64, 0u);
      tc::commit(bar);
      if (done > 0) mma_dw1(aD4, done > 1 ? 1u : 0u);
    });
    wait_for(0);
    epi_hidden(0, aA1);
    issue([&] {   // Z = A1 W2^T
      mma_forward64(TZ, aA1, aW2, id64);
      tc::commit(bar);
    });
    wait_for(0);
    epi_hidden(1, aA2);
    issue([&] {   // Z = A2 W3^T
      mma_forward64(TZ, aA2, aW3, id64);
      tc::commit(bar);
    });
    const bool valid = half == 0 && p < m && (!mask || mask[p]);
    const float4 t = valid ? tgt[p] : make_float4(0.f, 0.f, 0.f, 0.f);
    wait_for(0);
    f2 ds[16];    // SiLU'(Z_3)
    {
      f2 z[16];
      ld_frag_nowait(tlane + TZ + c0, z);
      tc::wait_ld();
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const f2 v = f2_add(z[k], bias2(2, (k & 7) >> 1)), s = sigmoid2(v);
        z[k] = f2_mul(v, s);
        ds[k] = dsilu2(v, s);
      }
      store_frag(aA3 + st1, z, 1024);
    }
    issue([&] {   // Y = A3 W4^T (in the DA columns)
      mma_forward64(TDA, aA3, aW4, id16);
      tc::commit(bar);
    });
    wait_for(0);
    if (half == 0) {  // output: loss, d4 = 2 (y - t) / count on masked rows, bf16 D4 row
      float y[4];
      tc::ld4(tlane + TDA, y);
      float d4[3];
      const float tv[3] = {t.x, t.y, t.z};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float diff = valid ? (y[c] + bias[192 + c] - tv[c]) : 0.f;
        lsum += diff * diff;
        d4[c] = 2.f * diff * inv_cnt;
        bs4[c] += d4[c];
      }
      *reinterpret_cast<uint4*>(smem + d4o + tc::cm_off(row, 0, 256)) =
          make_uint4(pack2(d4[0], d4[1]), pack2(d4[2], 0.f), 0u, 0u);
      *reinterpret_cast<uint4*>(smem + d4o + tc::cm_off(row, 8, 256)) = make_uint4(0u, 0u, 0u, 0u);
    }
    issue([&] {   // DA = D4 W4; Z = A1 W2^T (Z_2 again), dW4^T += A3^T D4 under the epilogue
      tc::mma(tbase + TDA, tc::desc_k(aD4, 256), tc::desc_mn(aW4, 1024), idB64, 0u);
      tc::commit(bar);
      mma_forward64(TZ, aA1, aW2, id64);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        tc::mma(tbase + TW4, tc::desc_mn(aA3 + 2048 * kk, 1024), tc::desc_mn(aD4 + 512 * kk, 256), idT16,
                (kk > 0 || done > 0) ? 1u : 0u);
    });
    wait_for(0);
    {
      f2 d[16];
      ld_frag_nowait(tlane + TDA + c0, d);
      tc::wait_ld();
#pragma unroll
      for (int k = 0; k < 16; ++k) d[k] = f2_mul(d[k], ds[k]);
      bs3 += put_delta(d, 0, true);
    }
    issue([&] {   // DA = Delta_3 W3; [dW3 | dW2] += [Delta_3 | 0]^T A2
      mma_data_grad(aDL, aW3);
      tc::commit(bar);
      mma_weight_grad(aA2, done > 0 ? 1u : 0u);
      tc::commit(bar + 1);
    });
    wait_for(0);
    // D4 has been read (the commit above came after its MMAs): the next features go there
    if (tile + gridDim.x < ntiles) load_features(tile + gridDim.x, smem + d4o);
    bs2 += epi_back(1, 1, true);
    issue([&] {   // DA = Delta_2 W2; Z = X W1^T (Z_1 again); [dW3 | dW2] += [0 | Delta_2]^T A1
      mma_data_grad(aDL + 1024, aW2);
      tc::mma(tbase + TZ, tc::desc_k(aX, 256), tc::desc_k(aW1, 256), id64, 0u);
      tc::commit(bar);
      mma_weight_grad(aA1, 1u);
      tc::commit(bar + 1);
    });
    wait_for(0);
    bs1 += epi_back(0, 0, false);
    const int swap = xo;
    xo = d4o;
    d4o = swap;
  }
  issue([&] {     // the last tile's dW1
    mma_dw1(smem_addr(smem + d4o), done > 1 ? 1u : 0u);
    tc::commit(bar);
  });
  wait_for(0);

  {
    float* out = partial + (size_t)blockIdx.x * kNP;
    // weight gradients: dW1 and dW4^T rows in lanes 0..63 (warps 0, 1), dW3 rows o in
    // lanes 0..63 and dW2 rows o in lanes 64..127 of the shared accumulator
    if ((warp & 3) < 2 && half == 0) {
      float v[16];
      tc::ld16(tlane + TW1, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) out[OFF_W1 + row * 16 + i] = v[i];
      float w4[4];
      tc::ld4(tlane + TW4, w4);
#pragma unroll
      for (int o = 0; o < 3; ++o) out[OFF_W4 + o * 64 + row] = w4[o];
    }
    {
      float v[32];
      tc::ld32(tlane + TW23 + c0, v);
      const int o = row & 63;
      float* dst = out + (row < 64 ? OFF_W3 : OFF_W2) + o * 64 + c0;
#pragma unroll
      for (int i = 0; i < 32; ++i) dst[i] = v[i];
    }
    // bias gradients: lane l of warp w holds column 32 (w / 4) + frag_column(l) summed over its rows
    const int col = frag_column(lane);
    float* red = reinterpret_cast<float*>(smem + SM_RED);
    red[(0 * 8 + warp) * 32 + col] = bs1;
    red[(1 * 8 + warp) * 32 + col] = bs2;
    red[(2 * 8 + warp) * 32 + col] = bs3;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float b4 = warp_sum(bs4[c]);
      if (lane == 0) red[8 * 32 * 3 + warp * 4 + c] = b4;
    }
    const float ls = warp_sum(lsum);
    if (lane == 0) red[8 * 32 * 3 + 8 * 4 + warp] = ls;
    __syncthreads();
    if (tid < 192) {
      const int l = tid / 64, col = tid % 64, h = col / 32;
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < 4; ++w) s += red[(l * 8 + 4 * h + w) * 32 + (col & 31)];
      const int off = l == 0 ? OFF_B1 : (l == 1 ? OFF_B2 : OFF_B3);
      out[off + col] = s;
    } else if (tid < 195) {
      const int c = tid - 192;
      float s = 0.f;
      for (int w = 0; w < 4; ++w) s += red[8 * 32 * 3 + w * 4 + c];
      out[OFF_B4 + c] = s;
    } else if (tid == 195) {
      float s = 0.f;
      for (int w = 0; w < 8; ++w) s += red[8 * 32 * 3 + 8 * 4 + w];
      loss_part[blockIdx.x] = s;
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after();
    tc::dealloc(tbase, kTmemCols);
  }
}

}  // namespace

// per-block partial gradients [blocks][9603] and losses [blocks] of the network M
// over m rows, on tensor cores; blocks <= number of 128-row tiles; *err (device) is
// set when a wait on the tensor cores gave up
sph_status mlp_grad_tc(const sph_mlp* M, const __nv_bfloat16* feats, const float4* tgt, const uint8_t* mask,
                       int64_t m, float inv_cnt, float* partial, float* loss_part, int* err, int blocks,
                       cudaStream_t st) {
  static bool attr_set = false;
  if (!attr_set) {
    SPH_TRY_CUDA(cudaFuncSetAttribute(k_mlp_grad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemDyn));
    attr_set = true;
  }
  size_t ow1, ow2, ow3, ow4, ob;
  mlp_pack_layout(&ow1, &ow2, &ow3, &ow4, &ob);
  SPH_LAUNCH(k_mlp_grad_tc, blocks, kThreads, kSmemDyn, st)(
      reinterpret_cast<const char*>(mlp_pack_ptr(M)), (int64_t)ow1, (int64_t)ow2, (int64_t)ow3, (int64_t)ow4,
      (int64_t)ob, feats, tgt, mask, m, inv_cnt, partial, loss_part, err);
  SPH_TRY_CUDA(cudaGetLastError());
  return SPH_OK;
}

// grid of the training kernel: one CTA per 128-row tile, at most two per SM
int64_t mlp_grad_blocks(int64_t m, int num_sms) {
  int64_t blocks = (m + kRows - 1) / kRows;
  if (blocks > 2 * (int64_t)num_sms) blocks = 2 * (int64_t)num_sms;
  return blocks < 1 ? 1 : blocks;
}

}  // namespace sph
