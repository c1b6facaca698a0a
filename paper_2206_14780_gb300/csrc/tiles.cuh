// Tiles: runs of TS consecutive 32-row slices of the cell-sorted order whose
// neighbours are kept as 16-bit positions in a tile-local list of distinct
// neighbours (the union), so that a block can hold every value its rows gather
// in shared memory.
//
// Rows that are consecutive along the Morton curve share most of their
// neighbours: 256 rows of the lava box have ~20,000 neighbour entries but only
// ~1,150 distinct neighbours (18 KB as float4).  A gather from L1 costs one tag
// look-up per distinct 128-byte line, ~17 per warp; a 16-byte gather from shared
// memory costs one cycle per 8-lane quarter plus bank conflicts.  Each row's
// entries are ordered so that lane l of a warp reads bank group (l + j - 2) mod 8 at
// step j while it has such an entry left (5.1 cycles per warp instead of 9.3 in
// ascending order, counted on the host for the box).
//
// Storage: entry j of row s lies at lbase(slice) + 128 (j / 4) + 4 (s % 32) +
// j % 4, i.e. a lane's four consecutive entries are contiguous: one 8-byte load
// brings four positions, one 16-byte load four coefficients.  Positions are
// stored times 16 (the byte offset of the float4), so a union holds at most
// kTileUnion rows.  The last group of a row is filled up with its first entry's
// position and zero coefficients.  Wall rows list their fluid neighbours first.
#pragma once

#include "apply.cuh"
#include "dfloat.cuh"
#include "sph_internal.cuh"

namespace sph {

constexpr int kTileUnion = 4095;    // distinct neighbours a tile may have (positions x 16 in 16 bits)
constexpr int kTileCells = 256;     // cells a tile's search region may span
constexpr int kTileHeads = 64;      // cells the rows of a tile may lie in

struct TileView {
  const uint16_t* idx;     // union positions x 16, at slice * istride
  int64_t istride;         // entries per slice of idx (32 x the capacity)
  const float* hi;         // coefficients of A(dt), at off[slice]
  const float* lo;         // a = hi + lo
  const int64_t* off;      // [nslices + 1] entry offsets of hi and lo
  const int32_t* cnt;      // [n_pad] entries with a coefficient
  const uint8_t* kind;     // [n_pad]
  const float* invD;       // [n_pad]
  const int32_t* uni;      // [ntiles][ustride] the rows of each union, ascending
  const int32_t* unum;     // [ntiles]
  int32_t ustride;
  int32_t ntiles;
  int64_t nslices;
};

// 16-byte asynchronous copy global -> shared (the thread's own group)
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// u[i] = v[uni[i]] for the tile's union; every thread of the block calls it and
// then __syncthreads (the copies are complete for the calling thread on return)
__device__ __forceinline__ void tile_load_union(const TileView& op, int64_t tile, const float4* __restrict__ v,
                                                float4* __restrict__ u) {
  const int32_t* __restrict__ ids = op.uni + tile * op.ustride;
  const int nu = op.unum[tile];
  for (int i = threadIdx.x; i < nu; i += blockDim.x) cp_async16(u + i, v + ids[i]);
}

// the four byte offsets of a lane's group
__device__ __forceinline__ void tile_unpack(uint2 p, uint32_t (&o)[4]) {
  o[0] = p.x & 0xffffu;
  o[1] = p.x >> 16;
  o[2] = p.y & 0xffffu;
  o[3] = p.y >> 16;
}

__device__ __forceinline__ const float4& tile_at(const float4* u, uint32_t off) {
  return *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(u) + off);
}

// The coefficient and position stream of one row: groups first, first + step, ...
// (first: the thread's split, step: the splits), kTileDepth groups in flight in
// registers.  The stream is what the apply waits on: 24 bytes a lane and group, and
// with 32 warps per SM one group ahead keeps only 25 KB in flight; start() is called
// before the union is waited for.
constexpr int kTileDepth = 2;
constexpr int kTileBlocks = 5;   // resident blocks per SM asked of the compiler

template <int D>
struct TileStreamD {
  float4 a[D];
  uint2 p[D];
  const float4* ph;
  const uint2* pi;
  int ng, ngw;   // groups of this row, most groups of the warp's rows

  // unconditional for the whole warp: a shorter row reads its last group again
  __device__ __forceinline__ void fetch(int d, int g) {
    if (g < ngw) {
      const int at = min(g, ng > 0 ? ng - 1 : 0) * 32;
      a[d] = __ldcs(ph + at);
      p[d] = __ldcs(pi + at);
    }
  }
  __device__ __forceinline__ void start(const TileView& op, int64_t sl, int lane, int c, int first, int step) {
    start_at(op, sl, __any_sync(0xffffffffu, c > 0) ? op.off[sl] : 0, lane, c, first, step);
  }
  // o0 = op.off[sl]
  __device__ __forceinline__ void start_at(const TileView& op, int64_t sl, int64_t o0, int lane, int c, int first,
                                           int step) {
    ng = (c + 3) >> 2;
    ngw = __reduce_max_sync(0xffffffffu, ng);
    ph = reinterpret_cast<const float4*>(op.hi + o0) + lane;
    pi = reinterpret_cast<const uint2*>(op.idx + sl * op.istride) + lane;
#pragma unroll
    for (int d = 0; d < D; ++d) fetch(d, first + d * step);
  }
  // ax,ay,az += sum of a (k - v_a)
  __device__ __forceinline__ void sum(const float4* __restrict__ u, int first, int step, float kx, float ky, float kz,
                                      float& ax, float& ay, float& az) {
    for (int g0 = first; g0 < ngw; g0 += D * step) {
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const int g = g0 + d * step;
        if (g < ngw) {
          const float4 ac = a[d];
          const uint2 pc = p[d];
          fetch(d, g + D * step);
          if (g < ng) {
            uint32_t o[4];
            tile_unpack(pc, o);
            const float av[4] = {ac.x, ac.y, ac.z, ac.w};
            float4 va[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) va[k] = tile_at(u, o[k]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              ax = fmaf(av[k], kx - va[k].x, ax);
              ay = fmaf(av[k], ky - va[k].y, ay);
              az = fmaf(av[k], kz - va[k].z, az);
            }
          }
        }
      }
    }
  }
};

using TileStream = TileStreamD<kTileDepth>;

// f(byte offset of a float4 in the union) for every neighbour of a row, wall neighbours
// of wall rows included: nf interleaved entries, then c - nf from the next group on.
// The row's groups first, first + step, ...; the next group's positions are loaded
// before the current one is worked on.
template <class F>
__device__ __forceinline__ void tile_walk(const uint16_t* __restrict__ idx, int64_t istride, int64_t sl, int lane, int nf,
                                          int c, int first, int step, F f) {
  const uint2* __restrict__ pi = reinterpret_cast<const uint2*>(idx + sl * istride) + lane;
  const int gf = (nf + 3) >> 2, ng = gf + ((c - nf + 3) >> 2);
  uint2 p = first < ng ? pi[first * 32] : make_uint2(0u, 0u);
  for (int g = first; g < ng; g += step) {
    const uint2 pn = g + step < ng ? pi[(g + step) * 32] : p;
    uint32_t o[4];
    tile_unpack(p, o);
    const int left = g < gf ? nf - 4 * g : c - nf - 4 * (g - gf);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < left) f(o[k]);
    p = pn;
  }
}

// the row's value from its sum, as apply_row
__device__ __forceinline__ float4 tile_finish(uint8_t kd, float4 vb, float ax, float ay, float az, float sc) {
  if (kd == KIND_FLUID) return make_float4((vb.x + ax) * sc, (vb.y + ay) * sc, (vb.z + az) * sc, 0.f);
  if (kd == KIND_SHEPARD) return make_float4((vb.x - ax) * sc, (vb.y - ay) * sc, (vb.z - az) * sc, 0.f);
  return make_float4(vb.x * sc, vb.y * sc, vb.z * sc, 0.f);
}

// Adds the partial sums of the S = 8 / TS threads that share a row (split > 0
// hand theirs over through `part`, [S - 1][32 TS][3] floats); only split 0 holds
// the result.  Every thread of the block calls it.
template <int TS>
__device__ __forceinline__ void tile_combine(float* part, int split, int row, float& ax, float& ay, float& az) {
  constexpr int S = 8 / TS, R = 32 * TS;
  if (S == 1) return;
  if (split > 0) {
    float* q = part + ((split - 1) * R + row) * 3;
    q[0] = ax;
    q[1] = ay;
    q[2] = az;
  }
  __syncthreads();
  if (split == 0) {
#pragma unroll
    for (int k = 0; k < S - 1; ++k) {
      const float* q = part + (k * R + row) * 3;
      ax += q[0];
      ay += q[1];
      az += q[2];
    }
  }
}

// A row's operator sum in double-float arithmetic over the tile form (residual_row
// of residual_row.cuh with the gathers from shared memory).  X2: x = hi + lo in two
// arrays uh, ul; else a float32 vector in uh.
template <bool X2>
__device__ __forceinline__ void tile_residual_row(const TileView& op, const float4* uh, const float4* ul, int64_t sl,
                                                  int lane, int c, int first, int step, float4 kh, float4 kl,
                                                  DFAcc& a0, DFAcc& a1, DFAcc& a2) {
  const int64_t o0 = op.off[sl];
  const float4* __restrict__ ph = reinterpret_cast<const float4*>(op.hi + o0) + lane;
  const float4* __restrict__ pl = reinterpret_cast<const float4*>(op.lo + o0) + lane;
  const uint2* __restrict__ pi = reinterpret_cast<const uint2*>(op.idx + sl * op.istride) + lane;
  const int ng = (c + 3) >> 2;
  float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
  uint2 p = make_uint2(0u, 0u);
  if (first < ng) {
    h = __ldcs(ph + first * 32);
    l = __ldcs(pl + first * 32);
    p = __ldcs(pi + first * 32);
  }
  for (int g = first; g < ng; g += step) {
    float4 hn = h, ln = l;
    uint2 pn = p;
    if (g + step < ng) {
      hn = __ldcs(ph + (g + step) * 32);
      ln = __ldcs(pl + (g + step) * 32);
      pn = __ldcs(pi + (g + step) * 32);
    }
    uint32_t o[4];
    tile_unpack(p, o);
    const float hv[4] = {h.x, h.y, h.z, h.w}, lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 xh = tile_at(uh, o[k]);
      const float4 xl = X2 ? tile_at(ul, o[k]) : make_float4(0.f, 0.f, 0.f, 0.f);
      a0.add(hv[k], lv[k], kh.x, xh.x, kl.x, xl.x);
      a1.add(hv[k], lv[k], kh.y, xh.y, kl.y, xl.y);
      a2.add(hv[k], lv[k], kh.z, xh.z, kl.z, xl.z);
    }
    h = hn;
    l = ln;
    p = pn;
  }
}

TileView tile_view(const sph_neighbors* H);
// dynamic shared memory of a kernel that holds `bytes_per_row` of every union row
size_t tile_smem(const sph_neighbors* H, int bytes_per_row);
// one of a kernel template's four instances, by the handle's slices per tile
#define SPH_TILE_PICK(H, name, ...)                                                                              \
  ((H)->tile_ts == 8 ? name<8 __VA_ARGS__>                                                                       \
                     : ((H)->tile_ts == 4 ? name<4 __VA_ARGS__> : ((H)->tile_ts == 2 ? name<2 __VA_ARGS__> : name<1 __VA_ARGS__>)))
#define SPH_COMMA ,

// blocks for a tile kernel: every tile, or as many as are resident at once
int tile_grid(const sph_neighbors* H, const void* kernel, size_t smem);

}  // namespace sph
