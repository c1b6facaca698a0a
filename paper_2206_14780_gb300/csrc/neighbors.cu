// Cell binning, counting sort and neighbour lists (paper Sec. 5.2: a Wendland
// particle at h = 1.3 dp has about 80 neighbours; App. A: the relative position
// is one difference so r_ab = -r_ba bit for bit).
//
// Steps (one launch each):
//   keys      cell of every particle: floor((x - lo) / cell) per axis in float64,
//             wrapped on periodic axes, clamped on open ones; per-cell counts.
//             Cells are ordered along a Morton (Z-order) curve: segment r of the
//             sorted order holds the cell of rank r, so 32-row slices and the
//             slices a block works on are compact in space and their neighbour
//             gathers share cache lines (the apply is bound by those gathers)
//   scan      exclusive prefix sum of the counts -> cell_start
//   scatter   particles into their cell's segment (atomics: any order)
//   sort      each particle's place in its segment by caller index (makes the
//             layout deterministic), with the sorted copies of pos / rho / mu /
//             type, perm and iperm
//   search    per tile of consecutive rows: the particles of all cells around the
//             tile into shared memory once, then each row scans its 27 cells there
//   plan      per tile: the distinct neighbours (the union) and each row's entries
//             as positions in it, in the order the apply reads them (tiles.cuh)
// Where a tile's cells do not fit (very uneven densities), the lists are built by
// a scan of global memory instead, as 32-bit rows (k_neighbors).  The host reads
// the flags and totals back once, at the end.
//
// The predicate is decided exactly as the float64 definition: a float32 test
// decides every pair outside a band around (R h)^2 (R h: the kernel support radius) whose half-width bounds the
// float32 rounding of r^2; pairs inside the band are recomputed in float64 with
// the same operations, in the same order and without contraction.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "f32x2.cuh"
#include "tiles.cuh"

namespace sph {

namespace {

// flags[0]: bits below; [1] largest |coordinate| (bits), [2] fullest cell, [3]
// largest union, [4] largest search region.  FLAG_REGION: a tile's region is larger than
// the places asked for; FLAG_UNEVEN: a tile's cells are too many for any region size.
enum : int32_t { FLAG_NONFINITE = 1, FLAG_CAPACITY = 2, FLAG_BADFIELD = 4, FLAG_REGION = 8, FLAG_UNEVEN = 16 };

// a cell this full cannot belong to a particle set of at most maxnb neighbours;
// the quadratic steps below are not run on one
__host__ __device__ inline int64_t cell_limit(int32_t maxnb) { return 64LL * (maxnb + 1); }

__device__ __forceinline__ bool build_stopped(const int32_t* flags, int32_t maxnb) {
  return (flags[0] & FLAG_NONFINITE) != 0 || (int64_t)flags[2] > cell_limit(maxnb);
}

__global__ void k_cell_keys(const float4* __restrict__ pos, int64_t n, Grid g, const int32_t* __restrict__ rank,
                            int32_t* __restrict__ key, int32_t* __restrict__ cell_count, int32_t* __restrict__ flags,
                            unsigned int* __restrict__ max_abs_bits) {
  float local_max = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float4 p = pos[i];
    float c3[3] = {p.x, p.y, p.z};
    bool finite = isfinite(p.x) && isfinite(p.y) && isfinite(p.z) && isfinite(p.w);
    if (!finite) atomicOr(&flags[0], FLAG_NONFINITE);
    int c[3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      double u = finite ? ((double)c3[ax] - g.lo[ax]) / g.cell[ax] : 0.0;
      u = fmin(fmax(u, -1.0e9), 1.0e9);
      long long k = (long long)floor(u);
      int nc = g.ncell[ax];
      if (g.periodic[ax]) {
        k %= nc;
        if (k < 0) k += nc;
      } else {
        k = k < 0 ? 0 : (k >= nc ? nc - 1 : k);
      }
      c[ax] = (int)k;
      if (finite) local_max = fmaxf(local_max, fabsf(c3[ax]));
    }
    int32_t kk = c[0] + g.ncell[0] * (c[1] + g.ncell[1] * c[2]);
    key[i] = kk;
    atomicAdd(&cell_count[rank[kk]], 1);
  }
  // warp max then one atomic per warp (non-negative floats order like their bits)
  for (int o = 16; o > 0; o >>= 1) local_max = fmaxf(local_max, __shfl_xor_sync(0xffffffffu, local_max, o));
  if ((threadIdx.x & 31) == 0) atomicMax(max_abs_bits, __float_as_uint(local_max));
}

// Single-block exclusive scan of m int32 values, each multiplied by `mul`;
// out has m + 1 entries (out[m] = total).  Also reports the largest input.
template <class TOut>
__global__ void k_scan(const int32_t* __restrict__ in, TOut* __restrict__ out, int64_t m, int64_t mul,
                       int32_t* __restrict__ max_out) {
  __shared__ long long s[1024];
  __shared__ int smax[1024];
  const int t = threadIdx.x;
  const int64_t chunk = (m + 1023) / 1024;
  const int64_t b = (int64_t)t * chunk;
  const int64_t e = b + chunk < m ? b + chunk : m;
  long long sum = 0;
  int mx = 0;
  for (int64_t i = b; i < e; ++i) {
    int v = in[i];
    sum += (long long)v * mul;
    mx = v > mx ? v : mx;
  }
  s[t] = sum;
  smax[t] = mx;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    long long v = t >= off ? s[t - off] : 0;
    int w = t >= off ? smax[t - off] : 0;
    __syncthreads();
    s[t] += v;
    smax[t] = smax[t] > w ? smax[t] : w;
    __syncthreads();
  }
  long long run = s[t] - sum;
  for (int64_t i = b; i < e; ++i) {
    out[i] = (TOut)run;
    run += (long long)in[i] * mul;
  }
  if (t == 1023) {
    out[m] = (TOut)s[1023];
    if (max_out) *max_out = smax[1023];
  }
}

// The same scan over many blocks, for long inputs (the one-block form walks
// m / 1024 values per thread one after the other: 54 us for the 65,600 cells of the
// 1.16M box against 5 us for these two kernels).  Tiles of 4096 values: first each
// tile's sum, then each block adds up the sums before its own and scans its tile.
constexpr int kScanTile = 4096;

__global__ void __launch_bounds__(1024) k_scan_sums(const int32_t* __restrict__ in, int64_t m,
                                                    long long* __restrict__ sums, int32_t* __restrict__ max_out) {
  __shared__ long long ws[32];
  __shared__ int wm[32];
  const int t = threadIdx.x;
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  long long sum = 0;
  int mx = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t i = base + k * 1024 + t;
    const int v = i < m ? in[i] : 0;
    sum += v;
    mx = max(mx, v);
  }
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((t & 31) == 0) {
    ws[t >> 5] = sum;
    wm[t >> 5] = mx;
  }
  __syncthreads();
  if (t < 32) {
    sum = ws[t];
    mx = wm[t];
    for (int o = 16; o > 0; o >>= 1) {
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (t == 0) {
      sums[blockIdx.x] = sum;
      if (max_out) atomicMax(max_out, mx);
    }
  }
}

template <class TOut>
__global__ void __launch_bounds__(1024) k_scan_tiles(const int32_t* __restrict__ in, TOut* __restrict__ out, int64_t m,
                                                     int64_t mul, const long long* __restrict__ sums) {
  __shared__ long long ws[32];
  __shared__ long long before;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  long long pre = 0;
  for (int64_t i = t; i < blockIdx.x; i += 1024) pre += sums[i];
  for (int o = 16; o > 0; o >>= 1) pre += __shfl_xor_sync(0xffffffffu, pre, o);
  if (lane == 0) ws[w] = pre;
  __syncthreads();
  if (t < 32) {
    pre = ws[t];
    for (int o = 16; o > 0; o >>= 1) pre += __shfl_xor_sync(0xffffffffu, pre, o);
    if (t == 0) before = pre;
  }
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kScanTile + 4 * t;
  int v[4];
  long long own = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = base + k < m ? in[base + k] : 0;
    own += v[k];
  }
  long long inc = own;
  for (int o = 1; o < 32; o <<= 1) {
    const long long x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  if (lane == 31) ws[w] = inc;
  __syncthreads();
  if (t < 32) {
    long long x = ws[t];
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    ws[t] = x;
  }
  __syncthreads();
  long long run = before + (w > 0 ? ws[w - 1] : 0) + inc - own;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (base + k < m) out[base + k] = (TOut)(run * mul);
    run += v[k];
    if (base + k == m - 1) out[m] = (TOut)(run * mul);
  }
}

__global__ void k_cell_scatter(const int32_t* __restrict__ key, const int32_t* __restrict__ rank, int64_t n,
                               const int32_t* __restrict__ cell_start, int32_t* __restrict__ cursor,
                               int32_t* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t k = rank[key[i]];
    int32_t slot = cell_start[k] + atomicAdd(&cursor[k], 1);
    out[slot] = (int32_t)i;
  }
}

// Each particle's row: its cell's start plus the number of smaller caller indices
// in the cell's (unordered) segment; ~18 L1-cached reads per particle at h = 1.3 dx.
// Writes the sorted copies at once.  (A sort by one thread per cell, then a gather,
// took 63 + 20 us on the 1.16M box and 190 us on 5,616 particles in cells of 64.)
__global__ void k_cell_sort(const int32_t* __restrict__ ids, const int32_t* __restrict__ cell_start, int64_t n,
                            int64_t n_pad, int32_t maxnb, const float4* __restrict__ pos, const float* __restrict__ rho,
                            const float* __restrict__ mu, const uint8_t* __restrict__ ptype,
                            const int32_t* __restrict__ key, const int32_t* __restrict__ rank,
                            int32_t* __restrict__ perm, int32_t* __restrict__ iperm, float4* __restrict__ pos_s,
                            float* __restrict__ rho_s, float* __restrict__ mu_s, uint8_t* __restrict__ type_s,
                            int32_t* __restrict__ key_s, int32_t* __restrict__ flags) {
  if (build_stopped(flags, maxnb)) return;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n_pad; s += (int64_t)gridDim.x * blockDim.x) {
    if (s < n) {
      const int32_t i = ids[s];
      const int32_t k = key[i], c = rank[k];
      const int32_t b = cell_start[c], e = cell_start[c + 1];
      int32_t at = b;
      for (int32_t t = b; t < e; ++t) at += ids[t] < i ? 1 : 0;
      perm[at] = i;
      iperm[i] = at;
      pos_s[at] = pos[i];
      const float r = rho[i], m = mu[i];
      if (!(isfinite(r) && r > 0.f && isfinite(m) && m > 0.f)) atomicOr(&flags[0], FLAG_BADFIELD);
      rho_s[at] = r;
      mu_s[at] = m;
      const uint8_t t = ptype[i];
      type_s[at] = t > 1 ? 1 : t;
      key_s[at] = k;
    } else {
      pos_s[s] = make_float4(0.f, 0.f, 0.f, 0.f);
      rho_s[s] = 1.f;
      mu_s[s] = 1.f;
      type_s[s] = 1;
      key_s[s] = 0;
    }
  }
}

// float64 form of the neighbour predicate, operation for operation.
__device__ __forceinline__ bool pair_inside_f64(float4 pt, float4 ps, const Grid& g, double R2) {
  double d[3] = {__dsub_rn((double)pt.x, (double)ps.x), __dsub_rn((double)pt.y, (double)ps.y),
                 __dsub_rn((double)pt.z, (double)ps.z)};
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    if (g.periodic[ax]) {
      double L = g.L[ax];
      double k = rint(__ddiv_rn(d[ax], L));
      d[ax] = __dsub_rn(d[ax], __dmul_rn(L, k));
    }
  }
  double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
  return r2 < R2;
}

struct Band {
  float lo2, hi2;   // float32 r^2 below lo2: inside; at or above hi2: outside
  double R2;        // (R h)^2 in float64, R h the support radius
  float L[3], invL[3];
};

// One pass over the 27 cells around each particle: the count and the list at
// once.  Lists live in a fixed-capacity SELL-32 layout (every slice maxnb
// entries wide, entry j of row s at (s / 32) 32 maxnb + 32 j + s % 32), so no
// counting pass has to size them first; a row with more than maxnb neighbours
// raises FLAG_CAPACITY and keeps its first maxnb.
__global__ void __launch_bounds__(kBlock) k_neighbors(const float4* __restrict__ pos_s, const int32_t* __restrict__ key_s,
                                                      const int32_t* __restrict__ rank,
                                                      const int32_t* __restrict__ cell_start, int64_t n, int64_t n_pad,
                                                      Grid g, Band band, int32_t maxnb, int32_t* __restrict__ cnt,
                                                      int32_t* __restrict__ nbr, int32_t* __restrict__ flags) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n_pad; s += (int64_t)gridDim.x * blockDim.x) {
    if (s >= n) {
      cnt[s] = 0;
      continue;
    }
    const float4 ps = pos_s[s];
    const int32_t key = key_s[s];
    const int nx = g.ncell[0], ny = g.ncell[1], nz = g.ncell[2];
    const int cx = key % nx, cy = (key / nx) % ny, cz = key / (nx * ny);
    int32_t count = 0;
    const int64_t base = (s / kSlice) * (int64_t)kSlice * maxnb + (s % kSlice);
    for (int dz = -1; dz <= 1; ++dz) {
      int z = cz + dz;
      if (g.periodic[2]) z = (z + nz) % nz;
      else if (z < 0 || z >= nz) continue;
      for (int dy = -1; dy <= 1; ++dy) {
        int y = cy + dy;
        if (g.periodic[1]) y = (y + ny) % ny;
        else if (y < 0 || y >= ny) continue;
        for (int dx = -1; dx <= 1; ++dx) {
          int x = cx + dx;
          if (g.periodic[0]) x = (x + nx) % nx;
          else if (x < 0 || x >= nx) continue;
          const int32_t cell = rank[x + nx * (y + ny * z)];
          const int32_t tb = cell_start[cell], te = cell_start[cell + 1];
          for (int32_t t = tb; t < te; ++t) {
            if (t == s) continue;
            const float4 pt = pos_s[t];
            float d0 = pt.x - ps.x, d1 = pt.y - ps.y, d2 = pt.z - ps.z;
            if (g.periodic[0]) d0 -= band.L[0] * rintf(d0 * band.invL[0]);
            if (g.periodic[1]) d1 -= band.L[1] * rintf(d1 * band.invL[1]);
            if (g.periodic[2]) d2 -= band.L[2] * rintf(d2 * band.invL[2]);
            const float r2 = d0 * d0 + d1 * d1 + d2 * d2;
            bool in;
            if (r2 < band.lo2) in = true;
            else if (r2 >= band.hi2) in = false;
            else in = pair_inside_f64(pt, ps, g, band.R2);
            if (in) {
              if (count < maxnb) nbr[base + (int64_t)count * kSlice] = t;
              ++count;
            }
          }
        }
      }
    }
    if (count > maxnb) {
      atomicOr(&flags[0], FLAG_CAPACITY);
      count = maxnb;
    }
    cnt[s] = count;
  }
}

// What the float32 filter's band is made of; the largest coordinate is on the device.
struct BandIn {
  double rsup, big;
  float L[3], invL[3];
};

// band of the float32 filter: coordinate differences carry at most a few float32
// roundings of the largest coordinate or period E; r^2 then errs by at most
// 2 sqrt(3) (R h) E + 3 E^2 plus its own three roundings
__host__ __device__ inline Band band_of(const BandIn& in, float max_abs) {
  Band band;
  const double big = (double)max_abs > in.big ? (double)max_abs : in.big;
  const double E = 4.0 * big * (1.0 / 8388608.0);
  band.R2 = in.rsup * in.rsup;
  const double B = 4.0 * in.rsup * E + 3.0 * E * E + 1e-6 * band.R2;
  const double low = (band.R2 - B) * (1.0 - 1e-7);
  band.lo2 = (float)(low > 0.0 ? low : 0.0);
  band.hi2 = (float)((band.R2 + B) * (1.0 + 1e-7));
  for (int ax = 0; ax < 3; ++ax) {
    band.L[ax] = in.L[ax];
    band.invL[ax] = in.invL[ax];
  }
  return band;
}

// offset (in 16-bit entries) of entry j of row `lane` inside its slice's list
__device__ __forceinline__ int tile_entry(int j, int lane) { return (j >> 2) * 128 + lane * 4 + (j & 3); }

// The neighbour search of one tile.  The distinct cells around the cells of the
// tile's rows (at most kTileCells; ~105 for 256 rows of the box) are collected in
// a hash table and sorted by Morton rank; their particles (~1,900 of up to `cap`)
// are read into shared memory once, as three coordinate arrays with each cell padded
// to a multiple of four places (the padding lies at infinity).  Every row then scans
// its 27 cells there, four candidates per step: three 16-byte loads, the distances in
// two-wide float32 instructions.  The scan is bound by issue slots (475 candidates
// per row), not by memory.  LPR = 8 / TS lanes share a row and take its groups of
// four in turn, list places from a prefix sum over the lanes, so small particle sets
// still fill the chip.  Entries are places in the region, entry j of a row at
// rstride * slice + 32 j + lane, in the order of k_neighbors; k_tile_plan turns them
// into union positions.  A tile that does not fit raises FLAG_REGION or FLAG_UNEVEN and
// is left.
template <int TS, bool PER>
__global__ void __launch_bounds__(256) k_tile_search(
    const float4* __restrict__ pos_s, const int32_t* __restrict__ key_s, const int32_t* __restrict__ rank,
    const int32_t* __restrict__ cell_start, int64_t n, int64_t nslices, Grid g, BandIn bin, int32_t maxnb, int cap,
    int32_t* __restrict__ cnt, uint16_t* __restrict__ raw, int2* __restrict__ tcells, int32_t* __restrict__ tncell,
    int32_t* __restrict__ width, unsigned long long* __restrict__ total, int32_t* __restrict__ maxc,
    int32_t* __restrict__ flags) {
  constexpr int R = 32 * TS, LPR = 8 / TS, HASH = 1024;
  extern __shared__ __align__(16) float reg[];    // x[cap], y[cap], z[cap]
  __shared__ int hash[HASH];
  __shared__ int crank[kTileCells], ccnt[kTileCells], srank[kTileCells], sstart[kTileCells], scnt[kTileCells];
  __shared__ int soff[kTileCells + 1];
  __shared__ int hd[kTileHeads * 27];             // cell rank, then offset | count << 16
  __shared__ int headrow[kTileHeads];
  __shared__ int wsum[8];
  __shared__ int rcnt[R];
  __shared__ int ncell;
  __shared__ Band band;
  if (build_stopped(flags, maxnb)) return;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t tile = blockIdx.x, row0 = tile * R;
  for (int i = tid; i < HASH; i += 256) hash[i] = -1;
  if (tid == 0) {
    ncell = 0;
    band = band_of(bin, __uint_as_float((unsigned)flags[1]));
  }
  // the runs of rows in one cell: one head each, in row order
  const int64_t hs = row0 + tid;
  const bool head = tid < R && hs < n && (tid == 0 || key_s[hs] != key_s[hs - 1]);
  const unsigned hb = __ballot_sync(0xffffffffu, head);
  if (lane == 0) wsum[wid] = __popc(hb);
  __syncthreads();
  int hbase = 0, nheads = 0;
  for (int w = 0; w < 8; ++w) {
    if (w < wid) hbase += wsum[w];
    nheads += wsum[w];
  }
  const int hidx = hbase + __popc(hb & ((2u << lane) - 1u)) - 1;   // the head of row tid
  if (tid < R) rcnt[tid] = hidx;
  if (head && hidx < kTileHeads) headrow[hidx] = tid;
  __syncthreads();
  const int nx = g.ncell[0], ny = g.ncell[1], nz = g.ncell[2];
  if (nheads <= kTileHeads) {
    for (int q = tid; q < nheads * 27; q += 256) {
      const int32_t key = key_s[row0 + headrow[q / 27]];
      const int o = q % 27;
      int x = key % nx + o % 3 - 1, y = (key / nx) % ny + (o / 3) % 3 - 1, z = key / (nx * ny) + o / 9 - 1;
      bool in = true;
      if (g.periodic[0]) x = (x + nx) % nx;
      else in = in && x >= 0 && x < nx;
      if (g.periodic[1]) y = (y + ny) % ny;
      else in = in && y >= 0 && y < ny;
      if (g.periodic[2]) z = (z + nz) % nz;
      else in = in && z >= 0 && z < nz;
      int c = -1;
      if (in) {
        c = rank[x + nx * (y + ny * z)];
        const int b = cell_start[c], many = cell_start[c + 1] - b;
        if (many == 0) {
          c = -1;
        } else {
          unsigned h = ((unsigned)c * 2654435761u) >> 22;
          for (int tries = 0; tries < HASH; ++tries) {
            const int was = atomicCAS(&hash[h], -1, c);
            if (was == c) break;
            if (was == -1) {
              const int at = atomicAdd(&ncell, 1);
              if (at < kTileCells) {
                crank[at] = c;
                ccnt[at] = many;
              }
              break;
            }
            h = (h + 1) & (HASH - 1);
          }
        }
      }
      hd[q] = c;
    }
  }
  __syncthreads();
  const int m = min(ncell, kTileCells);
  if (nheads > kTileHeads || ncell > kTileCells) {
    if (tid == 0) atomicOr(&flags[0], FLAG_UNEVEN);
    return;
  }
  // cells by rank, and their offsets in the region
  if (tid < m) {
    const int myrank = crank[tid];
    int place = 0;
    for (int k = 0; k < m; ++k) place += crank[k] < myrank ? 1 : 0;
    srank[place] = myrank;
    sstart[place] = cell_start[myrank];
    scnt[place] = ccnt[tid];
  }
  __syncthreads();
  {
    const int v = tid < m ? (scnt[tid] + 3) & ~3 : 0;
    int inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    int pre = 0;
    for (int w = 0; w < wid; ++w) pre += wsum[w];
    if (tid < m) soff[tid] = pre + inc - v;
    if (tid == m - 1) soff[m] = pre + inc;
  }
  __syncthreads();
  const int nreg = m > 0 ? soff[m] : 0;
  if (tid == 0) atomicMax(&flags[4], nreg);
  if (nreg > cap) {
    if (tid == 0) atomicOr(&flags[0], FLAG_REGION);
    return;
  }
  for (int q = tid; q < nheads * 27; q += 256) {
    const int c = hd[q];
    int pk = 0;
    if (c >= 0) {
      int lo = 0, hi = m - 1;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (srank[mid] < c) lo = mid + 1;
        else hi = mid;
      }
      pk = soff[lo] | (scnt[lo] << 16);
    }
    hd[q] = pk;
  }
  float* __restrict__ rx = reg;
  float* __restrict__ ry = reg + cap;
  float* __restrict__ rz = reg + 2 * cap;
  for (int c = wid; c < m; c += 8) {
    const int b = sstart[c], o = soff[c], k1 = scnt[c], k2 = (k1 + 3) & ~3;
    for (int k = lane; k < k2; k += 32) {
      const float inf = __int_as_float(0x7f800000);
      float4 p = make_float4(inf, inf, inf, 0.f);
      if (k < k1) p = pos_s[b + k];
      rx[o + k] = p.x;
      ry[o + k] = p.y;
      rz[o + k] = p.z;
    }
  }
  if (tid < m) tcells[tile * (kTileCells + 1) + tid] = make_int2(sstart[tid], soff[tid] | (scnt[tid] << 16));
  if (tid == 0) {
    tcells[tile * (kTileCells + 1) + m] = make_int2(0, nreg);
    tncell[tile] = m;
  }
  __syncthreads();
  // the rows
  const int row = tid / LPR, sub = tid % LPR;
  const int64_t s = row0 + row;
  const int rl = row & 31;
  int count = 0;
  const bool live = s < n;
  {
    const float4 ps = live ? pos_s[s] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int* __restrict__ cells = hd + (live ? rcnt[row] : 0) * 27;
    uint16_t* __restrict__ list = raw + (s / kSlice) * (int64_t)(kSlice * maxnb) + rl;
    const f2 nx2 = f2_pack(-ps.x, -ps.x), ny2 = f2_pack(-ps.y, -ps.y), nz2 = f2_pack(-ps.z, -ps.z);
    const float lo2 = band.lo2, hi2 = band.hi2;
    const int selfk = live ? (int)(s - cell_start[rank[key_s[s]]]) : 0;   // the row's place in its cell
    f2 il[3], nl[3];
    bool per[3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      per[ax] = PER && g.periodic[ax];
      il[ax] = f2_pack(band.invL[ax], band.invL[ax]);
      nl[ax] = f2_pack(-band.L[ax], -band.L[ax]);
    }
    // the nearest whole number by adding and taking off 1.5 x 2^23 (exact below 2^22;
    // beyond, the band covers every distance and the float64 test decides)
    const f2 mg = f2_pack(12582912.f, 12582912.f), nmg = f2_pack(-12582912.f, -12582912.f);
    for (int o = 0; o < 27; ++o) {
      const int pk = live ? cells[o] : 0;
      const int b = pk & 0xffff, groups = ((pk >> 16) + 3) >> 2;
      const int rounds = LPR == 1 ? groups : (groups + LPR - 1) / LPR;
      for (int r = 0; r < rounds; ++r) {
        const int at = b + 4 * (r * LPR + sub);
        unsigned hit = 0;
        if (LPR == 1 || r * LPR + sub < groups) {
          const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(rx + at);
          const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(ry + at);
          const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(rz + at);
          float q[4];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            f2 d0 = f2_add(h ? X.y : X.x, nx2), d1 = f2_add(h ? Y.y : Y.x, ny2), d2 = f2_add(h ? Z.y : Z.x, nz2);
            if (per[0]) d0 = f2_fma(nl[0], f2_add(f2_add(f2_mul(d0, il[0]), mg), nmg), d0);
            if (per[1]) d1 = f2_fma(nl[1], f2_add(f2_add(f2_mul(d1, il[1]), mg), nmg), d1);
            if (per[2]) d2 = f2_fma(nl[2], f2_add(f2_add(f2_mul(d2, il[2]), mg), nmg), d2);
            f2_unpack(f2_fma(d2, d2, f2_fma(d1, d1, f2_mul(d0, d0))), q[2 * h], q[2 * h + 1]);
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) hit |= q[k] < lo2 ? 1u << k : 0u;
          unsigned near = 0;
#pragma unroll
          for (int k = 0; k < 4; ++k) near |= q[k] < hi2 ? 1u << k : 0u;
          near ^= hit;
          while (near) {   // inside the band: as the float64 definition
            const int k = __ffs(near) - 1;
            near &= near - 1;
            if (pair_inside_f64(make_float4(rx[at + k], ry[at + k], rz[at + k], 0.f), ps, g, band.R2)) hit |= 1u << k;
          }
          if (o == 13) {   // the own cell holds the row itself
            const int self = b + selfk - at;
            if (self >= 0 && self < 4) hit &= ~(1u << self);
          }
        }
        int put = count;
        if (LPR == 1) {
          count += __popc(hit);
        } else {
          const unsigned grp = ((1u << LPR) - 1u) << (lane & ~(LPR - 1));
          const int own = __popc(hit);
          int inc = own;
#pragma unroll
          for (int d = 1; d < LPR; d <<= 1) {
            const int x = __shfl_up_sync(grp, inc, d, LPR);
            if (sub >= d) inc += x;
          }
          put += inc - own;
          count += __shfl_sync(grp, inc, LPR - 1, LPR);
        }
        while (hit) {
          const int k = __ffs(hit) - 1;
          hit &= hit - 1;
          if (put < maxnb) list[put * kSlice] = (uint16_t)(at + k);
          ++put;
        }
      }
    }
    if (live && count > maxnb) {
      if (sub == 0) atomicOr(&flags[0], FLAG_CAPACITY);
      count = maxnb;
    }
  }
  __syncthreads();
  if (sub == 0) rcnt[row] = count;
  __syncthreads();
  if (wid < TS && (row0 >> 5) + wid < nslices) {
    const int c = rcnt[wid * 32 + lane];
    cnt[row0 + wid * 32 + lane] = c;
    int mx = c;
    unsigned sum = (unsigned)c;
    for (int o = 16; o > 0; o >>= 1) {
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (lane == 0) {
      width[(row0 >> 5) + wid] = (mx + 3) & ~3;
      atomicAdd(total, (unsigned long long)sum);
      atomicMax(maxc, mx);
    }
  }
}

// Eight small counters in registers: 8 bits each where a row has at most 255 entries,
// 16 bits each otherwise.
template <bool WIDE>
struct Fields;
template <>
struct Fields<false> {
  unsigned long long v = 0;
  __device__ __forceinline__ int get(int b) const { return (int)(v >> (8 * b)) & 0xff; }
  __device__ __forceinline__ void add(int b, int x) { v += (unsigned long long)x << (8 * b); }
};
template <>
struct Fields<true> {
  unsigned long long a = 0, c = 0;
  __device__ __forceinline__ int get(int b) const { return (int)((b < 4 ? a : c) >> (16 * (b & 3))) & 0xffff; }
  __device__ __forceinline__ void add(int b, int x) {
    const unsigned long long y = (unsigned long long)x << (16 * (b & 3));
    if (b < 4) a += y;
    else c += y;
  }
};

// The union of a tile and its rows' entries as positions in it (tiles.cuh).  The
// region's particles that some row references are marked, the marks are turned
// into positions by ballots and a prefix sum, and one thread per row sorts its
// entries into the 8 bank groups (position mod 8) and takes them out again so that
// lane l takes group (l + j - 2) mod 8 at step j while that group lasts, then the
// fullest one.  Wall rows: fluid neighbours first, then, at the next multiple of
// four entries, the wall neighbours; nfl counts the former.
template <int TS, bool WIDE>
__global__ void __launch_bounds__(256) k_tile_plan(const uint8_t* __restrict__ type_s, const int32_t* __restrict__ cnt,
                                                   int64_t n, int64_t nslices, const uint16_t* __restrict__ raw,
                                                   uint16_t* __restrict__ idx, int64_t istride,
                                                   const int2* __restrict__ tcells,
                                                   const int32_t* __restrict__ tncell, int cap, int32_t maxnb,
                                                   int32_t* __restrict__ nfl, int32_t* __restrict__ uni,
                                                   int32_t ustride, int32_t* __restrict__ unum,
                                                   int32_t* __restrict__ flags) {
  constexpr int R = 32 * TS, S = 8 / TS;
  extern __shared__ __align__(16) uint16_t dyn[];
  uint16_t* list = dyn;                                        // [maxnb][R]
  uint16_t* map = list + (size_t)maxnb * R;                    // [cap]: place | kRef | kWall
  constexpr unsigned kRef = 0x4000u, kWall = 0x8000u;
  __shared__ int wpre[256];
  __shared__ int wsum[8];
  if (build_stopped(flags, maxnb) || (flags[0] & (FLAG_REGION | FLAG_UNEVEN | FLAG_CAPACITY)) != 0) return;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t tile = blockIdx.x, row0 = tile * R;
  const int2* __restrict__ cells = tcells + tile * (kTileCells + 1);
  const int m = tncell[tile], nreg = cells[m].y;
  for (int c = wid; c < m; c += 8) {
    const int2 a = cells[c];
    const int off = a.y & 0xffff, many = a.y >> 16, padded = (many + 3) & ~3;
    for (int k = lane; k < padded; k += 32)
      map[off + k] = k < many && type_s[a.x + k] != SPH_FLUID ? kWall : 0;
  }
  __syncthreads();
  const int row = tid % R, split = tid / R, rl = row & 31;
  const int64_t s = row0 + row;
  const bool live = s < n;
  const int c = live ? cnt[s] : 0;
  const uint16_t* __restrict__ mine = raw + (s / kSlice) * (int64_t)(kSlice * maxnb) + rl;
#pragma unroll 4
  for (int j = split; j < c; j += S) map[mine[j * kSlice]] |= kRef;
  __syncthreads();
  // positions: word w covers region places 32 w .. 32 w + 31
  const int words = (nreg + 31) >> 5;
  for (int w = wid; w < words; w += 8) {
    const int p = w * 32 + lane;
    const unsigned f = p < nreg ? map[p] : 0u;
    const unsigned bl = __ballot_sync(0xffffffffu, (f & kRef) != 0);
    if (lane == 0) wpre[w] = __popc(bl);
    if (p < nreg) map[p] = (uint16_t)(f | __popc(bl & ((1u << lane) - 1u)));
  }
  __syncthreads();
  {
    const int v = tid < words ? wpre[tid] : 0;
    int inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    int pre = 0, all = 0;
    for (int w = 0; w < 8; ++w) {
      if (w < wid) pre += wsum[w];
      all += wsum[w];
    }
    if (tid < words) wpre[tid] = pre + inc - v;
    if (tid == 0) {
      unum[tile] = all;
      atomicMax(&flags[3], all);
    }
  }
  __syncthreads();
  // map: union position, kWall on walls (positions stay below 4,096)
  for (int q = wid; q < m; q += 8) {
    const int2 a = cells[q];
    const int off = a.y & 0xffff, many = a.y >> 16;
    for (int k = lane; k < many; k += 32) {
      const int p = off + k;
      const unsigned f = map[p];
      const int u = (int)(f & 31u) + wpre[p >> 5];
      map[p] = (uint16_t)(u | (f & kWall));
      if ((f & kRef) && u < ustride) uni[tile * ustride + u] = a.x + k;
    }
  }
  __syncthreads();
  if (split > 0 || s >= nslices * kSlice) return;
  const bool fluid = live && type_s[s] == SPH_FLUID;
  const unsigned skip = fluid ? 0u : kWall;   // entries left out of the interleaving
  Fields<WIDE> left, cur;
  int nf = 0;
#pragma unroll 4
  for (int j = 0; j < c; ++j) {
    const unsigned u = map[mine[j * kSlice]];
    if (!(u & skip)) {
      left.add(u & 7, 1);
      ++nf;
    }
  }
  int run = 0;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    cur.add(b, run);
    run += left.get(b);
  }
  Fields<WIDE> to = cur;
  int rest = nf;
#pragma unroll 4
  for (int j = 0; j < c; ++j) {
    const unsigned u = map[mine[j * kSlice]];
    int at;
    if (!(u & skip)) {
      at = to.get(u & 7);
      to.add(u & 7, 1);
    } else {
      at = rest++;
    }
    list[at * R + row] = (uint16_t)((u & 0xfffu) << 4);
  }
  uint16_t* __restrict__ out = idx + (s / kSlice) * istride;
  unsigned fill = 0;
  for (int j0 = 0; j0 < nf; j0 += 4) {
    unsigned v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = fill;
      if (j0 + k < nf) {
        int b = (rl + k + j0 + 6) & 7;
        if (left.get(b) == 0) {
          int most = 0;
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            const int many = left.get(x);
            if (many > most) {
              most = many;
              b = x;
            }
          }
        }
        v[k] = list[cur.get(b) * R + row];
        cur.add(b, 1);
        left.add(b, -1);
        if (j0 + k == 0) fill = v[k];
      }
    }
    *reinterpret_cast<uint2*>(out + (j0 >> 2) * 128 + rl * 4) = make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
  }
  const int base = (nf + 3) & ~3;
  for (int j = nf; j < c; ++j) out[tile_entry(base + j - nf, rl)] = list[j * R + row];
  nfl[s] = nf;
}

// The lists as 32-bit rows in the fixed-capacity SELL-32 layout of k_neighbors and in its
// order, from the search's region places (raw has that layout and order), so that what
// sums along them does not depend on how the lists were made.  The plan's entries are
// ordered for shared-memory banks; rows expanded from those cost the export's sort most
// (rebuild and export of 77k rows of ~250: 7.69 ms against 6.50, 12k: 3.43 against 2.97)
// and the on-the-fly apply a little (rebuild and apply, 58k rows: 352 against 336 us),
// while applies along stored 32-bit rows are 4% faster on them (58k: 44.5 against 45.9 us
// an iteration).  One block per tile: the region's rows into shared memory, then
// one coalesced pass over the entries.
__global__ void __launch_bounds__(256) k_tile_expand(const uint16_t* __restrict__ raw, const int2* __restrict__ tcells,
                                                     const int32_t* __restrict__ tncell, const int32_t* __restrict__ cnt,
                                                     int slices_per_tile, int64_t nslices, int64_t n, int32_t maxnb,
                                                     int32_t* __restrict__ nbr) {
  extern __shared__ int32_t place[];   // region place -> row
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t tile = blockIdx.x;
  const int2* __restrict__ cells = tcells + tile * (kTileCells + 1);
  const int m = tncell[tile];
  for (int q = wid; q < m; q += 8) {
    const int2 a = cells[q];
    for (int k = lane; k < a.y >> 16; k += 32) place[(a.y & 0xffff) + k] = a.x + k;
  }
  __syncthreads();
  const int64_t sl1 = min((tile + 1) * slices_per_tile, nslices);
  for (int64_t sl = tile * slices_per_tile; sl < sl1; ++sl) {
    const int64_t s = sl * kSlice + lane, base = sl * kSlice * (int64_t)maxnb + lane;
    const int c = s < n ? cnt[s] : 0, most = __reduce_max_sync(0xffffffffu, c);
#pragma unroll 4
    for (int j = wid; j < most; j += 8)
      if (j < c) nbr[base + (int64_t)j * kSlice] = place[raw[base + (int64_t)j * kSlice]];
  }
}

// slice offsets of the fixed-capacity list layout
__global__ void k_fixed_offsets(int64_t nslices, int64_t width, int64_t* __restrict__ off) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k <= nslices; k += (int64_t)gridDim.x * blockDim.x)
    off[k] = k * kSlice * width;
}

// slice widths (max count over the 32 rows), total entries and the largest row
__global__ void k_slice_width(const int32_t* __restrict__ cnt, int64_t nslices, int32_t* __restrict__ width,
                              unsigned long long* __restrict__ total, int32_t* __restrict__ maxc) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = warp; k < nslices; k += nwarps) {
    int c = cnt[k * kSlice + lane];
    int m = c;
    unsigned long long sum = (unsigned long long)c;
    for (int o = 16; o > 0; o >>= 1) {
      m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (lane == 0) {
      width[k] = m;
      atomicAdd(total, sum);
      atomicMax(maxc, m);
    }
  }
}

// caller-order CSR export: row lengths, then entries mapped through perm and sorted
__global__ void k_export_counts(const int32_t* __restrict__ iperm, const int32_t* __restrict__ cnt, int64_t n,
                                int32_t* __restrict__ rowlen) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    rowlen[i] = cnt[iperm[i]];
}

__global__ void k_export_fill(const int32_t* __restrict__ iperm, const int32_t* __restrict__ perm,
                              const int32_t* __restrict__ cnt, const int64_t* __restrict__ slice_off,
                              const int32_t* __restrict__ nbr, int64_t n, const int64_t* __restrict__ offsets,
                              int32_t* __restrict__ idx) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = iperm[i];
    const int32_t c = cnt[s];
    const int64_t base = slice_off[s / kSlice] + (s % kSlice);
    int32_t* row = idx + offsets[i];
    for (int32_t j = 0; j < c; ++j) {
      int32_t v = perm[nbr[base + (int64_t)j * kSlice]];
      int32_t k = j - 1;
      while (k >= 0 && row[k] > v) {
        row[k + 1] = row[k];
        --k;
      }
      row[k + 1] = v;
    }
  }
}

}  // namespace

// rank[row-major cell] = position of the cell along the Morton curve that
// interleaves the bits of its (x, y, z) cell coordinates (ties impossible); grids
// of more than 2^24 cells keep the row-major order (the host table and its sort
// would cost more than the locality gains)
static void morton_ranks(const int nc[3], std::vector<int32_t>& rank) {
  auto spread = [](uint64_t v) {
    uint64_t r = 0;
    for (int b = 0; b < 21; ++b) r |= ((v >> b) & 1ull) << (3 * b);
    return r;
  };
  const int64_t ncells = (int64_t)nc[0] * nc[1] * nc[2];
  rank.assign((size_t)ncells, 0);
  if (ncells > ((int64_t)1 << 24)) {
    for (int64_t c = 0; c < ncells; ++c) rank[(size_t)c] = (int32_t)c;
    return;
  }
  std::vector<std::pair<uint64_t, int32_t>> code((size_t)ncells);
  for (int z = 0; z < nc[2]; ++z)
    for (int y = 0; y < nc[1]; ++y)
      for (int x = 0; x < nc[0]; ++x) {
        const int64_t c = x + (int64_t)nc[0] * (y + (int64_t)nc[1] * z);
        code[(size_t)c] = {spread((uint64_t)x) | (spread((uint64_t)y) << 1) | (spread((uint64_t)z) << 2), (int32_t)c};
      }
  std::sort(code.begin(), code.end());
  for (int64_t r = 0; r < ncells; ++r) rank[(size_t)code[(size_t)r].second] = (int32_t)r;
}

int grid_for(const sph_neighbors* H, int64_t work_items, int block) {
  int64_t want = (work_items + block - 1) / block;
  int64_t cap = (int64_t)(H->num_sms > 0 ? H->num_sms : 148) * 16;
  if (want > cap) want = cap;
  if (want < 1) want = 1;
  return (int)want;
}

// exclusive scan of m values times mul; one block up to 8,192 values (2 tiles: the
// second launch would cost more than it saves), the tiled kernels above that, and one
// block again beyond 2^25, where a block's walk over the earlier tile sums is long
template <class TOut>
static sph_status scan(sph_neighbors* H, const int32_t* in, TOut* out, int64_t m, int64_t mul, int32_t* max_out,
                       cudaStream_t st) {
  if (m <= 2 * kScanTile || m > ((int64_t)1 << 25)) {
    SPH_LAUNCH(k_scan<TOut>, 1, 1024, 0, st)(in, out, m, mul, max_out);
  } else {
    const int nt = (int)((m + kScanTile - 1) / kScanTile);
    SPH_TRY(H->scan_sums.alloc(nt));
    SPH_LAUNCH(k_scan_sums, nt, 1024, 0, st)(in, m, H->scan_sums.p, max_out);
    SPH_LAUNCH(k_scan_tiles<TOut>, nt, 1024, 0, st)(in, out, m, mul, H->scan_sums.p);
  }
  SPH_TRY_CUDA(cudaGetLastError());
  return SPH_OK;
}

// Builds slice widths + offsets for a per-row count array; returns the padded
// entry total, the true entry total and the largest row (synchronises).
sph_status build_slices(sph_neighbors* H, const int32_t* cnt, int64_t* off, int64_t* total_pad,
                        int64_t* total, int32_t* maxc, cudaStream_t st) {
  SPH_TRY(H->tmp_i32b.alloc(H->nslices + 1));
  SPH_TRY(H->tmp_i64.alloc(4));
  SPH_TRY_CUDA(cudaMemsetAsync(H->tmp_i64.p, 0, 4 * sizeof(int64_t), st));
  int grid = grid_for(H, H->nslices * 32);
  SPH_LAUNCH(k_slice_width, grid, kBlock, 0, st)(cnt, H->nslices, H->tmp_i32b.p,
                                         reinterpret_cast<unsigned long long*>(H->tmp_i64.p),
                                         reinterpret_cast<int32_t*>(H->tmp_i64.p + 1));
  SPH_TRY_CUDA(cudaGetLastError());
  SPH_TRY(scan<int64_t>(H, H->tmp_i32b.p, off, H->nslices, kSlice, nullptr, st));
  int64_t host[2];
  SPH_TRY_CUDA(cudaMemcpyAsync(host, H->tmp_i64.p, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SPH_TRY_CUDA(cudaMemcpyAsync(total_pad, off + H->nslices, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SPH_TRY_CUDA(cudaStreamSynchronize(st));
  *total = host[0];
  *maxc = (int32_t)(host[1] & 0xffffffff);
  return SPH_OK;
}

// places in shared memory for a tile's search region, tried in turn: 256-row tiles of the
// box need up to ~3,100 (2,757 particles and the cells' padding), the Gaussian's narrow
// channels ~3,600, h = 2.5 dp 6,656.  With the first and 128 entries a row three blocks of
// the plan fit an SM (72.7 KB each; two with 4,608 places); above 160 entries a row it
// changes nothing and the second comes first.  A handle starts with the size that its
// last rebuild needed (a smaller one only where that leaves a sixteenth free, so that a
// need that moves about a limit is not searched twice).  A set that no tiles hold is
// searched globally at once by its next kUntiledRebuilds rebuilds: a dense block under a
// spray, 54k rows, takes 257 us a rebuild; with failed tile searches each time 634.
constexpr int kRegions[] = {3584, 4608, 7168};
constexpr int kRegionSizes = 3;
constexpr int kRegionLarge = kRegions[kRegionSizes - 1];
constexpr int kUntiledRebuilds = 32;

// the smallest size class from `least` on with `need` places, kRegionSizes if there is none
static int region_class(int need, int least) {
  int k = least;
  while (k < kRegionSizes && kRegions[k] < need) ++k;
  return k;
}

// Slices per tile.  Large tiles share more of their neighbours (4.4 union rows per row
// at 8 slices, 5.8 at 4, 7.8 at 2 on the box); small ones give a small set more blocks
// and a row more threads.  Whole passes (rebuild, start, solve to 1e-8) at 8 / 4 / 2 / 1
// slices, us, all on the cooperative kernel (persist.cu) where it takes them:
//   rows of ~80    2.2k  1124 /  949 /  896 /  921      rows of ~250
//                  2.7k  1142 / 1025 / 1010 /  935         3.1k 1487 / 1210 / 1068 / 1034
//                  6.8k  1626 / 1441 / 1584 / 1499        11.5k 2449 / 1999 / 1880 / 1916
//                   16k  2142 / 2093 / 2153 / 2117        34.7k 3633 / 3449 / 4219 / 4602
//                   30k  3160 / 3062 / 3103 / 3345        77.4k 6858 / 7886 / 8528 / 8371
//                   51k  4173 / 4268 / 4221 / 5721
//                   59k  4044 / 4195 / 4587 / 6004
//                   79k  6176 / 6265 / 7150
//                   97k  6507 / 7636 / 7642
// (iteration counts differ by up to 5% with the sums' order, which is part of these).  One
// slice where that gives fewer tiles than SMs (twice as many with rows of ~250), 2 up to
// 600 slices, 4 up to 1,800, then 8: of the columns above the fastest or within 3% of it,
// but at 6.8k rows 10% behind 4 slices.  Applies of the five-kernel loop, 8 / 4 / 2: 64k rows
// 17.3 / 16.5 / 18.0 us, 274k 37.5 / 37.5 / 41.4, 1,157k 128 / 138 / 161; the Gaussian's
// unions are larger: 190k rows 67.8 / 53.6 / 56.4, hence 4 slices again beyond what the
// cooperative kernel holds (18 slices per SM).
// Beyond 320 (640) entries per row the lists of 8 (4) slices exceed the plan's shared
// memory.
static int tile_slices_for(int64_t nslices, int32_t maxnb, int num_sms) {
  if (nslices < (maxnb > 160 ? 2 : 1) * (int64_t)num_sms) return 1;
  if (nslices < 600 || maxnb > 640) return 2;
  if (nslices < 1800 || maxnb > 320) return 4;
  return maxnb > 160 && nslices > 18 * (int64_t)num_sms ? 4 : 8;
}

static sph_status fixed_offsets(sph_neighbors* H, cudaStream_t st) {
  SPH_TRY(H->slice_off.alloc(H->nslices + 1));
  SPH_LAUNCH(k_fixed_offsets, grid_for(H, H->nslices + 1), kBlock, 0, st)(H->nslices, H->maxnb, H->slice_off.p);
  SPH_TRY_CUDA(cudaGetLastError());
  return SPH_OK;
}

sph_status require_lists(const sph_neighbors* H) {
  if (H->lists_ok) return SPH_OK;
  set_error("the last sph_build_neighbors on this handle failed: it has no neighbour lists until a build succeeds");
  return SPH_ERR_INVALID;
}

bool stream_capturing(cudaStream_t st) {
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &s) == cudaSuccess) return s != cudaStreamCaptureStatusNone;
  (void)cudaGetLastError();   // (the legacy stream while another one captures: what follows fails by itself)
  return false;
}

sph_status ensure_nbr(sph_neighbors* H, cudaStream_t st) {
  SPH_TRY(require_lists(H));
  if (H->nbr_ready) return SPH_OK;
  const bool capturing = stream_capturing(st);
  if (H->nbr_valid && !capturing) {   // expanded by an earlier call, on whatever stream
    if (cudaEventQuery(H->nbr_event) == cudaSuccess) {
      H->nbr_ready = true;
      return SPH_OK;
    }
    (void)cudaGetLastError();   // cudaErrorNotReady is no failure of the next launch
    SPH_TRY_CUDA(cudaStreamWaitEvent(st, H->nbr_event, 0));
    return SPH_OK;
  }
  SPH_TRY(H->nbr.alloc(H->n_pad * (int64_t)H->maxnb));
  SPH_TRY(fixed_offsets(H, st));
  SPH_LAUNCH(k_tile_expand, (int)H->ntiles, 256, H->tile_cap * sizeof(int32_t), st)(
      H->t_raw.p, H->t_cells.p, H->t_ncell.p, H->cnt.p, H->tile_ts, H->nslices, H->n, H->maxnb, H->nbr.p);
  SPH_TRY_CUDA(cudaGetLastError());
  if (capturing) return SPH_OK;
  if (!H->nbr_event) SPH_TRY_CUDA(cudaEventCreateWithFlags(&H->nbr_event, cudaEventDisableTiming));
  SPH_TRY_CUDA(cudaEventRecord(H->nbr_event, st));
  H->nbr_valid = true;
  return SPH_OK;
}

template <int TS>
static sph_status launch_search_ts(sph_neighbors* H, const Grid& g, const BandIn& bin, int32_t maxnb, int cap,
                                   cudaStream_t st) {
  const size_t smem = (size_t)cap * 3 * sizeof(float);
  const size_t plan = (size_t)maxnb * 32 * TS * sizeof(uint16_t) + (size_t)cap * sizeof(uint16_t);
  const bool per = g.periodic[0] || g.periodic[1] || g.periodic[2];
  auto search = per ? k_tile_search<TS, true> : k_tile_search<TS, false>;
  auto planner = maxnb > 255 ? k_tile_plan<TS, true> : k_tile_plan<TS, false>;
  SPH_TRY_CUDA(cudaFuncSetAttribute((const void*)search, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kRegionLarge * 3 * (int)sizeof(float)));
  SPH_TRY_CUDA(cudaFuncSetAttribute((const void*)planner, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  SPH_LAUNCH(search, (int)H->ntiles, 256, smem, st)(
      H->pos_s.p, H->key_s.p, H->cell_rank.p, H->cell_start.p, H->n, H->nslices, g, bin, maxnb, cap, H->cnt.p, H->t_raw.p,
      H->t_cells.p, H->t_ncell.p, H->tmp_i32b.p, reinterpret_cast<unsigned long long*>(H->tmp_i64.p),
      reinterpret_cast<int32_t*>(H->tmp_i64.p + 1), H->flags.p);
  SPH_TRY_CUDA(cudaGetLastError());
  SPH_LAUNCH(planner, (int)H->ntiles, 256, plan, st)(H->type_s.p, H->cnt.p, H->n, H->nslices, H->t_raw.p, H->t_idx.p,
                                                     H->t_istride, H->t_cells.p, H->t_ncell.p, cap, maxnb, H->t_nfl.p,
                                                     H->t_uni.p, H->t_ustride, H->t_unum.p, H->flags.p);
  SPH_TRY_CUDA(cudaGetLastError());
  return SPH_OK;
}

// search and plan of every tile, and the coefficient offsets of the slices
static sph_status launch_tile_search(sph_neighbors* H, const Grid& g, const BandIn& bin, int32_t maxnb, int cap,
                                     cudaStream_t st) {
  const int ts = tile_slices_for(H->nslices, maxnb, H->num_sms);
  H->tile_ts = ts;
  H->tile_cap = cap;
  H->ntiles = (H->nslices + ts - 1) / ts;
  H->t_istride = 32 * (((maxnb + 3) & ~3) + 4);
  H->t_ustride = cap < kTileUnion + 1 ? cap : kTileUnion + 1;
  SPH_TRY(H->t_idx.alloc(H->nslices * H->t_istride));
  SPH_TRY(H->t_raw.alloc(H->nslices * kSlice * (int64_t)maxnb));
  SPH_TRY(H->t_cells.alloc(H->ntiles * (kTileCells + 1)));
  SPH_TRY(H->t_ncell.alloc(H->ntiles));
  SPH_TRY(H->t_nfl.alloc(H->n_pad));
  SPH_TRY(H->t_uni.alloc(H->ntiles * H->t_ustride));
  SPH_TRY(H->t_unum.alloc(H->ntiles));
  SPH_TRY(H->t_off.alloc(H->nslices + 1));
  SPH_TRY_CUDA(cudaMemsetAsync(H->tmp_i32b.p, 0, H->nslices * sizeof(int32_t), st));
  if (ts == 8) SPH_TRY(launch_search_ts<8>(H, g, bin, maxnb, cap, st));
  else if (ts == 4) SPH_TRY(launch_search_ts<4>(H, g, bin, maxnb, cap, st));
  else if (ts == 2) SPH_TRY(launch_search_ts<2>(H, g, bin, maxnb, cap, st));
  else SPH_TRY(launch_search_ts<1>(H, g, bin, maxnb, cap, st));
  return scan<int64_t>(H, H->tmp_i32b.p, H->t_off.p, H->nslices, kSlice, nullptr, st);
}

sph_status build_neighbors(const sph_scene* sc, int32_t maxnb, sph_neighbors** out, cudaStream_t st) {
  if (!sc || !out) {
    set_error("sph_build_neighbors: null scene or handle pointer");
    return SPH_ERR_INVALID;
  }
  if (sc->n < 1 || sc->n > (int64_t)INT32_MAX - 64 || !sc->pos || !sc->rho || !sc->mu || !sc->ptype) {
    set_error("sph_build_neighbors: n must be in [1, 2^31-64] and every array non-null");
    return SPH_ERR_INVALID;
  }
  if (!(sc->h > 0.f) || !std::isfinite(sc->h)) {
    set_error("sph_build_neighbors: h must be positive and finite");
    return SPH_ERR_INVALID;
  }
  if (maxnb < 1 || maxnb > 1024) {
    set_error("sph_build_neighbors: max_neighbors must be in [1, 1024]");
    return SPH_ERR_INVALID;
  }
  if (sc->kernel != SPH_KERNEL_WENDLAND && sc->kernel != SPH_KERNEL_GAUSSIAN) {
    set_error("sph_build_neighbors: unknown kernel %d", sc->kernel);
    return SPH_ERR_INVALID;
  }
  Grid g{};
  // the support radius: 2h (Wendland) or 3h (truncated Gaussian)
  const double rsup = (sc->kernel == SPH_KERNEL_GAUSSIAN ? 3.0 : 2.0) * (double)sc->h;
  int64_t ncells = 1;
  for (int ax = 0; ax < 3; ++ax) {
    double L = sc->hi[ax] - sc->lo[ax];
    if (!(L > 0.0) || !std::isfinite(L)) {
      set_error("sph_build_neighbors: hi[%d] must exceed lo[%d]", ax, ax);
      return SPH_ERR_INVALID;
    }
    // cells strictly larger than the support radius (with a relative margin for rounding)
    double nc = std::floor(L / (rsup * (1.0 + 1e-6)));
    if (nc < 1.0) nc = 1.0;
    if (nc > 1.0e6) nc = 1.0e6;
    g.periodic[ax] = sc->periodic[ax] ? 1 : 0;
    if (g.periodic[ax] && nc < 3.0) {
      set_error("sph_build_neighbors: periodic axis %d is shorter than three cells of the support radius "
                "(L = %g, radius = %g)", ax, L, rsup);
      return SPH_ERR_INVALID;
    }
    g.ncell[ax] = (int)nc;
    g.cell[ax] = L / nc;
    g.lo[ax] = sc->lo[ax];
    g.L[ax] = L;
    ncells *= (int64_t)nc;
  }
  if (ncells > (int64_t)1 << 30) {
    set_error("sph_build_neighbors: %lld cells exceed the 2^30 limit (box too large for h)", (long long)ncells);
    return SPH_ERR_INVALID;
  }
  g.ncells = ncells;

  bool fresh = (*out == nullptr);
  sph_neighbors* H = fresh ? new sph_neighbors() : *out;
  auto fail = [&](sph_status s) {
    if (fresh) {
      sph_neighbors_destroy(H);
      *out = nullptr;
    }
    return s;
  };
#define TRYF(expr)                      \
  do {                                  \
    sph_status s__ = (expr);            \
    if (s__ != SPH_OK) return fail(s__); \
  } while (0)
#define TRYF_CUDA(call)                                                                         \
  do {                                                                                          \
    cudaError_t e__ = (call);                                                                   \
    if (e__ != cudaSuccess) {                                                                   \
      set_error("%s:%d %s: %s", __FILE__, __LINE__, #call, cudaGetErrorString(e__));           \
      return fail(SPH_ERR_CUDA);                                                                \
    }                                                                                           \
  } while (0)

  TRYF_CUDA(cudaGetDevice(&H->device));
  TRYF_CUDA(cudaDeviceGetAttribute(&H->num_sms, cudaDevAttrMultiProcessorCount, H->device));
  const int64_t n = sc->n;
  const bool same_shape = H->n == n && H->h == sc->h && H->kernel == sc->kernel && H->maxnb == maxnb &&
                          std::equal(g.ncell, g.ncell + 3, H->grid.ncell);
  H->lists_ok = false;
  ++H->list_version;
  if (H->row_scaled && H->n != n) {   // a caller-order row scale no longer fits
    H->row_scaled = false;
    ++H->rs_version;
  }
  H->n = n;
  H->n_pad = (n + kSlice - 1) / kSlice * kSlice;
  H->nslices = H->n_pad / kSlice;
  H->grid = g;
  H->h = sc->h;
  H->kernel = sc->kernel;
  H->op_valid = H->op_tile_valid = H->op_ih_valid = false;
  H->mu_version++;

  TRYF(H->pos_s.alloc(H->n_pad));
  TRYF(H->rho_s.alloc(H->n_pad));
  TRYF(H->mu_s.alloc(H->n_pad));
  TRYF(H->type_s.alloc(H->n_pad));
  TRYF(H->perm.alloc(n));
  TRYF(H->iperm.alloc(n));
  TRYF(H->key_s.alloc(H->n_pad));
  TRYF(H->cell_start.alloc(ncells + 1));
  TRYF(H->cnt.alloc(H->n_pad));
  TRYF(H->tmp_i32a.alloc(n));                                 // keys
  TRYF(H->tmp_ids.alloc(n));                                  // particles by cell, unordered
  TRYF(H->tmp_i64.alloc(4));
  TRYF(H->flags.alloc(8));
  TRYF(H->tmp_i32b.alloc(ncells > H->nslices + 1 ? ncells : H->nslices + 1));
  TRYF_CUDA(cudaMemsetAsync(H->flags.p, 0, 8 * sizeof(int32_t), st));
  TRYF_CUDA(cudaMemsetAsync(H->tmp_i32b.p, 0, ncells * sizeof(int32_t), st));

  const float4* pos = reinterpret_cast<const float4*>(sc->pos);
  int32_t* key = H->tmp_i32a.p;
  int grid_n = grid_for(H, n);
  if (H->rank_dims[0] != g.ncell[0] || H->rank_dims[1] != g.ncell[1] || H->rank_dims[2] != g.ncell[2]) {
    TRYF(H->cell_rank.alloc(ncells));
    std::vector<int32_t> rank;
    morton_ranks(g.ncell, rank);
    TRYF_CUDA(cudaMemcpy(H->cell_rank.p, rank.data(), ncells * sizeof(int32_t), cudaMemcpyHostToDevice));
    for (int ax = 0; ax < 3; ++ax) H->rank_dims[ax] = g.ncell[ax];
  }
  SPH_LAUNCH(k_cell_keys, grid_n, kBlock, 0, st)(pos, n, g, H->cell_rank.p, key, H->tmp_i32b.p, H->flags.p,
                                         reinterpret_cast<unsigned int*>(H->flags.p + 1));
  TRYF_CUDA(cudaGetLastError());
  TRYF(scan<int32_t>(H, H->tmp_i32b.p, H->cell_start.p, ncells, 1, H->flags.p + 2, st));
  // scatter into segments (cursor counts reuse tmp_i32b), then sort and copy
  TRYF_CUDA(cudaMemsetAsync(H->tmp_i32b.p, 0, ncells * sizeof(int32_t), st));
  SPH_LAUNCH(k_cell_scatter, grid_n, kBlock, 0, st)(key, H->cell_rank.p, n, H->cell_start.p, H->tmp_i32b.p,
                                                    H->tmp_ids.p);
  SPH_LAUNCH(k_cell_sort, grid_for(H, H->n_pad), kBlock, 0, st)(
      H->tmp_ids.p, H->cell_start.p, n, H->n_pad, maxnb, pos, sc->rho, sc->mu, sc->ptype, key, H->cell_rank.p,
      H->perm.p, H->iperm.p, H->pos_s.p, H->rho_s.p, H->mu_s.p, H->type_s.p, H->key_s.p, H->flags.p);
  TRYF_CUDA(cudaGetLastError());

  BandIn bin{};
  bin.rsup = rsup;
  for (int ax = 0; ax < 3; ++ax) {
    bin.big = std::fmax(bin.big, std::fabs(sc->lo[ax]));
    bin.big = std::fmax(bin.big, std::fabs(sc->hi[ax]));
    bin.big = std::fmax(bin.big, g.L[ax]);
    bin.L[ax] = (float)g.L[ax];
    bin.invL[ax] = (float)(1.0 / g.L[ax]);
  }

  H->maxnb = maxnb;
  H->nbr_valid = H->nbr_ready = false;
  H->tile_ok = false;
  int32_t hflags[8];
  int64_t tot[2], t_entries = 0;
  // the tile search with the region size that the last rebuild needed, once more with
  // the size that it turns out to need (h = 2.5 dp: 150 particles per cell), then the
  // global scan
  if (!same_shape) H->untiled = 0;
  const int least = maxnb > 160 ? 1 : 0;
  int round = H->untiled > 0 ? kRegionSizes : std::max(H->region, least);
  for (;;) {
    const bool tiles = round < kRegionSizes;
    TRYF_CUDA(cudaMemsetAsync(H->tmp_i64.p, 0, 2 * sizeof(int64_t), st));
    if (tiles) {
      TRYF(launch_tile_search(H, g, bin, maxnb, kRegions[round], st));
      TRYF_CUDA(cudaMemcpyAsync(&t_entries, H->t_off.p + H->nslices, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    } else {
      TRYF_CUDA(cudaMemcpyAsync(hflags, H->flags.p, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
      TRYF_CUDA(cudaStreamSynchronize(st));
      float max_abs;
      std::memcpy(&max_abs, &hflags[1], sizeof(float));
      TRYF(H->nbr.alloc(H->n_pad * (int64_t)maxnb));
      SPH_LAUNCH(k_neighbors, grid_for(H, H->n_pad), kBlock, 0, st)(H->pos_s.p, H->key_s.p, H->cell_rank.p,
                                                                    H->cell_start.p, n, H->n_pad, g,
                                                                    band_of(bin, max_abs), maxnb, H->cnt.p, H->nbr.p,
                                                                    H->flags.p);
      TRYF_CUDA(cudaGetLastError());
      TRYF(fixed_offsets(H, st));
      // entry total and the longest row (k_slice_width's widths land in scratch)
      SPH_LAUNCH(k_slice_width, grid_for(H, H->nslices * 32), kBlock, 0, st)(
          H->cnt.p, H->nslices, H->tmp_i32b.p, reinterpret_cast<unsigned long long*>(H->tmp_i64.p),
          reinterpret_cast<int32_t*>(H->tmp_i64.p + 1));
      TRYF_CUDA(cudaGetLastError());
    }
    TRYF_CUDA(cudaMemcpyAsync(hflags, H->flags.p, 8 * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    TRYF_CUDA(cudaMemcpyAsync(tot, H->tmp_i64.p, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    TRYF_CUDA(cudaStreamSynchronize(st));
    if (hflags[0] & FLAG_NONFINITE) {
      set_error("sph_build_neighbors: non-finite particle position or mass");
      return fail(SPH_ERR_NONFINITE);
    }
    if ((int64_t)hflags[2] > cell_limit(maxnb)) {
      set_error("sph_build_neighbors: a cell holds %d particles, more than any %d-neighbour particle set allows",
                hflags[2], maxnb);
      return fail(SPH_ERR_CAPACITY);
    }
    if (hflags[0] & FLAG_BADFIELD) {
      set_error("sph_build_neighbors: non-finite or non-positive density / viscosity");
      return fail(SPH_ERR_NONFINITE);
    }
    if (tiles && ((hflags[0] & (FLAG_REGION | FLAG_UNEVEN)) || hflags[3] > kTileUnion)) {
      TRYF_CUDA(cudaMemsetAsync(H->flags.p, 0, sizeof(int32_t), st));
      TRYF_CUDA(cudaMemsetAsync(H->flags.p + 3, 0, 2 * sizeof(int32_t), st));
      const bool larger = !(hflags[0] & FLAG_UNEVEN) && hflags[3] <= kTileUnion;   // whether that helps
      round = larger ? region_class(hflags[4], round + 1) : kRegionSizes;
      if (round == kRegionSizes) H->untiled = kUntiledRebuilds + 1;
      continue;
    }
    if (hflags[0] & FLAG_CAPACITY) {
      set_error("sph_build_neighbors: a particle has more than max_neighbors = %d neighbours", maxnb);
      return fail(SPH_ERR_CAPACITY);
    }
    H->tile_ok = tiles;
    H->nbr_valid = H->nbr_ready = !tiles;
    if (tiles) H->region = std::min(round, region_class(hflags[4] + hflags[4] / 16, 0));
    else --H->untiled;
    break;
  }
  H->tile_umax = hflags[3];
  H->t_entries = t_entries;
  const int64_t total = tot[0], total_pad = H->n_pad * (int64_t)maxnb;
  const int32_t maxc = (int32_t)(tot[1] & 0xffffffff);
  H->nnz = total;
  H->nnz_pad = total_pad;
  H->max_cnt = maxc;
  H->lists_ok = true;
  *out = H;
  return SPH_OK;
#undef TRYF
#undef TRYF_CUDA
}

sph_status export_neighbors(const sph_neighbors* H, int64_t* offsets, int32_t* idx, cudaStream_t st) {
  if (!H || !offsets || (!idx && H->nnz > 0)) {
    set_error("sph_neighbors_export: null argument");
    return SPH_ERR_INVALID;
  }
  SPH_TRY(require_lists(H));
  sph_neighbors* M = const_cast<sph_neighbors*>(H);
  SPH_TRY(M->tmp_i32a.alloc(H->n));
  int grid = grid_for(H, H->n);
  SPH_LAUNCH(k_export_counts, grid, kBlock, 0, st)(H->iperm.p, H->cnt.p, H->n, M->tmp_i32a.p);
  SPH_TRY_CUDA(cudaGetLastError());
  SPH_TRY(scan<int64_t>(M, M->tmp_i32a.p, offsets, H->n, 1, nullptr, st));
  SPH_TRY(ensure_nbr(M, st));
  if (H->nnz > 0) {
    SPH_LAUNCH(k_export_fill, grid, kBlock, 0, st)(H->iperm.p, H->perm.p, H->cnt.p, H->slice_off.p, H->nbr.p, H->n, offsets,
                                           idx);
    SPH_TRY_CUDA(cudaGetLastError());
  }
  SPH_TRY_CUDA(cudaStreamSynchronize(st));
  return SPH_OK;
}

}  // namespace sph
