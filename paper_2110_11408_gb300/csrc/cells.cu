// Cell binning, kernel density and L0 friends-of-friends.
//
// Particles are binned into nc^3 cells of side 2^21/nc >= b (a counting sort
// into a dense cell table, x fastest, each cell ordered by x inside), so
// every neighbour within b of a particle lies in the 27 cells around its own
// and, for the three cells of one (y, z) row, in one contiguous run of the
// sorted array, itself sorted by x.  Periodic wrap
// is handled per run by shifting the query point by one box length, never
// per pair.  With side <= 2^14 grid units every |dx| inside the stencil is
// below 2^15, so squared distances fit uint32 exactly.
#include <limits.h>
#include <math.h>

#include "cells.cuh"
#include "rank2.cuh"

namespace {

// Table cell of input particle i under the rules of k_cell_count: a position
// outside the box counts as (0, 0, 0) and a window particle outside the
// window's columns is filed under table column 0 with y = z = 0 (both set
// *bad_code).
__device__ __forceinline__ uint32_t bin_key(const int32_t* __restrict__ pos, size_t i, const CellGrid& g,
                                            int* bad_code) {
  int x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
  *bad_code = 0;
  if ((unsigned)x >= (unsigned)CSO_BOX || (unsigned)y >= (unsigned)CSO_BOX || (unsigned)z >= (unsigned)CSO_BOX) {
    *bad_code = 1;
    x = y = z = 0;
  }
  // table column from the grid x (whole box or window alike)
  int tc = g.colmap ? g.colmap[cell_coord(x, g.nc)] : cell_coord(x, g.nc);
  if (tc < 0) {
    *bad_code = 2;
    tc = 0;
    y = z = 0;
  }
  return (uint32_t)grid_cell(g, cell_coord(z, g.nc), cell_coord(y, g.nc), tc);
}

// Stored position of input particle i: x relative to the table's x0 (a
// window never wraps), y, z, and w = i.  A particle that k_cell_count
// rejected is stored at the low corner of table column 0, so every later
// kernel derives an in-range cell from it (the request still fails on the bad
// flag, but no kernel indexes past the table).
__device__ __forceinline__ int4 stored_pos(const int32_t* __restrict__ pos, size_t i, const CellGrid& g) {
  int x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
  const bool out = (unsigned)x >= (unsigned)CSO_BOX || (unsigned)y >= (unsigned)CSO_BOX ||
                   (unsigned)z >= (unsigned)CSO_BOX || (g.colmap && g.colmap[cell_coord(x, g.nc)] < 0);
  if (out) {
    x = g.colmap ? cell_lo(g.cols[0], g.nc) : 0;
    y = z = 0;
  }
  return make_int4((x - g.x0) & (CSO_BOX - 1), y, z, (int)i);
}

// Cells are sorted by x (k_cell_place), so a run of adjacent x cells is
// sorted by stored x: trim [lo, hi) to the neighbours with xl <= x <= xh by
// two binary searches in lockstep.
__device__ __forceinline__ void x_trim(const int4* __restrict__ spos, uint32_t& lo, uint32_t& hi, int xl, int xh) {
  uint32_t a = lo, b = hi, c = lo, d = hi;
  while (a < b || c < d) {
    if (a < b) {
      const uint32_t m = (a + b) >> 1;
      if (spos[m].x < xl) a = m + 1; else b = m;
    }
    if (c < d) {
      const uint32_t m = (c + d) >> 1;
      if (spos[m].x <= xh) c = m + 1; else d = m;
    }
  }
  lo = a;
  hi = c > a ? c : a;
}

// Rank of particle i among its cell's arrivals, in input order of the atomics.
__global__ void k_cell_count(const int32_t* __restrict__ pos, long long n, CellGrid g, uint32_t* __restrict__ key,
                             uint32_t* __restrict__ rank, uint32_t* __restrict__ count, int* __restrict__ bad) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int code;
  const uint32_t k = bin_key(pos, (size_t)i, g, &code);
  if (code) atomicExch(bad, code);
  key[i] = k;
  rank[i] = atomicAdd(&count[k], 1u);
}

// The same with two 16-bit counts to a word.  The add that takes a count past
// 65,535 sees it full, carries into the neighbour and sets *over: k_recount then
// counts again in 32 bits.
__global__ void k_cell_count_half(const int32_t* __restrict__ pos, long long n, CellGrid g, uint32_t* __restrict__ key,
                                  uint32_t* __restrict__ rank, uint32_t* __restrict__ count, int* __restrict__ over,
                                  int* __restrict__ bad) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int code;
  const uint32_t k = bin_key(pos, (size_t)i, g, &code);
  if (code) atomicExch(bad, code);
  key[i] = k;
  const int sh = (k & 1u) * 16;
  const uint32_t r = (atomicAdd(&count[k >> 1], 1u << sh) >> sh) & 0xffffu;
  if (r == 0xffffu) atomicExch(over, 1);
  rank[i] = r;
}

__global__ void k_recount_clear(uint32_t* __restrict__ count, long long ncell, const int* __restrict__ over) {
  if (*over == 0) return;
  const long long step = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < ncell; i += step) count[i] = 0;
}

__global__ void k_recount(long long n, const uint32_t* __restrict__ key, uint32_t* __restrict__ rank,
                          uint32_t* __restrict__ count, const int* __restrict__ over) {
  if (*over == 0) return;
  const long long step = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += step)
    rank[i] = atomicAdd(&count[key[i]], 1u);
}

// Everything k_cell_place needs of the particle at a provisional slot: its
// sort key (stored x << 32 | input index), its cell's range, its stored y and
// z and its id.  One record is one 32-byte sector, so the scatter writes
// whole sectors and the placement reads nothing from scattered places.
struct __align__(32) BinRec {
  unsigned long long key;
  uint32_t c0, m;
  int y, z;
  unsigned long long id;
};

// Provisional slot of every particle (cell start + arrival rank): the record
// is scattered there, and inv (optional) receives the provisional slot in
// input order.
__global__ void k_cell_scatter(const int32_t* __restrict__ pos, const uint64_t* __restrict__ ids, long long n,
                               CellGrid g, const uint32_t* __restrict__ key, const uint32_t* __restrict__ rank,
                               const uint32_t* __restrict__ start, BinRec* __restrict__ rec,
                               uint32_t* __restrict__ inv) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int4 q = stored_pos(pos, (size_t)i, g);
  const uint32_t k = key[i], c0 = start[k], c1 = start[k + 1];
  const uint32_t p = c0 + rank[i];
  // one 256-bit store: the whole sector in one scattered write
  const unsigned long long w0 = ((unsigned long long)(unsigned)q.x << 32) | (unsigned long long)i;
  const unsigned long long w1 = (unsigned long long)c0 | ((unsigned long long)(c1 - c0) << 32);
  const unsigned long long w2 = (unsigned long long)(unsigned)q.y | ((unsigned long long)(unsigned)q.z << 32);
  const unsigned long long w3 = ids[i];
  asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};" ::"l"(rec + p), "l"(w0), "l"(w1), "l"(w2), "l"(w3)
               : "memory");
  if (inv) inv[i] = p;
}

// Final slot of every particle: its cell's start plus its rank by (stored x,
// input index) among the cell's particles, so every cell, and with it every
// (y, z) row of adjacent x cells, is sorted by x (the density pass bounds its
// runs by x).  A lane counts a cell of up to 32 particles alone; the warp
// streams each larger cell once through shared memory for all its lanes in
// that cell.  Position and id come with the record and are written into the
// cell's range; fin (optional) maps the provisional slot to the final one
// (k_cell_inv composes it into inv).
constexpr int PLACE_SMALL = 32;
__global__ void __launch_bounds__(256) k_cell_place(long long n, const BinRec* __restrict__ rec,
                                                    int4* __restrict__ spos, uint64_t* __restrict__ sid,
                                                    uint32_t* __restrict__ fin) {
  __shared__ unsigned long long tile[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = t < n;
  unsigned long long kt = 0, id = 0;
  uint32_t c0 = 0, c1 = 0;
  int y = 0, z = 0;
  if (act) {
    unsigned long long w0, w1, w2, w3;
    asm volatile("ld.global.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(w0), "=l"(w1), "=l"(w2), "=l"(w3) : "l"(rec + t));
    kt = w0;
    c0 = (uint32_t)w1;
    c1 = c0 + (uint32_t)(w1 >> 32);
    y = (int)(uint32_t)w2;
    z = (int)(uint32_t)(w2 >> 32);
    id = w3;
  }
  const bool big = act && c1 - c0 > (uint32_t)PLACE_SMALL;
  uint32_t rk = 0;
  if (act && !big)
    for (uint32_t u = c0; u < c1; ++u) rk += rec[u].key < kt;
  unsigned pend = __ballot_sync(0xffffffffu, big);
  while (pend) {
    const int L = __ffs(pend) - 1;
    const uint32_t b0 = __shfl_sync(0xffffffffu, c0, L), b1 = __shfl_sync(0xffffffffu, c1, L);
    const bool mine = big && c0 == b0;
    for (uint32_t u0 = b0; u0 < b1; u0 += 32) {
      tile[w][lane] = u0 + lane < b1 ? rec[u0 + lane].key : ~0ull;  // past the cell: never below a key
      __syncwarp();
      if (mine) {
#pragma unroll 8
        for (int k = 0; k < 32; ++k) rk += tile[w][k] < kt;
      }
      __syncwarp();
    }
    pend &= ~__ballot_sync(0xffffffffu, mine);
  }
  if (!act) return;
  const uint32_t d = c0 + rk;
  spos[d] = make_int4((int)(kt >> 32), y, z, (int)(uint32_t)kt);
  sid[d] = id;
  if (fin) fin[t] = d;
}

// inv[i] = fin[inv[i]]: the final slot of every input particle (a gather in
// input order instead of a scattered write from the placement)
__global__ void k_cell_inv(long long n, const uint32_t* __restrict__ fin, uint32_t* __restrict__ inv) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) inv[i] = fin[inv[i]];
}

__device__ __forceinline__ uint32_t kern(int4 q, int xq, int yq, int zq, uint32_t b2) {
  const int dx = xq - q.x, dy = yq - q.y, dz = zq - q.z;
  const uint32_t d = (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
  return b2 - (d < b2 ? d : b2);  // b2 - d inside the kernel support, else 0
}

// Sigma_s = sum over j != s with d < b2 of (b2 - d)   (Eq. 1 times b2).
//
// A warp takes 32 consecutive cell-sorted particles.  When they all sit in
// one (y, z) row of cells and span at most max_span + 1 adjacent x cells
// (the common case wherever the work is: in and around dense cells), they
// share the nine stencil rows, each the union of their x ranges, which is one
// contiguous run of the sorted array (plus a wrapped run at the periodic x
// edge).  The runs are flattened into one index range that the warp walks 32
// neighbours at a time: every lane loads one neighbour of the next 32 (in
// flight while the current 32 are summed, across run boundaries too) and
// stores its offset and -|c|^2 into the warp's shared tile.  Warps whose
// particles span more cells walk the stencil lane by lane.
//
// Every lane sums DENS_Q = 4 of the warp's 32 queries over every fourth
// neighbour of a tile (lanes l, l + 8, l + 16, l + 24 hold the same queries
// and take one neighbour in four each; their sums meet in two shuffles at
// the end): one 128-bit shared load then serves four pairs per lane instead
// of one.  A broadcast 128-bit load returns 512 bytes to the registers, 8
// cycles of a sub-core's load path against 6 of its multiply-add pipe for a
// pair, so one load per pair was the kernel's limit.
//
// Offsets are taken from the warp's first particle o: the query is
// q = p - o, a staged neighbour c = t - shift - o, and b2 - d =
// (b2 - |q|^2) - |c|^2 + 2 q.c, three multiply-adds from the staged -|c|^2:
//   * when every true d is below 2^31 (cells below 9,459 grid units), b2 - d
//     is a signed 32-bit integer and max(b2 - d, 0) one add-and-max;
//   * otherwise d is formed modulo 2^32 and b2 - min(d, b2) summed; it is
//     exact because the true d of every staged pair is below 2^32 (max_span
//     is chosen on the host so that ((max_span + 2)^2 + 8) cell^2 < 2^32).
// The multiply-adds (half rate: 6 cycles of a sub-core per 32 pairs) are what
// is left as the bound of the shared walk: of 4.69 ms on a side-256 box (16.8M
// particles; another draw of the same recipe, the benchmark's, takes 4.9) its inner
// loop takes 2.7, the set-up of the rows 0.7 and the lane-by-lane walks the rest.
// One query per lane: 5.36 ms, and 1.03 ms against 0.70 on a side-128 box.
//
// Blocks run heaviest first: a cost pass files each block under
// floor(log2) of its warps' summed cell counts and the density launch takes
// block order[blockIdx.x], so the dense-halo blocks start in the first wave
// instead of forming the tail.
constexpr int DENS_WARPS = 8;
constexpr int DENS_CLASSES = 33;
constexpr int DENS_Q = 4;            // queries per lane
constexpr int DENS_L = 32 / DENS_Q;  // lanes holding the warp's 32 queries

__device__ __forceinline__ uint32_t sq3(int x, int y, int z) {
  return (uint32_t)x * (uint32_t)x + (uint32_t)y * (uint32_t)y + (uint32_t)z * (uint32_t)z;
}

// The shared-walk setup of one warp: whether its valid particles share a
// (y, z) cell row and a short x span, and, for lanes 0-8, the runs of stencil
// row (dz + 1) * 3 + (dy + 1): main run [lo0, hi0) and the wrapped run
// [lo1, hi1) with its x shift sx1.
struct WarpRows {
  bool uniform;
  int src;  // first valid lane
  uint32_t lo0, hi0, lo1, hi1;
  int sy, sz, sx1;
};

__device__ __forceinline__ WarpRows warp_rows(const CellGrid& g, int4 p, bool valid, unsigned vmask, int lane,
                                              int max_span) {
  WarpRows R{};
  const int nc = g.nc;
  const int cy = cell_coord(p.y, nc), cz = cell_coord(p.z, nc), tc = grid_col(g, p.x);
  R.src = __ffs(vmask) - 1;
  const int yz = cz * nc + cy;
  const int yz0 = __shfl_sync(0xffffffffu, yz, R.src);
  const int tmin = __reduce_min_sync(0xffffffffu, valid ? tc : INT_MAX);
  const int tmax = __reduce_max_sync(0xffffffffu, valid ? tc : INT_MIN);
  R.uniform = __all_sync(0xffffffffu, !valid || yz == yz0) && tmax - tmin <= max_span;
  if (!R.uniform) return R;
  int a = tmin, b = tmax, wl = -1, wr = -1;
  if (!g.colmap) {
    if (tmin > 0) a = tmin - 1; else wl = nc - 1;
    if (tmax + 1 < nc) b = tmax + 1; else wr = 0;
  } else {
    // table columns tmin..tmax must be adjacent columns of the box
    const int k = tmin + lane;
    const bool gap = k < tmax && g.cols[k + 1] != (g.cols[k] + 1) % nc;
    if (__any_sync(0xffffffffu, gap)) {
      R.uniform = false;
      return R;
    }
    if (tmin > 0 && g.cols[tmin - 1] == (g.cols[tmin] + nc - 1) % nc) a = tmin - 1;
    if (tmax + 1 < g.ncols && g.cols[tmax + 1] == (g.cols[tmax] + 1) % nc) b = tmax + 1;
  }
  if (lane < 9) {
    const int ccy = yz0 % nc, ccz = yz0 / nc;
    const int zz = wrap_yz(ccz + lane / 3 - 1, nc, R.sz);
    const int yy = wrap_yz(ccy + lane % 3 - 1, nc, R.sy);
    const uint32_t* row = grid_row(g, zz, yy);
    R.lo0 = row[a];
    R.hi0 = row[b + 1];
    if (wl >= 0) { R.lo1 = row[wl]; R.hi1 = row[wl + 1]; R.sx1 = CSO_BOX; }
    if (wr >= 0) { R.lo1 = row[wr]; R.hi1 = row[wr + 1]; R.sx1 = -CSO_BOX; }
  }
  return R;
}

// Cost class and in-class rank of every density block: one thread per warp of
// the density pass, charging it the cell of its first particle.
__global__ void __launch_bounds__(256) k_density_cost(CellGrid g, const int4* __restrict__ spos, int n, int nb,
                                                      uint8_t* __restrict__ cls, uint32_t* __restrict__ rank,
                                                      uint32_t* __restrict__ counts) {
  const int wi = blockIdx.x * blockDim.x + threadIdx.x;  // warp of the density pass
  const long long s = (long long)wi * 32;
  uint32_t m = 0;
  if (s < n) {
    const int4 p = spos[s];
    const size_t k = grid_cell(g, cell_coord(p.z, g.nc), cell_coord(p.y, g.nc), grid_col(g, p.x));
    m = g.start[k + 1] - g.start[k];
  }
#pragma unroll
  for (int o = 1; o < DENS_WARPS; o <<= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
  const int blk = wi / DENS_WARPS, lane = threadIdx.x & 31;
  const bool lead = wi % DENS_WARPS == 0 && blk < nb;
  const int k = lead ? 31 - __clz((int)(m | 1u)) : -1;
  const unsigned peers = __match_any_sync(0xffffffffu, k);
  if (!lead) return;
  const int first = __ffs(peers) - 1;
  uint32_t base = 0;
  if (lane == first) base = atomicAdd(&counts[k], (uint32_t)__popc(peers));
  base = __shfl_sync(peers, base, first);
  cls[blk] = (uint8_t)k;
  rank[blk] = base + __popc(peers & ((1u << lane) - 1u));
}

// order[position] = block, classes in decreasing cost
__global__ void k_density_order(const uint8_t* __restrict__ cls, const uint32_t* __restrict__ rank,
                                const uint32_t* __restrict__ counts, int nb, uint32_t* __restrict__ order) {
  __shared__ uint32_t first[DENS_CLASSES];
  if (threadIdx.x == 0) {
    uint32_t acc = 0;
    for (int k = DENS_CLASSES - 1; k >= 0; --k) {
      first[k] = acc;
      acc += counts[k];
    }
  }
  __syncthreads();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < nb) order[first[cls[b]] + rank[b]] = (uint32_t)b;
}

// The flattened runs of a shared walk: run r = 2 * row + wrapped holds the
// neighbours f < end[r] (and not of an earlier run) at sorted index
// f + off.w, their image's offset origin in off.xyz.
struct DensRuns {
  uint32_t end[18];
  int4 off[18];
};

// The stencil of one lane whose warp spans too many cells to share rows (the
// background and halo outskirts: few neighbours per row).  The bounds of a
// plane's three rows are loaded together before any is walked (a row by
// itself waits for its bounds first), and the rows walked one by one, so that
// lanes of one cell read the same neighbours together: one flat sequence per
// lane over all nine rows measured 1.6 times slower for the whole pass.
__device__ __forceinline__ unsigned long long lane_walk(const CellGrid& g, const int4* __restrict__ spos, int4 p,
                                                        uint32_t b2) {
  const int nc = g.nc;
  const int cy = cell_coord(p.y, nc), cz = cell_coord(p.z, nc);
  const XCells X = x_cells(g, grid_col(g, p.x));
  unsigned long long acc = 0;
#pragma unroll 1
  for (int dz = -1; dz <= 1; ++dz) {
    uint32_t lo[3], hi[3];
    int yq[3], zq[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      int sy, sz;
      const uint32_t* row = grid_row(g, wrap_yz(cz + dz, nc, sz), wrap_yz(cy + k - 1, nc, sy));
      yq[k] = p.y + sy;
      zq[k] = p.z + sz;
      lo[k] = row[X.a];
      hi[k] = row[X.b + 1];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll 8
      for (uint32_t t = lo[k]; t < hi[k]; ++t) acc += kern(spos[t], p.x, yq[k], zq[k], b2);
    }
  }
  const int wc = X.wl >= 0 ? X.wl : X.wr;  // the row's far end, at the periodic x edge of a whole box
  if (wc >= 0)
    for (int r = 0; r < 9; ++r) {
      int sy, sz;
      const uint32_t* row = grid_row(g, wrap_yz(cz + r / 3 - 1, nc, sz), wrap_yz(cy + r % 3 - 1, nc, sy));
      for (uint32_t t = row[wc], e = row[wc + 1]; t < e; ++t)
        acc += kern(spos[t], X.wl >= 0 ? p.x + CSO_BOX : p.x - CSO_BOX, p.y + sy, p.z + sz, b2);
    }
  return acc;
}

template <bool SIGNED>
__global__ void __launch_bounds__(DENS_WARPS * 32, 4) k_density(CellGrid g, const int4* __restrict__ spos, int n,
                                                                 uint32_t b2, int reach, int include_self,
                                                                 long long* __restrict__ sigma,
                                                                 const uint8_t* __restrict__ only,
                                                                 const uint32_t* __restrict__ order, int max_span) {
  __shared__ int4 tile[DENS_WARPS][2][32];
  __shared__ DensRuns runs[DENS_WARPS];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int blk = order ? (int)order[blockIdx.x] : (int)blockIdx.x;
  const int s = blk * blockDim.x + threadIdx.x;
  const bool valid = s < n && (!only || only[s]);
  const int4 p = s < n ? spos[s] : make_int4(0, 0, 0, 0);
  const unsigned vmask = __ballot_sync(0xffffffffu, valid);
  if (!vmask) return;
  WarpRows R = warp_rows(g, p, valid, vmask, lane, max_span);
  unsigned long long acc = 0;
  if (R.uniform) {
    // keep the neighbours within reach (the largest e with e^2 < b2) of the
    // warp's x extent in x: a neighbour farther out in x is farther than b
    // from every query of the warp
    const int xmin = __reduce_min_sync(0xffffffffu, valid ? p.x : INT_MAX);
    const int xmax = __reduce_max_sync(0xffffffffu, valid ? p.x : INT_MIN);
    const int ox = __shfl_sync(0xffffffffu, p.x, R.src), oy = __shfl_sync(0xffffffffu, p.y, R.src),
              oz = __shfl_sync(0xffffffffu, p.z, R.src);
    if (lane < 9) {
      // neighbour image x = stored x - shift
      if (R.hi0 - R.lo0 > 16u) x_trim(spos, R.lo0, R.hi0, xmin - reach, xmax + reach);
      if (R.hi1 - R.lo1 > 16u) x_trim(spos, R.lo1, R.hi1, xmin - reach + R.sx1, xmax + reach + R.sx1);
    }
    const uint32_t n0 = lane < 9 ? R.hi0 - R.lo0 : 0u, n1 = lane < 9 ? R.hi1 - R.lo1 : 0u;
    uint32_t inc = n0 + n1;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, inc, 8);
    DensRuns& F = runs[w];
    if (lane < 9) {
      const uint32_t f1 = inc - n1, f0 = f1 - n0;
      F.end[2 * lane] = f1;
      F.end[2 * lane + 1] = inc;
      F.off[2 * lane] = make_int4(ox, oy + R.sy, oz + R.sz, (int)(R.lo0 - f0));
      F.off[2 * lane + 1] = make_int4(ox + R.sx1, oy + R.sy, oz + R.sz, (int)(R.lo1 - f1));
    }
    // this lane's queries: lanes lq + DENS_L i of the warp
    const int lq = lane & (DENS_L - 1), grp = lane / DENS_L;
    uint32_t ax[DENS_Q], ay[DENS_Q], az[DENS_Q], B[DENS_Q];
    unsigned long long sum[DENS_Q];
#pragma unroll
    for (int i = 0; i < DENS_Q; ++i) {
      const int from = lq + DENS_L * i;
      const int qx = __shfl_sync(0xffffffffu, p.x, from) - ox, qy = __shfl_sync(0xffffffffu, p.y, from) - oy,
                qz = __shfl_sync(0xffffffffu, p.z, from) - oz;
      const uint32_t P = sq3(qx, qy, qz);
      // SIGNED: B + (-|c|^2 + 2 q.c) = b2 - d; else P - (-|c|^2 + 2 q.c) = d
      B[i] = SIGNED ? b2 - P : P;
      ax[i] = 2u * (uint32_t)qx;
      ay[i] = 2u * (uint32_t)qy;
      az[i] = 2u * (uint32_t)qz;
      sum[i] = 0;
    }
    __syncwarp();
    // past the last neighbour: a staged value no query counts (b2 - d becomes
    // -|q|^2 in the signed form, and d |q|^2 + 2^31 with |q|^2 below 2^31 in the
    // general one)
    const int4 none = make_int4(0, 0, 0, SIGNED ? -(int)b2 : INT_MIN);
    int r = 0;
    uint32_t rend = F.end[0], f = (uint32_t)lane;
    int4 next = make_int4(0, 0, 0, 0);
    if (f < total) {
      while (f >= rend) rend = F.end[++r];
      next = spos[f + (uint32_t)F.off[r].w];
    }
    for (uint32_t t0 = 0, buf = 0; t0 < total; t0 += 32, buf ^= 1) {
      int4* tl = tile[w][buf];
      if (f < total) {
        const int4 o = F.off[r];
        const int cx = next.x - o.x, cy = next.y - o.y, cz = next.z - o.z;
        tl[lane] = make_int4(cx, cy, cz, -(int)sq3(cx, cy, cz));
      } else {
        tl[lane] = none;
      }
      f += 32;
      if (f < total) {
        while (f >= rend) rend = F.end[++r];
        next = spos[f + (uint32_t)F.off[r].w];
      }
      __syncwarp();  // the other buffer's readers are past the last barrier
      const int it = total - t0 < 32u ? (int)(total - t0 + DENS_Q - 1) / DENS_Q : DENS_L;
      // b2 - d < b2 <= 2^28: eight of them fit 32 bits
      uint32_t part[DENS_Q] = {};
#pragma unroll 4
      for (int k = 0; k < it; ++k) {
        const int4 c = tl[k * DENS_Q + grp];
#pragma unroll
        for (int i = 0; i < DENS_Q; ++i) {
          const uint32_t t = (uint32_t)c.w + ax[i] * (uint32_t)c.x + ay[i] * (uint32_t)c.y + az[i] * (uint32_t)c.z;
          if (SIGNED) {
            part[i] += (uint32_t)__viaddmax_s32((int)t, (int)B[i], 0);
          } else {
            const uint32_t d = B[i] - t;
            part[i] += b2 - (d < b2 ? d : b2);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < DENS_Q; ++i) sum[i] += part[i];
    }
    // the lanes of one set of queries add up; every lane keeps its own particle's
#pragma unroll
    for (int i = 0; i < DENS_Q; ++i) {
#pragma unroll
      for (int o = DENS_L; o < 32; o <<= 1) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
      if (grp == i) acc = sum[i];
    }
  } else if (valid) {
    acc = lane_walk(g, spos, p, b2);
  }
  if (!valid) return;
  if (!include_self) acc -= b2;
  sigma[s] = (long long)acc;
}

// number of ordered pairs j != s with d < b2 (the algorithmic work of the
// density pass; a separate diagnostic launch)
__global__ void __launch_bounds__(256) k_count_pairs(CellGrid g, const int4* __restrict__ spos, int n, uint32_t b2,
                                                     unsigned long long* __restrict__ pairs) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned cnt = 0;
  if (s < n) {
    const int4 p = spos[s];
    for_stencil(g, p.x, p.y, p.z, [&](uint32_t t, int xq, int yq, int zq) { cnt += kern(spos[t], xq, yq, zq, b2) != 0; });
    cnt -= 1;  // the particle itself
  }
  unsigned tot = __reduce_add_sync(0xffffffffu, cnt);
  if ((threadIdx.x & 31) == 0) atomicAdd(pairs, (unsigned long long)tot);
}

// ---------------------------------------------------------------------------
// union-find over sorted indices: parent[x] <= x always, roots are the
// smallest index of their component, hooks go from the larger root to the
// smaller one by compare-and-swap (lock-free; any interleaving ends in the
// same components).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int uf_root(int* parent, int x) {
  int p = parent[x];
  while (p != x) {
    int gp = parent[p];
    if (gp != p) parent[x] = gp;  // halve the path; gp is still an ancestor of x
    x = p;
    p = gp;
  }
  return x;
}

__device__ __forceinline__ void uf_unite(int* parent, int a, int b) {
  a = uf_root(parent, a);
  b = uf_root(parent, b);
  while (a != b) {
    if (a < b) {
      int t = a;
      a = b;
      b = t;
    }
    // hook root a (larger) under b
    int old = atomicCAS(&parent[a], a, b);
    if (old == a) return;
    // a was hooked elsewhere meanwhile: climb and retry
    a = uf_root(parent, old);
    b = uf_root(parent, b);
  }
}

// Every cell that holds dense particles has a main tree: the tree of its
// first dense particle after pass one, kept at slot start[c] of a
// per-particle array (the first slot of every non-empty cell is its own) so
// the summary costs n entries instead of one per cell of the sparse table;
// CELL_EMPTY marks cells without dense particles.  A dense particle outside
// its cell's main tree at that point is a straggler.
constexpr int CELL_EMPTY = -2;

__device__ __forceinline__ uint32_t cell_id(const CellGrid& g, int4 p) {
  return (uint32_t)grid_cell(g, cell_coord(p.z, g.nc), cell_coord(p.y, g.nc), grid_col(g, p.x));
}

// The forest's start (parent[s] = s for dense particles, -1 for the rest: one
// load answers both), the cells' summaries and the groups' smallest ids
// cleared, and two lists in cell order: the dense particles (FoF threads take
// one each, so a warp holds 32 dense particles instead of 32 slots of which
// only the dense ones work), and the first dense particle of every cell that
// holds any.  counts[0] and counts[1] receive their lengths.  (A pass each
// for the flags, their scans and the lists: 0.39 ms on the side-256 box, this
// one 0.16.)

// dense slot i is the first one of its cell: no dense slot before it there (the
// one next to it, mostly)
__device__ __forceinline__ bool first_dense(const CellGrid& g, const int4* __restrict__ spos,
                                            const long long* __restrict__ sigma, long long T_L0, long long i) {
  const uint32_t c = cell_id(g, spos[i]);
  for (long long t = i - 1; t >= 0 && cell_id(g, spos[t]) == c; --t)
    if (sigma[t] > T_L0) return false;
  return true;
}

template <int ITEMS>
__global__ void __launch_bounds__(R2_THREADS, 8) k_fof_lists(CellGrid g, const int4* __restrict__ spos, int n,
                                                          const long long* __restrict__ sigma, long long T_L0,
                                                          int* __restrict__ parent, int* __restrict__ cell_root,
                                                          unsigned long long* __restrict__ minid,
                                                          int* __restrict__ didx, int* __restrict__ clist,
                                                          uint32_t* __restrict__ counts,
                                                          unsigned long long* __restrict__ status, long long ntiles,
                                                          long long patience) {
  __shared__ Rank2Shared S;
  const long long tile = rank2_tile(S, status, ntiles);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long base = tile * (R2_THREADS * ITEMS) + (long long)w * 32 * ITEMS;
  unsigned dense[ITEMS], head[ITEMS];
#pragma unroll
  for (int q = 0; q < ITEMS; ++q) {
    const long long i = base + q * 32 + lane;
    const bool in = i < n;
    const bool d = in && sigma[i] > T_L0;
    dense[q] = __ballot_sync(0xffffffffu, d);
    if (in) {
      parent[i] = d ? (int)i : -1;
      cell_root[i] = CELL_EMPTY;
      minid[i] = ~0ull;
    }
  }
  uint32_t na = 0, nb = 0;
#pragma unroll
  for (int q = 0; q < ITEMS; ++q) {
    const bool h = (dense[q] >> lane & 1u) && first_dense(g, spos, sigma, T_L0, base + q * 32 + lane);
    head[q] = __ballot_sync(0xffffffffu, h);
    na += __popc(dense[q]);
    nb += __popc(head[q]);
  }
  uint32_t ta, tb;
  rank2_prefix(S, status, tile, na, nb, ta, tb, patience, [&](long long t) {
    return rank2_count<ITEMS>(t, [&](long long i) {
      return sigma[i] > T_L0 ? 1u | (first_dense(g, spos, sigma, T_L0, i) ? 2u : 0u) : 0u;
    });
  });
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int q = 0; q < ITEMS; ++q) {
    const int i = (int)(base + q * 32 + lane);
    if (dense[q] >> lane & 1u) didx[na + __popc(dense[q] & lt)] = i;
    if (head[q] >> lane & 1u) clist[nb + __popc(head[q] & lt)] = i;
    na += __popc(dense[q]);
    nb += __popc(head[q]);
  }
  if (tile == ntiles - 1 && threadIdx.x == 0) {
    counts[0] = ta;
    counts[1] = tb;
  }
}

// Pass one (in the spirit of Afforest, Sutton et al. 2018): each dense
// particle tests the W = 32 slots after it in its cell, cyclically, so every
// pair of a cell of up to 33 particles is tested and a big cell is joined by
// a band of links around it.  The band joins almost every dense particle of
// a big cell into one tree; the few it misses are handled one by one later.
// A narrower band gains 2% where it suffices (16: FoF 3.24 against 3.31 ms on a
// side-256 box) and costs 40% where it does not (16 on the benchmark's box of
// that size: 4.64 against 3.30; 8 on the first: 4.54), by the cells whose trees
// it leaves in pieces.
//
// A warp whose particles share a cell streams the union of its lanes'
// windows through shared memory; the lane that stages a particle also stages
// its current root (-1 if not dense), so a lane pays a forest update only for
// a link into another tree.  A staged root that has since been hooked
// elsewhere is still a member of its tree, so the test stays correct.
constexpr uint32_t FOF_BAND = 32;

__global__ void __launch_bounds__(256) k_fof_sample(CellGrid g, const int4* __restrict__ spos,
                                                    const int* __restrict__ didx, const uint32_t* __restrict__ nd_ptr,
                                                    uint32_t lfof2, int* __restrict__ parent) {
  __shared__ int4 tile[8][32];
  __shared__ int troot[8][32];
  const int nd = (int)*nd_ptr;
  if ((int)(blockIdx.x * blockDim.x) >= nd) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = i < nd;
  const unsigned vmask = __ballot_sync(0xffffffffu, valid);
  if (!vmask) return;
  const int s = valid ? didx[i] : -1;
  const int4 p = valid ? spos[s] : make_int4(0, 0, 0, 0);
  const size_t cell = grid_cell(g, cell_coord(p.z, g.nc), cell_coord(p.y, g.nc), grid_col(g, p.x));
  const int src = __ffs(vmask) - 1;
  const size_t cell0 = __shfl_sync(0xffffffffu, cell, src);
  const bool uniform = __all_sync(0xffffffffu, !valid || cell == cell0);
  int rs = valid ? uf_root(parent, s) : -1;
  if (uniform) {
    // cell-relative positions: lane j tests j + 1 .. j + h (mod m)
    const uint32_t c_lo = g.start[cell0], c_hi = g.start[cell0 + 1];
    const uint32_t m = c_hi - c_lo;
    const uint32_t h = m - 1 < FOF_BAND ? m - 1 : FOF_BAND;
    const uint32_t j = valid ? (uint32_t)s - c_lo : 0;
    const uint32_t j_first = __shfl_sync(0xffffffffu, j, src);
    const uint32_t j_last = __shfl_sync(0xffffffffu, j, 31 - __clz(vmask));
    const uint32_t v_end = j_last + h + 1;
    for (uint32_t v0 = j_first + 1; v0 < v_end; v0 += 32) {
      const uint32_t v = v0 + lane;
      int tr = -1;
      if (v < v_end) {
        const uint32_t t = c_lo + (v < m ? v : v - m);  // v < 2m
        tile[w][lane] = spos[t];
        if (parent[t] >= 0) tr = uf_root(parent, (int)t);
      }
      troot[w][lane] = tr;
      __syncwarp();
      const int cnt = v_end - v0 < 32 ? (int)(v_end - v0) : 32;
      if (valid) {
        for (int k = 0; k < cnt; ++k) {
          const int rt = troot[w][k];
          const uint32_t off = v0 + k - j;  // cyclic distance after this lane's slot
          if (rt < 0 || rt == rs || off - 1 >= h) continue;
          const int4 q = tile[w][k];
          const int dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
          const uint32_t d = (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
          if (d >= lfof2) continue;
          uf_unite(parent, rs, rt);
          rs = uf_root(parent, rs);
        }
      }
      __syncwarp();
    }
    return;
  }
  if (!valid) return;
  // lanes of several cells: each walks its own band
  const uint32_t c_lo = g.start[cell], m = g.start[cell + 1] - c_lo;
  const uint32_t h = m - 1 < FOF_BAND ? m - 1 : FOF_BAND;
  for (uint32_t o = 1, j = (uint32_t)s - c_lo; o <= h; ++o) {
    const uint32_t v = j + o;
    const uint32_t t = c_lo + (v < m ? v : v - m);
    const int4 q = spos[t];
    const int dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
    const uint32_t d = (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
    if (d >= lfof2) continue;
    const int pt = parent[t];
    if (pt < 0 || pt == rs) continue;
    const int rt = uf_root(parent, pt);
    if (rt != rs) {
      uf_unite(parent, rs, rt);
      rs = uf_root(parent, rs);
    }
  }
}

// the main tree of every cell that holds dense particles, after pass one
__global__ void k_cell_main(const int4* __restrict__ spos, CellGrid g, const int* __restrict__ clist,
                            const uint32_t* __restrict__ ncl_ptr, int* __restrict__ parent,
                            int* __restrict__ cell_root) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int)*ncl_ptr) return;
  const int s0 = clist[i];
  cell_root[g.start[cell_id(g, spos[s0])]] = uf_root(parent, s0);
}

// The stragglers, listed in cell order; srange[start[c]] = the run of cell c
// (one with dense particles) in that list.  Also points every dense particle
// straight at its root.  Tiles are of the dense list: those past its end have
// nothing to publish.
template <int ITEMS>
__global__ void __launch_bounds__(R2_THREADS) k_stragglers(const int4* __restrict__ spos, CellGrid g,
                                                           const int* __restrict__ didx, uint32_t* __restrict__ counts,
                                                           int* __restrict__ parent, const int* __restrict__ cell_root,
                                                           uint8_t* __restrict__ strag, int* __restrict__ slist,
                                                           uint2* __restrict__ srange,
                                                           unsigned long long* __restrict__ status, long long ntiles,
                                                           long long patience) {
  __shared__ Rank2Shared S;
  const long long nd = counts[0];
  const long long tile = rank2_tile(S, status, ntiles);
  if (tile * (R2_THREADS * ITEMS) >= nd) return;  // counts[2] starts at zero
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long base = tile * (R2_THREADS * ITEMS) + (long long)w * 32 * ITEMS;
  unsigned flag[ITEMS];
  uint32_t lo[ITEMS];  // the cell's first slot
  unsigned first = 0, last = 0;
  uint32_t na = 0, nb = 0;
#pragma unroll
  for (int q = 0; q < ITEMS; ++q) {
    const long long i = base + q * 32 + lane;
    bool f = false, a = false, z = false;
    uint32_t c = 0;
    const bool in = i < nd;
    int s = 0;
    if (in) {
      s = didx[i];
      c = cell_id(g, spos[s]);
    }
    uint32_t cp = __shfl_up_sync(0xffffffffu, c, 1), cn = __shfl_down_sync(0xffffffffu, c, 1);
    lo[q] = 0;
    if (in) {
      if (lane == 0) cp = i > 0 ? cell_id(g, spos[didx[i - 1]]) : ~c;
      if (lane == 31) cn = i + 1 < nd ? cell_id(g, spos[didx[i + 1]]) : ~c;
      a = cp != c;
      z = cn != c || i + 1 == nd;
      lo[q] = g.start[c];
      const int r = uf_root(parent, s);
      parent[s] = r;
      f = r != cell_root[lo[q]];
      strag[s] = (uint8_t)f;
    }
    first |= (unsigned)a << q;
    last |= (unsigned)z << q;
    flag[q] = __ballot_sync(0xffffffffu, f);
    na += __popc(flag[q]);
  }
  uint32_t ta, tb;
  // (roots do not change in this pass, so a tile counted here counts as it does itself)
  rank2_prefix(S, status, tile, na, nb, ta, tb, patience, [&](long long t) {
    return rank2_count<ITEMS>(t, [&](long long i) {
      const int s = didx[i];
      return uf_root(parent, s) != cell_root[g.start[cell_id(g, spos[s])]] ? 1u : 0u;
    });
  });
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int q = 0; q < ITEMS; ++q) {
    const uint32_t r = na + __popc(flag[q] & lt);
    const uint32_t f = flag[q] >> lane & 1u;
    if (f) slist[r] = didx[base + q * 32 + lane];
    if (first >> q & 1u) srange[lo[q]].x = r;
    if (last >> q & 1u) srange[lo[q]].y = r + f;
    na += __popc(flag[q]);
  }
  if ((tile + 1) * (R2_THREADS * ITEMS) >= nd && threadIdx.x == 0) counts[2] = ta;
}

__device__ __forceinline__ int fold21(int v) { return (int)((unsigned)v << 11) >> 11; }  // nearest image

// lane whose run of the flat sequence holds f (incl: inclusive ends of the lanes' runs)
__device__ __forceinline__ int flat_owner(uint32_t incl, uint32_t f) {
  int r = 0;
#pragma unroll
  for (int o = 16; o; o >>= 1)
    if (__shfl_sync(0xffffffffu, incl, r + o - 1) <= f) r += o;
  return r;
}

__device__ __forceinline__ uint32_t warp_incl_u32(uint32_t v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Pair of cells one of which holds more than 32 slots, by the whole warp:
// whether any member of main tree A (slots a_lo .. a_hi) links with any of B
// (slots lo .. hi, whose image our positions shifted by (sx, sy, sz) meet).
// The warp holds 32 slots of A at a time, streams B through shared memory and
// stops at the first link, so a pair of dense cells costs one tile instead of
// a test per particle.
__device__ __forceinline__ bool fof_big_pair(const int4* __restrict__ spos, uint32_t a_lo, uint32_t a_hi, uint32_t lo,
                                             uint32_t hi, int sx, int sy, int sz, uint32_t lfof2, int lreach,
                                             const int* __restrict__ parent, const uint8_t* __restrict__ strag,
                                             int4* tile, int* tmain, int lane) {
  bool found = false;
  // only our slots within l_FoF in x of the neighbour's x extent can link
  uint32_t ta = a_lo, tb = a_hi;
  if (lane == 0 && tb - ta > 32u) {
    const int bx0 = spos[lo].x - sx, bx1 = spos[hi - 1].x - sx;
    x_trim(spos, ta, tb, bx0 - lreach, bx1 + lreach);
  }
  ta = __shfl_sync(0xffffffffu, ta, 0);
  tb = __shfl_sync(0xffffffffu, tb, 0);
  for (uint32_t a0 = ta; a0 < tb && !found; a0 += 32) {
    const uint32_t a = a0 + lane;
    const bool av = a < tb && parent[a] >= 0 && !strag[a];
    const int4 pa = av ? spos[a] : make_int4(0, 0, 0, 0);
    const int xq = pa.x + sx, yq = pa.y + sy, zq = pa.z + sz;
    if (!__any_sync(0xffffffffu, av)) continue;
    // the neighbour's slots within l_FoF of this tile in x (cells are sorted by x)
    const int xqmin = __reduce_min_sync(0xffffffffu, av ? xq : INT_MAX);
    const int xqmax = __reduce_max_sync(0xffffffffu, av ? xq : INT_MIN);
    uint32_t blo = lo, bhi = hi;
    if (lane == 0 && bhi - blo > 32u) x_trim(spos, blo, bhi, xqmin - lreach, xqmax + lreach);
    blo = __shfl_sync(0xffffffffu, blo, 0);
    bhi = __shfl_sync(0xffffffffu, bhi, 0);
    for (uint32_t b0 = blo; b0 < bhi; b0 += 32) {
      const uint32_t t = b0 + lane;
      const bool tv = t < bhi && parent[t] >= 0 && !strag[t];
      tile[lane] = tv ? spos[t] : make_int4(0, 0, 0, 0);
      tmain[lane] = tv;
      __syncwarp();
      const int m = bhi - b0 < 32 ? (int)(bhi - b0) : 32;
      bool found_here = false;
      if (av) {
        for (int k = 0; k < m; ++k) {
          if (!tmain[k]) continue;
          const int4 qb = tile[k];
          const int dx = xq - qb.x, dy = yq - qb.y, dz = zq - qb.z;
          const uint32_t d = (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
          if (d < lfof2) {
            found_here = true;
            break;
          }
        }
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, found_here)) {
        found = true;
        break;
      }
    }
  }
  return found;
}

// Pass two, main trees as units: for every cell with dense particles and
// each of its 13 forward neighbours (every adjacent pair of cells once), the
// two main trees are joined if any pair of their members links.  Half a warp
// per cell: lanes 0-12 of the half look up a neighbour each (its range, its
// summary and both trees' roots: a chain of dependent loads that is all the
// time there is to a small cell, so a warp runs two), pairs already in one
// tree drop out, and the pairs of two cells of up to 32 slots are tested
// together, the half's lanes spread over (neighbour, slot) pairs against the
// cell staged once.  The whole warp then takes the other pairs of both cells
// in turn.  (Those on a list of their own, a warp per cell or per pair, were
// slower: joining one neighbour often joins the next, and sooner is better.)
// Full occupancy (32 registers, a few spilled) is worth more here than none
// spilled: FoF of the side-256 box 3.86 ms with a warp per cell, 3.75 with
// half a warp, 3.46 at eight blocks per SM.
__device__ __forceinline__ int forward_col(const XCells& X, int tc, int dx) {
  return dx < 0 ? (X.a < tc ? X.a : X.wl) : (dx > 0 ? (X.b > tc ? X.b : X.wr) : tc);
}

__global__ void __launch_bounds__(256, 8) k_fof_cells(CellGrid g, const int4* __restrict__ spos,
                                                   const int* __restrict__ clist, const uint32_t* __restrict__ ncl_ptr,
                                                   uint32_t lfof2, int lreach, int* __restrict__ parent,
                                                   const int* __restrict__ cell_root,
                                                   const uint8_t* __restrict__ strag) {
  __shared__ int4 tile[16][32];
  __shared__ int tmains[8][32];
  const int lane = threadIdx.x & 31, l16 = lane & 15, sub = lane >> 4;
  int4* tileA = tile[threadIdx.x >> 4];
  const int ncl = (int)*ncl_ptr;
  const int nc = g.nc;
  for (int i0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5 << 1; i0 < ncl; i0 += gridDim.x * blockDim.x >> 4) {
    const bool valid = i0 + sub < ncl;
    const int s0 = clist[valid ? i0 + sub : i0];
    const int4 p0 = spos[s0];
    const int cy = cell_coord(p0.y, nc), cz = cell_coord(p0.z, nc), tc = grid_col(g, p0.x);
    const size_t cA = grid_cell(g, cz, cy, tc);
    const uint32_t a_lo = g.start[cA], mA = g.start[cA + 1] - a_lo;
    const int crA = cell_root[a_lo];
    // lane r < 13: forward neighbour q = 14 + r, (dz, dy, dx) = (q / 9 - 1, q / 3 % 3 - 1, q % 3 - 1)
    uint32_t b_hi = 0, mB = 0;
    int crB = CELL_EMPTY, bsx = 0, bsy = 0, bsz = 0;
    if (l16 < 13) {
      const int q = 14 + l16, dx1 = q % 3 - 1;
      const int zz = wrap_yz(cz + q / 9 - 1, nc, bsz), yy = wrap_yz(cy + q / 3 % 3 - 1, nc, bsy);
      const XCells X = x_cells(g, tc);
      const int col = forward_col(X, tc, dx1);
      bsx = dx1 < 0 ? (X.a < tc ? 0 : CSO_BOX) : (dx1 > 0 ? (X.b > tc ? 0 : -CSO_BOX) : 0);
      if (col >= 0) {
        const size_t c = grid_cell(g, zz, yy, col);
        const uint32_t lo = g.start[c];
        b_hi = g.start[c + 1];
        mB = b_hi - lo;
        if (mB) crB = cell_root[lo];
      }
    }
    // every neighbour's tree against ours at once (a stale answer only costs a search)
    const bool need = valid && crB >= 0 && uf_root(parent, crB) != uf_root(parent, crA);
    const bool small = mA <= 32 && mB <= 32;
    unsigned big = __ballot_sync(0xffffffffu, need && !small);  // bit 16 sub + r
    const uint32_t cnt = need && small ? mB : 0;
    const unsigned any = __ballot_sync(0xffffffffu, cnt > 0);
    if (any) {
      const bool mine = any >> (16 * sub) & 0xffffu;
      unsigned amask = 0;
  #pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint32_t o = l16 + 16 * k;
        const bool av = mine && o < mA && parent[a_lo + o] >= 0 && !strag[a_lo + o];
        if (av) tileA[o] = spos[a_lo + o];
        amask |= (__ballot_sync(0xffffffffu, av) >> (16 * sub) & 0xffffu) << (16 * k);
      }
      uint32_t incl = cnt;
  #pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o, 16);
        if (l16 >= o) incl += t;
      }
      const uint32_t total = __shfl_sync(0xffffffffu, incl, 15, 16);
      const uint32_t longest = max(total, __shfl_xor_sync(0xffffffffu, total, 16));
      __syncwarp();
      unsigned hits = 0;  // bit 16 sub + r: pair r of the half links
      for (uint32_t f0 = 0; f0 < longest; f0 += 16) {
        const uint32_t f = f0 + l16;
        int r = 0;
  #pragma unroll
        for (int o = 8; o; o >>= 1)
          if (__shfl_sync(0xffffffffu, incl, r + o - 1, 16) <= f) r += o;
        const uint32_t end = __shfl_sync(0xffffffffu, incl, r, 16), hi = __shfl_sync(0xffffffffu, b_hi, r, 16);
        bool hit = false;
        if (f < total && !(hits >> (16 * sub + r) & 1u)) {
          const uint32_t t = hi - (end - f);
          if (parent[t] >= 0 && !strag[t]) {
            const int4 q = spos[t];
            for (unsigned m = amask; m; m &= m - 1) {
              const int4 pa = tileA[__ffs(m) - 1];
              const int dx = fold21(pa.x - q.x), dy = fold21(pa.y - q.y), dz = fold21(pa.z - q.z);
              if ((uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz) < lfof2) {
                hit = true;
                break;
              }
            }
          }
        }
        hits |= __reduce_or_sync(0xffffffffu, hit ? 1u << (16 * sub + r) : 0u);
      }
      if (hits >> lane & 1u) uf_unite(parent, crA, crB);
      __syncwarp();
    }
    for (; big; big &= big - 1) {
      const int r = __ffs(big) - 1;
      const uint32_t hi = __shfl_sync(0xffffffffu, b_hi, r), lo = hi - __shfl_sync(0xffffffffu, mB, r);
      const uint32_t alo = __shfl_sync(0xffffffffu, a_lo, r), ahi = alo + __shfl_sync(0xffffffffu, mA, r);
      const int ca = __shfl_sync(0xffffffffu, crA, r), cb = __shfl_sync(0xffffffffu, crB, r);
      const int sx = __shfl_sync(0xffffffffu, bsx, r), sy = __shfl_sync(0xffffffffu, bsy, r),
                sz = __shfl_sync(0xffffffffu, bsz, r);
      int same = 0;
      if (lane == 0) same = uf_root(parent, ca) == uf_root(parent, cb);
      if (__shfl_sync(0xffffffffu, same, 0)) continue;
      const bool found = fof_big_pair(spos, alo, ahi, lo, hi, sx, sy, sz, lfof2, lreach, parent, strag,
                                      tile[threadIdx.x >> 5 << 1], tmains[threadIdx.x >> 5], lane);
      if (found && lane == 0) uf_unite(parent, ca, cb);
      __syncwarp();
    }
  }
}

// Pass three, the stragglers: against every neighbour cell in l_FoF reach (its
// own included), the first link into the cell's main tree (skipped when that
// tree is already the straggler's) and every link to a later straggler (each
// straggler pair once).  A warp per straggler: lanes 0-26 look up one cell
// each (skipping those out of reach by the particle's distance to the home
// cell's faces, and trimming the rest to l_FoF in x), so the lookups' chain
// of dependent loads is paid once and not once per cell, and the slots of all
// cells are tested as one flat sequence, 32 at a time (a lane per straggler
// walking its cells in turn: 202 us for the 3,000 stragglers of the side-64
// box, where the longest walk set the time).
__global__ void __launch_bounds__(256, 8) k_fof_stragglers(CellGrid g, const int4* __restrict__ spos,
                                                        const int* __restrict__ slist,
                                                        const uint32_t* __restrict__ ns_ptr, uint32_t lfof2,
                                                        int lreach, int* __restrict__ parent,
                                                        const int* __restrict__ cell_root,
                                                        const uint8_t* __restrict__ strag,
                                                        const uint2* __restrict__ srange) {
  const int lane = threadIdx.x & 31;
  const int ns = (int)*ns_ptr;
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < ns; i += (gridDim.x * blockDim.x) >> 5) {
    const int s = slist[i];
    const int4 p = spos[s];
    const int nc = g.nc;
    const int cy = cell_coord(p.y, nc), cz = cell_coord(p.z, nc), tc = grid_col(g, p.x);
    const int rs = uf_root(parent, s);
    int cm = CELL_EMPTY;
    uint32_t t0 = 0, t1 = 0;
    uint2 sr = make_uint2(0, 0);
    if (lane < 27) {
      const XCells X = x_cells(g, tc);
      const int dz = lane / 9 - 1, dy = lane / 3 % 3 - 1, dx = lane % 3 - 1;
      const int gx = (p.x + g.x0) & (CSO_BOX - 1), gcx = cell_coord(gx, nc);
      const long long fx = dx < 0 ? gx - cell_lo(gcx, nc) + 1 : dx > 0 ? cell_lo(gcx + 1, nc) - gx : 0;
      const long long fy = dy < 0 ? p.y - cell_lo(cy, nc) + 1 : dy > 0 ? cell_lo(cy + 1, nc) - p.y : 0;
      const long long fz = dz < 0 ? p.z - cell_lo(cz, nc) + 1 : dz > 0 ? cell_lo(cz + 1, nc) - p.z : 0;
      const int col = dx < 0 ? (X.a < tc ? X.a : X.wl) : dx > 0 ? (X.b > tc ? X.b : X.wr) : tc;
      if (col >= 0 && fx * fx + fy * fy + fz * fz < (long long)lfof2) {
        int sh;
        const size_t c = grid_cell(g, wrap_yz(cz + dz, nc, sh), wrap_yz(cy + dy, nc, sh), col);
        t0 = g.start[c];
        t1 = g.start[c + 1];
        if (t0 < t1) cm = cell_root[t0];
        if (cm != CELL_EMPTY) {
          sr = srange[t0];
          if (uf_root(parent, cm) == rs) {
            t1 = t0;  // the main tree is the straggler's already
          } else if (t1 - t0 > 16u) {
            const int xq = dx < 0 && X.a == tc ? p.x + CSO_BOX : dx > 0 && X.b == tc ? p.x - CSO_BOX : p.x;
            x_trim(spos, t0, t1, xq - lreach, xq + lreach);
          }
        } else {
          t1 = t0;
        }
      }
    }
    // main trees: any link joins all of one
    uint32_t incl = warp_incl_u32(t1 - t0, lane);
    uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    const unsigned want = __ballot_sync(0xffffffffu, t1 > t0);
    unsigned hits = 0;
    for (uint32_t f0 = 0; f0 < total && hits != want; f0 += 32) {
      const uint32_t f = f0 + lane;
      const int r = flat_owner(incl, f) & 31;
      const uint32_t end = __shfl_sync(0xffffffffu, incl, r), hi = __shfl_sync(0xffffffffu, t1, r);
      bool hit = false;
      if (f < total && !(hits >> r & 1u)) {
        const uint32_t t = hi - (end - f);
        if (parent[t] >= 0 && !strag[t]) {
          const int4 q = spos[t];
          const int ex = fold21(p.x - q.x), ey = fold21(p.y - q.y), ez = fold21(p.z - q.z);
          hit = (uint32_t)(ex * ex) + (uint32_t)(ey * ey) + (uint32_t)(ez * ez) < lfof2;
        }
      }
      hits |= __reduce_or_sync(0xffffffffu, hit ? 1u << r : 0u);
    }
    if (hits >> lane & 1u) uf_unite(parent, rs, cm);
    // the cells' stragglers after this one, from their runs of the list
    incl = warp_incl_u32(sr.y - sr.x, lane);
    total = __shfl_sync(0xffffffffu, incl, 31);
    for (uint32_t f0 = 0; f0 < total; f0 += 32) {
      const uint32_t f = f0 + lane;
      const int r = flat_owner(incl, f) & 31;
      const uint32_t end = __shfl_sync(0xffffffffu, incl, r), hi = __shfl_sync(0xffffffffu, sr.y, r);
      if (f < total) {
        const int t = slist[hi - (end - f)];
        if (t > s) {
          const int4 q = spos[t];
          const int ex = fold21(p.x - q.x), ey = fold21(p.y - q.y), ez = fold21(p.z - q.z);
          if ((uint32_t)(ex * ex) + (uint32_t)(ey * ey) + (uint32_t)(ez * ez) < lfof2) uf_unite(parent, s, t);
        }
      }
    }
    __syncwarp();
  }
}

// root of every dense particle (-1 otherwise); smallest id per root
__global__ void k_fof_finish(int* __restrict__ parent, int n, const long long* __restrict__ sigma, long long T_L0,
                             const uint64_t* __restrict__ sid, int* __restrict__ root,
                             unsigned long long* __restrict__ minid) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int r = parent[s] < 0 ? -1 : uf_root(parent, s);
  root[s] = r;
  // smallest id per root: reduce over the lanes that share a root first
  const unsigned peers = __match_any_sync(__activemask(), r);
  const unsigned long long v = r >= 0 ? (unsigned long long)sid[s] : ~0ull;
  // (the high words first, the low words among the lanes that hold the smallest)
  const unsigned hi = __reduce_min_sync(peers, (unsigned)(v >> 32));
  const unsigned lo = __reduce_min_sync(peers, (unsigned)(v >> 32) == hi ? (unsigned)v : ~0u);
  if (r >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1) atomicMin(&minid[r], (unsigned long long)hi << 32 | lo);
}

}  // namespace

// the largest e >= 0 with e^2 < v (v >= 1): the farthest x offset at which
// a pair can still be closer than sqrt(v)
static int reach_below(long long v) {
  long long e = (long long)sqrt((double)v);
  while (e > 0 && e * e >= v) --e;
  while ((e + 1) * (e + 1) < v) ++e;
  return (int)e;
}

int cells_choose(long long b2, int* nc_out) {
  // largest nc with (2^21 / nc)^2 >= b2: cells at least as wide as b
  double b = sqrt((double)b2);
  long long nc = (long long)floor((double)CSO_BOX / b);
  while (nc > 1 && (long double)CSO_BOX * CSO_BOX < (long double)b2 * nc * nc) --nc;
  while ((long double)CSO_BOX * CSO_BOX >= (long double)b2 * (nc + 1) * (nc + 1)) ++nc;
  if (nc < 128) {
    cso_set_error("kernel radius b = %.0f grid units is too large (cells must be <= 2^14 units, u <= 40960)", b);
    return CSO_ERR_ARG;
  }
  if (nc > CSO_MAX_NC) {
    cso_set_error("kernel radius b = %.0f grid units is too small (more than %d cells per side)", b, CSO_MAX_NC);
    return CSO_ERR_ARG;
  }
  *nc_out = (int)nc;
  return CSO_OK;
}

int cells_check_dense(int nc) {
  if (nc > CSO_MAX_DENSE_NC) {
    cso_set_error("box too fine for one dense cell table (%d cells per side > %d): deliver it as x-slabs", nc,
                  CSO_MAX_DENSE_NC);
    return CSO_ERR_ARG;
  }
  return CSO_OK;
}

// Tables from this size on count in 16 bits first: the clearing, the atomics and
// the scan's two reads then move half the bytes.  Binning with a 262M-cell table
// 2.13 -> 1.92 ms (2^24 particles), 0.87 -> 0.67 (4M); with 34M cells 0.31 ->
// 0.28.  At 2M to 4M cells the launches of the unused recount cost more than is
// saved (0.039 -> 0.048 ms).
static constexpr long long HALF_CELLS = 1ll << 24;
static constexpr size_t HALF_ROOM = 1 << 20;  // left for the scan's sums: without it the count stays in 32 bits

int cells_bin(const int32_t* pos, const uint64_t* ids, long long n, const CellGrid& g, uint32_t* start,
              int4* spos, uint64_t* sid, int* bad, Workspace& ws, cudaStream_t st, uint32_t* inv) {
  long long ncell = (long long)g.ncols * g.nc * g.nc;
  size_t mark = ws.off;
  // the cell keys and arrival ranks live in the output spos (16 bytes per
  // particle) until k_cell_place overwrites it; the records (and the slot map
  // when inv is wanted) take workspace
  uint32_t* key = reinterpret_cast<uint32_t*>(spos);
  uint32_t* rank = key + n;
  BinRec* rec = ws.get<BinRec>(n);
  uint32_t* fin = inv ? ws.get<uint32_t>(n) : nullptr;
  if (!rec || (inv && !fin)) {
    cso_set_error("workspace exhausted in binning");
    return CSO_ERR_BUDGET;
  }
  const size_t half_bytes = sizeof(uint16_t) * ((size_t)ncell + 8) / 16 * 16;
  if (n > 0 && ncell + 1 >= HALF_CELLS && ws.off + half_bytes + HALF_ROOM <= ws.cap) {
    const size_t mark_half = ws.off;
    uint32_t* half = reinterpret_cast<uint32_t*>(ws.get<char>(half_bytes + sizeof(int)));
    int* over = reinterpret_cast<int*>(reinterpret_cast<char*>(half) + half_bytes);
    CSO_CUDA(cudaMemsetAsync(half, 0, half_bytes + sizeof(int), st));
    k_cell_count_half<<<CL(cdiv(n, 256)), 256, 0, st>>>(pos, n, g, key, rank, half, over, bad);
    const int gb = 4 * cso_sm_count();
    k_recount_clear<<<CL(gb), 512, 0, st>>>(start, ncell + 1, over);
    k_recount<<<CL(gb), 512, 0, st>>>(n, key, rank, start, over);
    CSO_CUDA(cudaGetLastError());
    CSO_TRY(scan_u32(start, ncell + 1, nullptr, ws, st, reinterpret_cast<const uint16_t*>(half), over));
    ws.off = mark_half;
  } else {
    CSO_CUDA(cudaMemsetAsync(start, 0, sizeof(uint32_t) * (ncell + 1), st));
    if (n > 0) {
      k_cell_count<<<CL(cdiv(n, 256)), 256, 0, st>>>(pos, n, g, key, rank, start, bad);
      CSO_CUDA(cudaGetLastError());
    }
    CSO_TRY(scan_u32(start, ncell + 1, nullptr, ws, st));
  }
  if (n > 0) {
    CellGrid gs = g;
    gs.start = start;
    k_cell_scatter<<<CL(cdiv(n, 256)), 256, 0, st>>>(pos, ids, n, gs, key, rank, start, rec, inv);
    k_cell_place<<<CL(cdiv(n, 256)), 256, 0, st>>>(n, rec, spos, sid, fin);
    if (inv) k_cell_inv<<<CL(cdiv(n, 256)), 256, 0, st>>>(n, fin, inv);
    CSO_CUDA(cudaGetLastError());
  }
  ws.off = mark;
  return CSO_OK;
}

// Widest x span of a warp's shared walk for cells of nc per side, and whether
// every staged squared distance stays below 2^31 (the signed form).  A staged
// pair is at most (span + 2) cells apart in x and 2 cells in y and z.
static void density_span(int nc, int* max_span, bool* is_signed) {
  const double side = ceil((double)CSO_BOX / nc);
  int sp = 0;
  for (int s = 2; s >= 0; --s)
    if (((s + 2.0) * (s + 2.0) + 8.0) * side * side < 4294967296.0) {
      sp = s;
      break;
    }
  // finer boxes share wider: up to nine cells while the signed form holds
  // (side 256: 1.3% of the pass with spans of up to 8 instead of 2)
  while (sp >= 2 && sp < 8 && ((sp + 3.0) * (sp + 3.0) + 8.0) * side * side < 2147483648.0) ++sp;
  *max_span = sp;
  *is_signed = ((sp + 2.0) * (sp + 2.0) + 8.0) * side * side < 2147483648.0;
}

int cells_density(const CellGrid& g, const int4* spos, int n, uint32_t b2, int include_self, long long* sigma,
                  unsigned long long* pairs, Workspace& ws, cudaStream_t st, const uint8_t* only) {
  if (n <= 0) return CSO_OK;
  const int nb = cdiv(n, DENS_WARPS * 32);
  const size_t mark = ws.off;
  uint32_t* order = ws.get<uint32_t>(nb);
  uint32_t* rank = ws.get<uint32_t>(nb);
  uint32_t* counts = ws.get<uint32_t>(DENS_CLASSES);
  uint8_t* cls = ws.get<uint8_t>(nb);
  if (!order || !rank || !counts || !cls) {
    cso_set_error("workspace exhausted in the density pass");
    return CSO_ERR_BUDGET;
  }
  int max_span;
  bool is_signed;
  density_span(g.nc, &max_span, &is_signed);
  const int reach = reach_below(b2);
  CSO_CUDA(cudaMemsetAsync(counts, 0, sizeof(uint32_t) * DENS_CLASSES, st));
  k_density_cost<<<CL(cdiv((long long)nb * DENS_WARPS, 256)), 256, 0, st>>>(g, spos, n, nb, cls, rank, counts);
  k_density_order<<<CL(cdiv(nb, 256)), 256, 0, st>>>(cls, rank, counts, nb, order);
  if (is_signed)
    k_density<true><<<CL(nb), DENS_WARPS * 32, 0, st>>>(g, spos, n, b2, reach, include_self, sigma, only, order,
                                                         max_span);
  else
    k_density<false><<<CL(nb), DENS_WARPS * 32, 0, st>>>(g, spos, n, b2, reach, include_self, sigma, only, order,
                                                          max_span);
  if (pairs) k_count_pairs<<<CL(cdiv(n, 256)), 256, 0, st>>>(g, spos, n, b2, pairs);
  CSO_CUDA(cudaGetLastError());
  ws.off = mark;
  return CSO_OK;
}

int cells_fof(const CellGrid& g, const int4* spos, int n, const long long* sigma, long long T_L0, uint32_t lfof2,
              const uint64_t* sid, int* parent, int* root, unsigned long long* minid, int* cell_root,
              Workspace& ws, cudaStream_t st) {
  if (n <= 0) return CSO_OK;
  const size_t mark = ws.off;
  const long long words = rank2_words(n);
  int* didx = ws.get<int>(n);
  int* clist = ws.get<int>(n);
  uint8_t* strag = ws.get<uint8_t>(n);
  int* slist = ws.get<int>(n);
  uint2* srange = ws.get<uint2>(n);
  // status words of the two lists' ranks, then the lists' lengths: dense
  // particles, cells that hold any, stragglers
  unsigned long long* status = ws.get<unsigned long long>((size_t)(2 * words + 2));
  if (!didx || !clist || !strag || !slist || !srange || !status) {
    cso_set_error("workspace exhausted in the FoF pass");
    return CSO_ERR_BUDGET;
  }
  uint32_t* counts = reinterpret_cast<uint32_t*>(status + 2 * words);
  const long long tiles = rank2_tiles(n);
  CSO_CUDA(cudaMemsetAsync(status, 0, sizeof(unsigned long long) * (size_t)(2 * words + 2), st));
  // launches over the lists are sized by n and blocks past the counts (read
  // on the device) return at once
  RANK2_LAUNCH(k_fof_lists, n, st, g, spos, n, sigma, T_L0, parent, cell_root, minid, didx, clist, counts, status, tiles,
               ws.patience);
  const uint32_t *nd = counts, *ncl = counts + 1, *ns = counts + 2;
  // pass one: bands inside cells; main trees and stragglers
  k_fof_sample<<<CL(cdiv(n, 256)), 256, 0, st>>>(g, spos, didx, nd, lfof2, parent);
  k_cell_main<<<CL(cdiv(n, 256)), 256, 0, st>>>(spos, g, clist, ncl, parent, cell_root);
  RANK2_LAUNCH(k_stragglers, n, st, spos, g, didx, counts, parent, cell_root, strag, slist, srange, status + words, tiles,
               ws.patience);
  // pass two: main trees of adjacent cells; pass three: stragglers
  const int lreach = reach_below(lfof2);
  k_fof_cells<<<CL(cso_sm_count() * 8), 256, 0, st>>>(g, spos, clist, ncl, lfof2, lreach, parent, cell_root, strag);
  k_fof_stragglers<<<CL(cso_sm_count() * 8), 256, 0, st>>>(g, spos, slist, ns, lfof2, lreach, parent, cell_root,
                                                           strag, srange);
  k_fof_finish<<<CL(cdiv(n, 256)), 256, 0, st>>>(parent, n, sigma, T_L0, sid, root, minid);
  CSO_CUDA(cudaGetLastError());
  ws.off = mark;
  return CSO_OK;
}
