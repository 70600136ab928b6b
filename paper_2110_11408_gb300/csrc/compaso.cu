// CompaSO levels (Sec. 2.2.2): the nucleus loop of steps 1-4 inside every
// group.  The nuclei come from the group's density peaks (peaks.cu), found
// beforehand by the whole GPU: the loop takes the peak first in key order
// (Sigma desc, id asc) among those still eligible until none is left.  The
// members of a group lie in cell order.
//
// Per nucleus:
//   pass A  squared distances d_j of the members to the nucleus;
//   select  R^2 = the smallest member distance d with n(<d)^2 u^6 < K d^3
//           (exact), found without a full sort: a 1024-bin histogram over a
//           window of d (first window binned by the threshold count
//           sqrt(K) d^1.5 / u^3, later windows linearly), the bins from the
//           first that could hold the answer on (by its interior count at its
//           largest d) are gathered into shared memory, up to 256 members, and
//           each counts the nearer ones; a larger bin alone is sorted and
//           scanned, or narrowed further when it holds more than 2048 members;
//           small groups are counted or sorted whole;
//   pass B  tentative membership / competitive reassignment (Eq. 3) and
//           eligibility of the peaks left.
//
// Groups above small_n (2,048) members are walked in tiles of 128 members,
// which are neighbours in space.  Where a group has several peaks, every tile
// has a bounding box, and a nucleus' passes visit only the tiles its radius
// can reach: the members of all tiles whose box is nearer than r are at least
// n(<r), so the first r (two steps an octave of r^2) at which that count is
// below the threshold density bounds the search, and R^2 bounds pass B.
#include <cooperative_groups.h>
#include <atomic>
#include <float.h>
#include <limits.h>

#include <algorithm>

#include "cells.cuh"
#include "compaso.cuh"

namespace {

constexpr int NB = 1024;      // histogram bins
constexpr int CAP = 2048;     // largest bin resolved by an in-block sort
constexpr int COUNT_N = 512;  // groups whose enclosed counts are counted directly

// ---------------------------------------------------------------------------
// exact predicate n^2 u^6 < K d^3 with K = Km 2^Ke (256-bit integers),
// behind a double-precision filter whose rounding error is far below 1e-12
// ---------------------------------------------------------------------------
struct U256 {
  unsigned long long w[4];
};

__device__ __forceinline__ void u256_mul(U256& a, unsigned long long b) {
  unsigned long long carry = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    unsigned long long lo = a.w[i] * b;
    unsigned long long hi = __umul64hi(a.w[i], b);
    lo += carry;
    hi += lo < carry;
    a.w[i] = lo;
    carry = hi;
  }
}

__device__ __forceinline__ void u256_shl(U256& a, int s) {
  while (s >= 64) {
    a.w[3] = a.w[2];
    a.w[2] = a.w[1];
    a.w[1] = a.w[0];
    a.w[0] = 0;
    s -= 64;
  }
  if (s) {
    a.w[3] = (a.w[3] << s) | (a.w[2] >> (64 - s));
    a.w[2] = (a.w[2] << s) | (a.w[1] >> (64 - s));
    a.w[1] = (a.w[1] << s) | (a.w[0] >> (64 - s));
    a.w[0] <<= s;
  }
}

__device__ __forceinline__ bool u256_less(const U256& a, const U256& b) {
  for (int i = 3; i >= 0; --i)
    if (a.w[i] != b.w[i]) return a.w[i] < b.w[i];
  return false;
}

__device__ __noinline__ bool pred_exact(unsigned long long n, unsigned long long d, const PredConst& c) {
  U256 L = {{n, 0, 0, 0}}, R = {{c.Km, 0, 0, 0}};
  u256_mul(L, n);
#pragma unroll
  for (int i = 0; i < 6; ++i) u256_mul(L, c.u);
  u256_mul(R, d);
  u256_mul(R, d);
  u256_mul(R, d);
  if (c.Ke > 0) u256_shl(R, c.Ke);
  else if (c.Ke < 0) u256_shl(L, -c.Ke);
  return u256_less(L, R);
}

// The enclosed count n inside squared radius d is below the level's density.
// The threshold count d^1.5 sqrt(K) / u^3 in float decides all but the counts
// within 1e-5 of it (its relative error is below 1e-6): double precision runs
// at a fiftieth of the float rate here.
__device__ __forceinline__ bool pred(unsigned long long n, unsigned long long d, const PredConst& c) {
  const float fd = (float)d, t = fd * sqrtf(fd) * c.bin_scale0, fn = (float)n;
  if (fn < t * (1.f - 1e-5f)) return true;
  if (fn > t * (1.f + 1e-5f)) return false;
  double L = (double)n * (double)n * c.u6;
  double dd = (double)d;
  double R = c.K * (dd * dd * dd);
  if (L < R * (1.0 - 1e-12)) return true;
  if (L > R * (1.0 + 1e-12)) return false;
  return pred_exact(n, d, c);
}

// smallest D > dmax with pred(n, D): the enclosed count stays n beyond the
// farthest member (single thread)
__device__ long long exhaust_radius(unsigned long long n, long long dmax, const PredConst& c) {
  unsigned long long lo = (unsigned long long)dmax, hi = lo + 1;
  while (!pred(n, hi, c)) hi *= 2;
  while (hi - lo > 1) {
    unsigned long long mid = lo + (hi - lo) / 2;
    if (pred(n, mid, c)) hi = mid;
    else lo = mid;
  }
  return (long long)hi;
}

__device__ __forceinline__ int mi(int v) {
  if (v >= CSO_HALF) return v - CSO_BOX;
  if (v < -CSO_HALF) return v + CSO_BOX;
  return v;
}

__device__ __forceinline__ long long dist2(int4 a, int4 b) {
  long long dx = mi(a.x - b.x), dy = mi(a.y - b.y), dz = mi(a.z - b.z);
  return dx * dx + dy * dy + dz * dz;
}

__device__ __forceinline__ unsigned warp_incl(unsigned v) {
  int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// block exclusive scan (NT threads), returns total
template <int NT>
__device__ unsigned block_scan(unsigned v, unsigned& excl, unsigned* sw) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned inc = warp_incl(v);
  if (lane == 31) sw[w] = inc;
  __syncthreads();
  if (w == 0) {
    unsigned s = lane < NT / 32 ? sw[lane] : 0;
    unsigned si = warp_incl(s);
    if (lane < NT / 32) sw[lane] = si - s;
    if (lane == 31) sw[32] = si;
  }
  __syncthreads();
  excl = inc - v + sw[w];
  unsigned tot = sw[32];
  __syncthreads();
  return tot;
}

__device__ void bitonic_sort(long long* a, int m) {  // m power of two
  for (int k = 2; k <= m; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < m; i += blockDim.x) {
        int l = i ^ j;
        if (l > i) {
          long long x = a[i], y = a[l];
          bool up = (i & k) == 0;
          if ((x > y) == up) {
            a[i] = y;
            a[l] = x;
          }
        }
      }
      __syncthreads();
    }
}

struct SelShared {
  unsigned cnt[NB];
  unsigned clo[NB];
  long long list[CAP];
  unsigned sw[33];
  int best;
  int nlist;
  unsigned long long pick;      // nearest listed member that qualifies
  unsigned long long lo, hi;    // smallest and largest distance of a bin too big to list
  unsigned long long dmax_all;  // farthest member visited
};

// In the sorted list s[0..m) with n(<s[0]) = base, the first element whose
// strictly-enclosed count satisfies the predicate; returns its index or m.
__device__ int scan_sorted(const long long* s, int m, unsigned long long base, const PredConst& c, int* best) {
  if (threadIdx.x == 0) *best = m;
  __syncthreads();
  for (int k = threadIdx.x; k < m; k += blockDim.x) {
    int f = k;
    while (f > 0 && s[f - 1] == s[k]) --f;
    if (pred(base + (unsigned long long)f, (unsigned long long)s[k], c)) atomicMin(best, k);
  }
  __syncthreads();
  int r = *best;
  __syncthreads();
  return r;
}

// A gather takes the bins from the first candidate on that hold up to RANGE
// members together: the candidates mostly fail one after the other, and each
// gather is a pass over the members.  A candidate of more members, or of more
// than the list may hold, is taken alone, so that a window narrowed to it shrinks.
// Level 2 of 2^18 particles 0.197 -> 0.179 ms, of the uneven groups 3.29 -> 3.25,
// level 1 there 1.69 -> 1.64; a RANGE of 64 or 128 is no faster.
constexpr int RANGE = 256;

// the last bin of the gather that starts at bin b
__device__ __forceinline__ int range_end(const SelShared& S, int b) {
  const unsigned top = S.clo[b] + RANGE;
  int lo = b, hi = NB - 1;
  while (lo < hi) {
    const int x = (lo + hi + 1) >> 1;
    if (S.clo[x] + S.cnt[x] <= top) lo = x;
    else hi = x - 1;
  }
  return lo;
}

// The smallest of the m <= RANGE distances s, unsorted, whose strictly-enclosed
// count satisfies the predicate (base members are nearer than all of s), every
// one counting the nearer ones; ~0 if none.  S.pick is ~0 at the start.
__device__ unsigned long long pick_listed(const long long* s, int m, unsigned long long base, const PredConst& c,
                                          SelShared& S) {
  if ((int)threadIdx.x < m) {
    const long long d = s[threadIdx.x];
    unsigned nearer = 0;
    for (int j = 0; j < m; ++j) nearer += s[j] < d;
    if (pred(base + nearer, (unsigned long long)d, c)) atomicMin(&S.pick, (unsigned long long)d);
  }
  __syncthreads();
  const unsigned long long r = S.pick;
  __syncthreads();
  return r;
}

__device__ __forceinline__ int pow2_at_least(int m) {
  int p = 1;
  while (p < m) p <<= 1;
  return p;
}

// Bin of distance d in the first window of the select.  Both binnings are
// monotone in d, and the select only prunes with the exact predicate at an
// upper bound of each bin's distances, so both give the same R^2:
//   * threshold-count bins (default): bin = sqrt(K) d^1.5 / u^3 / w with
//     w = n / (nb - 1) members of threshold count per bin;
//   * radial bins (the paper's cell-bounded search, Sec. 2.3.4): bins of
//     width sqrt(3)/3 cell sides in r; a bin is skipped when the members
//     inside it, placed at its outer edge, still meet the threshold.
__device__ __forceinline__ int first_bin(unsigned long long d, const PredConst& c, float scale0, int nb) {
  const float f = (float)d;
  const float g = c.radial ? sqrtf(f) * c.rbin_inv_w : f * sqrtf(f) * scale0;
  return g < (float)(nb - 1) ? (int)g : nb - 1;
}

// bins per unit of first_bin's threshold count: w members of threshold per
// bin, for the whole group or for a search bounded by lim
__device__ __forceinline__ float bin_scale(int n, unsigned long long lim, const PredConst& c, int nb) {
  float cnt = (float)n;
  if (lim) {
    const float f = (float)lim;
    cnt = fminf(cnt, f * sqrtf(f) * c.bin_scale0 + 2.f);
  }
  return c.bin_scale0 / ceilf(cnt / (float)(nb - 1));
}

// A window of the select: members with wlo <= d <= whi in nb bins, by
// first_bin (mode 0) or linearly (mode 1).
struct Window {
  unsigned long long wlo, whi, base;  // base = members below wlo
  int mode;
};

__device__ __forceinline__ int window_bin(const Window& W, unsigned long long d, const PredConst& c, float scale0,
                                          int nb) {
  if (W.mode == 0) return first_bin(d, c, scale0, nb);
  const unsigned long long span = W.whi - W.wlo + 1;
  return (int)(((d - W.wlo) * (unsigned long long)nb) / span);
}

// An upper bound of the distances that fall into bin b of the window, at
// most top (the inverse of first_bin in float, raised by far more than its
// rounding; the last bin of mode 0 is open).
__device__ __forceinline__ unsigned long long bin_top(const Window& W, int b, const PredConst& c, float scale0, int nb,
                                                      unsigned long long top) {
  if (b >= nb - 1) return top;
  unsigned long long e;
  if (W.mode == 0) {
    const float g = (float)(b + 1);
    const float f = c.radial ? (g / c.rbin_inv_w) * (g / c.rbin_inv_w) : powf(g / scale0, 2.f / 3.f);
    e = f < 9e18f ? (unsigned long long)(f * (1.f + 1e-4f)) + 1 : top;
  } else {
    const unsigned long long span = W.whi - W.wlo + 1;
    e = W.wlo + (unsigned long long)(b + 1) * (span / nb + 1);
  }
  return e < top ? e : top;
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, v, o);
    v = t > v ? t : v;
  }
  return v;
}

// ---------------------------------------------------------------------------
// tiles of a group: TILE consecutive members, their bounding boxes and the
// passes over the tiles within reach of a nucleus
// ---------------------------------------------------------------------------
constexpr int TILE = 128;
constexpr int TILE_LIST = 2048;  // tiles in reach that a block keeps as a list
constexpr int LEVELS = 88;  // squared radii tried for the search bound: two per octave up to 2^43

__device__ __forceinline__ int fold21(int v) { return (int)((unsigned)v << 11) >> 11; }  // nearest image

// squared radius at the lower edge of level k, and the level of d
__device__ __forceinline__ unsigned long long level_edge(int k) {
  return k < 2 ? (unsigned long long)k : (k & 1 ? 3ull << (k / 2 - 1) : 1ull << (k / 2));
}
__device__ __forceinline__ int level_of(unsigned long long d) {
  if (d < 2) return (int)d;
  const int m = 63 - __clzll((long long)d);
  return 2 * m + (int)((d >> (m - 1)) & 1);
}

// Boxes of runs of `per` tiles (a multiple of 32), for a block that looks over
// more tiles than two a thread.  Every tile's box of a group of 1.9M members is
// 470 KB out of L2, 5.6 us a look; through its 456 runs the look takes 3.1.
constexpr int SUPERS = 512;
struct SuperBoxes {
  int lo[3][SUPERS], hi[3][SUPERS];
  int n, per;  // n = 0: none
};

// The tiles a CTA owns: rank, rank + cs, ... of the group's nt (cs = 1 for a block).
struct Tiles {
  int nt, rank, cs;
  const int4* lo;  // boxes of the group's tiles, offsets from the group's first member; null: none
  const int4* hi;
  int4 q;          // the nucleus in those offsets
  const uint32_t* list;  // the group's tiles in reach of the nucleus, or
  int nlist;             // -1: no list
  __device__ __forceinline__ int own() const { return nt > rank ? (nt - rank + cs - 1) / cs : 0; }
};

__device__ __forceinline__ unsigned long long axis_gap2(int q, int lo, int hi) {
  // over the three images of the box's interval, which is shorter than a box side
  int g = max(max(lo - q, q - hi), 0);
  g = min(g, max(max(lo + CSO_BOX - q, q - hi - CSO_BOX), 0));
  g = min(g, max(max(lo - CSO_BOX - q, q - hi + CSO_BOX), 0));
  return (unsigned long long)g * (unsigned long long)g;
}

// squared distance from the nucleus to tile t's box: no member of it is nearer
__device__ __forceinline__ unsigned long long tile_gap2(const Tiles& T, int t) {
  const int4 a = T.lo[t], b = T.hi[t];
  return axis_gap2(T.q.x, a.x, b.x) + axis_gap2(T.q.y, a.y, b.y) + axis_gap2(T.q.z, a.z, b.z);
}

// f(j) for every member j < n of the CTA's tiles nearer than lim (0: of all
// its tiles): of those on the list if there is one, else warps take chunks
// of up to 32 tiles that lie a whole chunk count apart, so that the tiles in
// reach, neighbours of one another, spread over the warps.
template <class F>
__device__ __forceinline__ void tile_members(int t, int n, F f) {
#pragma unroll
  for (int k = 0; k < TILE / 32; ++k) {
    const int j = t * TILE + k * 32 + (threadIdx.x & 31);
    if (j < n) f(j);
  }
}

template <class F>
__device__ __forceinline__ void for_members(const Tiles& T, int n, unsigned long long lim, F f) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (T.nlist >= 0) {
    for (int i = threadIdx.x >> 5; i < T.nlist; i += nw) tile_members((int)T.list[i], n, f);
    return;
  }
  const int own = T.own();
  const int per = min(32, (own + nw - 1) / nw);
  const int nchunk = per > 0 ? (own + per - 1) / per : 0;
  for (int c = threadIdx.x >> 5; c < nchunk; c += nw) {
    const int i = lane * nchunk + c;
    const bool act = lane < per && i < own && (!lim || tile_gap2(T, T.rank + i * T.cs) < lim);
    for (unsigned m = __ballot_sync(0xffffffffu, act); m; m &= m - 1)
      tile_members(T.rank + ((__ffs(m) - 1) * nchunk + c) * T.cs, n, f);
  }
}

// The CTA's tiles nearer than lim, listed (T.nlist = -1 if they are too many):
// one look at every box, which the passes that follow then need not repeat.
__device__ __forceinline__ void list_tiles(Tiles& T, unsigned long long lim, uint32_t* list, int* count,
                                           const SuperBoxes* sup = nullptr) {
  if (threadIdx.x == 0) *count = 0;
  __syncthreads();
  const auto take = [&](int t) {
    if (tile_gap2(T, t) >= lim) return;
    const int k = atomicAdd(count, 1);
    if (k < TILE_LIST) list[k] = (uint32_t)t;
  };
  if (sup && sup->n > 0) {
    // a warp opens every 32nd run, so that neighbours spread over the warps
    const SuperBoxes& B = *sup;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int s0 = threadIdx.x >> 5; s0 < B.n; s0 += 32 * nw) {
      const int s = s0 + lane * nw;
      const bool in = s < B.n && axis_gap2(T.q.x, B.lo[0][s], B.hi[0][s]) + axis_gap2(T.q.y, B.lo[1][s], B.hi[1][s]) +
                                            axis_gap2(T.q.z, B.lo[2][s], B.hi[2][s]) < lim;
      for (unsigned m = __ballot_sync(0xffffffffu, in); m; m &= m - 1) {
        const int first = (s0 + (__ffs(m) - 1) * nw) * B.per;
        for (int t = first + lane; t < min(first + B.per, T.nt); t += 32) take(t);
      }
    }
  } else {
    const int own = T.own();
    for (int i = threadIdx.x; i < own; i += blockDim.x) take(T.rank + i * T.cs);
  }
  __syncthreads();
  const int k = *count;
  T.list = list;
  T.nlist = k <= TILE_LIST ? k : -1;
  __syncthreads();
}

// boxes of the CTA's own tiles, a warp per tile
__device__ void tile_boxes(const Tiles& T, const int4* __restrict__ epos, int n, int4* lo, int4* hi) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int4 ref = epos[0];
  for (int i = threadIdx.x >> 5; i < T.own(); i += nw) {
    const int t = T.rank + i * T.cs;
    int a[3] = {INT_MAX, INT_MAX, INT_MAX}, b[3] = {INT_MIN, INT_MIN, INT_MIN};
#pragma unroll
    for (int k = 0; k < TILE / 32; ++k) {
      const int j = t * TILE + k * 32 + lane;
      if (j >= n) continue;
      const int4 p = epos[j];
      const int o[3] = {fold21(p.x - ref.x), fold21(p.y - ref.y), fold21(p.z - ref.z)};
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        a[x] = min(a[x], o[x]);
        b[x] = max(b[x], o[x]);
      }
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      a[x] = __reduce_min_sync(0xffffffffu, a[x]);
      b[x] = __reduce_max_sync(0xffffffffu, b[x]);
    }
    if (lane == 0) {
      lo[t] = make_int4(a[0], a[1], a[2], 0);
      hi[t] = make_int4(b[0], b[1], b[2], 0);
    }
  }
}

// The squared radius that bounds the nucleus' search: the first level edge e
// at which the members of all tiles nearer than e are below the threshold
// density (then so are the members nearer than e, and R^2 is the smallest
// member distance below e that qualifies, or the first one past it); 0 if
// there is none.  Every thread of the block calls it; h: LEVELS counters.
__device__ unsigned long long search_bound(const Tiles& T, int n, const PredConst& c, unsigned* h, int* best) {
  for (int k = threadIdx.x; k < LEVELS; k += blockDim.x) h[k] = 0;
  if (threadIdx.x == 0) *best = LEVELS;
  __syncthreads();
  for (int t = threadIdx.x; t < T.nt; t += blockDim.x)
    atomicAdd(&h[min(level_of(tile_gap2(T, t)), LEVELS - 1)], (unsigned)min(TILE, n - t * TILE));
  __syncthreads();
  for (int k = 1 + threadIdx.x; k < LEVELS; k += blockDim.x) {
    unsigned long long cnt = 0;
    for (int q = 0; q < k; ++q) cnt += h[q];
    if (pred(cnt, level_edge(k), c)) atomicMin(best, k);
  }
  __syncthreads();
  const int k = *best;
  __syncthreads();
  return k < LEVELS ? level_edge(k) : 0;
}

// R^2 of nucleus pc over the n members at epos[0..n); the distances of the
// members the search visited are left in ed (null: computed again where they
// are needed).  lim > 0 bounds the search (the
// boxes of T are there): if nothing qualifies below lim, the answer is -1, or
// with `whole` the search goes on over all members.
template <int NT>
__device__ long long r_search(const int4* __restrict__ epos, long long* __restrict__ ed, int n, int4 pc,
                              const PredConst& c, SelShared& S, const int small_n, const int cap, const int nb,
                              Tiles& T, unsigned long long lim, bool whole) {
  const int tid = threadIdx.x;
  if (n <= small_n && n <= COUNT_N) {
    // every member's strictly enclosed count, counted directly: n(<d_i) =
    // #{j : d_j < d_i}; R^2 is the smallest d_i whose count satisfies the
    // predicate (2 barriers instead of a sort)
    for (int j = tid; j < n; j += blockDim.x) {
      long long d = dist2(pc, epos[j]);
      ed[j] = d;
      S.list[j] = d;
    }
    if (tid == 0) S.dmax_all = ~0ull;
    __syncthreads();
    unsigned long long best = ~0ull, dmax = 0;
    for (int i = tid; i < n; i += blockDim.x) {
      const long long di = S.list[i];
      unsigned cnt = 0;
      for (int j = 0; j < n; ++j) cnt += S.list[j] < di;
      if (pred(cnt, (unsigned long long)di, c) && (unsigned long long)di < best) best = (unsigned long long)di;
      dmax = (unsigned long long)di > dmax ? (unsigned long long)di : dmax;
    }
    atomicMin(&S.dmax_all, best);
    if (tid == 0) S.hi = 0;
    __syncthreads();
    atomicMax(&S.hi, dmax);
    __syncthreads();
    long long r = (long long)S.dmax_all;
    const long long far = (long long)S.hi;
    __syncthreads();
    if (S.dmax_all == ~0ull || r < 0) {
      if (tid == 0) S.list[0] = exhaust_radius((unsigned long long)n, far, c);
      __syncthreads();
      r = S.list[0];
      __syncthreads();
    }
    return r;
  }
  if (n <= small_n) {
    for (int j = tid; j < n; j += blockDim.x) {
      long long d = dist2(pc, epos[j]);
      ed[j] = d;
      S.list[j] = d;
    }
    int m = pow2_at_least(n);
    for (int j = n + tid; j < m; j += blockDim.x) S.list[j] = LLONG_MAX;
    __syncthreads();
    bitonic_sort(S.list, m);
    int k = scan_sorted(S.list, n, 0, c, &S.best);
    long long r;
    if (k < n) r = S.list[k];
    else r = S.list[n - 1];  // sentinel: exhaustion below
    __syncthreads();
    if (k >= n) {
      if (tid == 0) S.list[0] = exhaust_radius((unsigned long long)n, r, c);
      __syncthreads();
      r = S.list[0];
      __syncthreads();
    }
    return r;
  }

  // ---- windowed histogram select ----
  Window W{0, lim ? lim - 1 : ~0ull, 0, 0};
  float scale0 = bin_scale(n, lim, c, nb);
  bool first_pass = true;
  while (true) {
    for (int b = tid; b < NB; b += blockDim.x) S.cnt[b] = 0;
    if (tid == 0) {
      S.lo = ~0ull;
      S.hi = 0;
      if (first_pass) S.dmax_all = 0;
    }
    __syncthreads();
    unsigned long long dmax = 0;  // this thread's farthest member (first pass)
    for_members(T, n, lim, [&](int j) {
      unsigned long long d;
      if (first_pass) {
        d = (unsigned long long)dist2(pc, epos[j]);
        if (ed) ed[j] = (long long)d;
        dmax = d > dmax ? d : dmax;
      } else {
        d = (unsigned long long)(ed ? ed[j] : dist2(pc, epos[j]));
      }
      if (d >= W.wlo && d <= W.whi) atomicAdd(&S.cnt[window_bin(W, d, c, scale0, nb)], 1u);
    });
    if (first_pass) {
      // one shared atomic per warp (per member it serialised on one address)
      const unsigned long long m = warp_max_u64(dmax);
      if ((tid & 31) == 0) atomicMax(&S.dmax_all, m);
    }
    __syncthreads();
    first_pass = false;
    const unsigned long long dtop = S.dmax_all < W.whi ? S.dmax_all : W.whi;
    // interior counts
    {
      constexpr int per = NB / NT;
      unsigned loc[per];
      unsigned s = 0;
#pragma unroll
      for (int q = 0; q < per; ++q) {
        loc[q] = S.cnt[tid * per + q];
        s += loc[q];
      }
      unsigned excl;
      unsigned tot = block_scan<NT>(s, excl, S.sw);
      unsigned run = excl;
#pragma unroll
      for (int q = 0; q < per; ++q) {
        S.clo[tid * per + q] = run;
        run += loc[q];
      }
      if (tid == 0) S.nlist = (int)tot;  // members in the window
      __syncthreads();
    }
    const unsigned in_window = (unsigned)S.nlist;
    int from = 0;
    bool narrowed = false;
    while (true) {
      // first bin >= from that could hold the answer
      if (tid == 0) S.best = NB;
      __syncthreads();
      for (int b = from + tid; b < NB; b += blockDim.x)
        if (S.cnt[b] && pred(W.base + S.clo[b], bin_top(W, b, c, scale0, nb, dtop), c)) atomicMin(&S.best, b);
      __syncthreads();
      // read the chosen bin before the barrier: the next window pass rewrites it
      const int b = S.best;
      unsigned long long cb = 0;
      unsigned cntb = 0;
      int last = b;
      if (b < NB) {
        cb = W.base + S.clo[b];
        cntb = S.cnt[b];
        if (cntb <= (unsigned)min(cap, RANGE)) last = range_end(S, b);
      }
      __syncthreads();
      if (b == NB) break;  // nothing in this window
      const bool listed = cntb <= (unsigned)cap;
      if (listed && tid == 0) {
        S.nlist = 0;
        S.pick = ~0ull;
      }
      if (listed) __syncthreads();
      unsigned long long lo = ~0ull, hi = 0;
      for_members(T, n, lim, [&](int j) {
        const unsigned long long d = (unsigned long long)(ed ? ed[j] : dist2(pc, epos[j]));
        if (d < W.wlo || d > W.whi) return;
        const int x = window_bin(W, d, c, scale0, nb);
        if (x < b || x > last) return;
        if (listed) {
          S.list[atomicAdd(&S.nlist, 1)] = (long long)d;
        } else {
          lo = d < lo ? d : lo;
          hi = d > hi ? d : hi;
        }
      });
      if (listed) {
        __syncthreads();
        int m = S.nlist;
        if (m <= RANGE) {
          const unsigned long long r = pick_listed(S.list, m, cb, c, S);
          if (r != ~0ull) return (long long)r;
          from = last + 1;
          continue;
        }
        int p2 = pow2_at_least(m);
        for (int j = m + tid; j < p2; j += blockDim.x) S.list[j] = LLONG_MAX;
        __syncthreads();
        bitonic_sort(S.list, p2);
        int k = scan_sorted(S.list, m, cb, c, &S.best);
        if (k < m) {
          long long r = S.list[k];
          __syncthreads();
          return r;
        }
        from = b + 1;
        continue;
      }
      // too many members in the bin: narrow the window to it
      hi = warp_max_u64(hi);
      lo = ~warp_max_u64(~lo);
      if ((tid & 31) == 0) {
        atomicMin(&S.lo, lo);
        atomicMax(&S.hi, hi);
      }
      __syncthreads();
      lo = S.lo;
      hi = S.hi;
      __syncthreads();
      if (lo == hi) {
        // one distinct value: its enclosed count is cb, and it qualifies or not
        if (pred(cb, lo, c)) return (long long)lo;
        if (tid == 0) {
          S.lo = ~0ull;
          S.hi = 0;
        }
        from = b + 1;
        continue;
      }
      W = Window{lo, hi, cb, 1};
      narrowed = true;
      break;
    }
    if (narrowed) continue;
    // nothing in the window: move past it
    const unsigned long long top = lim ? lim - 1 : S.dmax_all;
    if (W.whi < top) {
      W = Window{W.whi + 1, top, W.base + in_window, 1};
    } else if (lim && !whole) {
      return -1;
    } else if (lim) {  // nothing below the bound: all members, from the start
      __syncthreads();  // every thread has read dmax_all
      lim = 0;
      T.nlist = -1;
      scale0 = bin_scale(n, 0, c, nb);
      W = Window{0, ~0ull, 0, 0};
      first_pass = true;
    } else {
      break;
    }
  }
  long long r = 0;
  if (tid == 0) S.list[0] = exhaust_radius((unsigned long long)n, (long long)S.dmax_all, c);
  __syncthreads();
  r = S.list[0];
  __syncthreads();
  return r;
}

// Nuclei after a group's first mostly have small radii: squared radii to try
// before the bounded search of the whole group, those whose threshold counts
// are 256 and 4,096 (a try that finds nothing costs a fraction of the next).
constexpr int TRIES = 2;
__device__ __forceinline__ unsigned long long try_bound(int k, const PredConst& c) {
  const float f = powf((k ? 4096.f : 256.f) / c.bin_scale0, 2.f / 3.f);
  return f < 9e18f ? (unsigned long long)f + 1 : 0;
}

// ---------------------------------------------------------------------------
// A try over so few tiles that every lane holds its members' distances: H tiles
// a warp.  For the nuclei of the 16-CTA clusters, which are chosen one after the
// other and mostly end in the first try, 25 tiles: 11.8 -> 7.5 us a try, and with
// the runs above level 2 of the uneven groups (1.9M members in the largest, 193
// nuclei) 4.96 -> 3.31 ms.  The smaller tiers gain nothing by it (8-CTA clusters
// 0.334 -> 0.342 ms, blocks 0.197 -> 0.210: their tries are over fewer tiles or
// the registers are missed) and stay on r_search.
// r_search's select with one histogram over the window below lim, without its
// second pass over memory and its sort: the members are put in bin order, and
// each one of a bin that may hold the answer counts the nearer ones of its bin,
// all bins at once.  R^2, -1 if nothing below lim qualifies, or -2 if the answer
// may lie in or behind a bin of more than HELD_BIN members or past the list.
constexpr int HELD = 2;
constexpr unsigned HELD_BIN = 128;

template <int NT>
__device__ __forceinline__ bool held_fits(const Tiles& T) {
  return T.nlist >= 0 && T.nlist <= HELD * (NT / 32);
}

template <int NT>
__device__ long long held_search(const int4* __restrict__ epos, int n, int4 pc, const PredConst& c, SelShared& S, int nb,
                                 const Tiles& T, unsigned long long lim) {
  constexpr int per = NB / NT, H = HELD, TL = TILE / 32;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const float scale0 = bin_scale(n, lim, c, nb);
  const Window W{0, lim - 1, 0, 0};
  unsigned long long d[H][TL];  // ~0: none
  unsigned at[H][TL];           // arrival in its bin << 10 | bin
  static_assert(NB <= 1024 && H * NT * TL <= 1 << 21, "packed");
#pragma unroll
  for (int q = 0; q < per; ++q) S.cnt[tid * per + q] = 0;
  if (tid == 0) {
    S.best = NB;
    S.lo = ~0ull;
  }
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const int i = w + h * (NT / 32);
    const int t = i < T.nlist ? (int)T.list[i] : -1;
#pragma unroll
    for (int k = 0; k < TL; ++k) {
      const int j = t * TILE + k * 32 + lane;
      d[h][k] = t >= 0 && j < n ? (unsigned long long)dist2(pc, epos[j]) : ~0ull;
    }
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int k = 0; k < TL; ++k)
      if (d[h][k] < lim) {
        const int b = window_bin(W, d[h][k], c, scale0, nb);
        at[h][k] = atomicAdd(&S.cnt[b], 1u) << 10 | (unsigned)b;
      }
  __syncthreads();
  unsigned loc[per], sum = 0;
#pragma unroll
  for (int q = 0; q < per; ++q) {
    loc[q] = S.cnt[tid * per + q];
    sum += loc[q];
  }
  unsigned first;
  block_scan<NT>(sum, first, S.sw);
#pragma unroll
  for (int q = 0; q < per; ++q) {
    const int b = tid * per + q;
    // could a member of the bin qualify?
    bool ok = loc[q] && pred(first, bin_top(W, b, c, scale0, nb, W.whi), c);
    if (ok && (loc[q] > HELD_BIN || first + loc[q] > CAP)) {
      atomicMin(&S.best, b);
      ok = false;
    }
    S.clo[b] = first | (ok ? 1u << 31 : 0u);
    first += loc[q];
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int k = 0; k < TL; ++k)
      if (d[h][k] < lim) {
        const unsigned f = S.clo[at[h][k] & 1023u];
        if (f >> 31) S.list[(f & 0x7fffffffu) + (at[h][k] >> 10)] = (long long)d[h][k];
      }
  __syncthreads();
  unsigned long long mine = ~0ull;
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int k = 0; k < TL; ++k)
      if (d[h][k] < lim) {
        const unsigned b = at[h][k] & 1023u, f = S.clo[b];
        if (!(f >> 31) || d[h][k] >= mine) continue;
        const unsigned lo = f & 0x7fffffffu, hi = lo + S.cnt[b];
        unsigned nearer = lo;
        for (unsigned j = lo; j < hi; ++j) nearer += S.list[j] < (long long)d[h][k];
        if (pred(nearer, d[h][k], c)) mine = d[h][k];
      }
  if (__any_sync(0xffffffffu, mine != ~0ull)) {
    mine = ~warp_max_u64(~mine);
    if (lane == 0) atomicMin(&S.lo, mine);
  }
  __syncthreads();
  const unsigned long long r = S.lo;
  const int big = S.best;
  if (big < NB && (r == ~0ull || window_bin(W, r, c, scale0, nb) > big)) {
    __syncthreads();  // the search that follows clears the shared words
    return -2;
  }
  return r == ~0ull ? -1 : (long long)r;
}

// ---------------------------------------------------------------------------
// the choice of the next nucleus among a group's peaks
// ---------------------------------------------------------------------------
struct Best {
  long long sig;
  uint64_t id;
  int i;  // -1: none
};

// Key order: Sigma desc, id asc, and cell order where a caller's ids repeat (the
// list of peaks is in no order).  pos: the group's peaks.
__device__ __forceinline__ void best_of(Best& a, const Best& b, const int4* pos) {
  if (b.i < 0) return;
  bool before = a.i < 0 || b.sig > a.sig || (b.sig == a.sig && b.id < a.id);
  if (a.i >= 0 && b.sig == a.sig && b.id == a.id) before = pos[b.i].w < pos[a.i].w;
  if (before) a = b;
}

__device__ __forceinline__ void warp_best(Best& a, const int4* pos) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    Best b;
    b.sig = __shfl_xor_sync(0xffffffffu, a.sig, o);
    b.id = __shfl_xor_sync(0xffffffffu, a.id, o);
    b.i = __shfl_xor_sync(0xffffffffu, a.i, o);
    best_of(a, b, pos);
  }
}

struct PickShared {
  Best w[32];
  Best all;
};

// Marks the peaks that nucleus pc of squared radius R2 makes ineligible (step
// 1: nearer than alpha R; `cur` is the nucleus itself) and returns the first
// of the others in key order, or -1.  cur < 0: the first choice.  Each CTA of
// a cluster calls it with the same arguments and gets the same answer.  The
// flags of up to 64 peaks per thread are bits of gone; those of longer lists
// are in memory, and there a cluster's CTAs must not be a nucleus apart.
__device__ __forceinline__ bool private_flags(int m) { return m <= 64 * (int)blockDim.x; }

__device__ int next_nucleus(const LevelArgs& a, unsigned p0, int m, int cur, int4 pc, long long R2,
                            unsigned long long& gone, PickShared& K) {
  const long long anum2 = (long long)a.alpha_num * a.alpha_num, aden2 = (long long)a.alpha_den * a.alpha_den;
  const bool priv = private_flags(m);
  const int4* pos = a.peaks.pos + p0;
  Best mine{0, 0, -1};
  for (int i = threadIdx.x, k = 0; i < m; i += blockDim.x, ++k) {
    if (cur >= 0) {
      if (priv ? gone >> k & 1 : a.peaks.out[p0 + i] != 0) continue;
      if (i == cur || (__int128)aden2 * dist2(pc, pos[i]) < (__int128)anum2 * R2) {
        if (priv) gone |= 1ull << k;
        else a.peaks.out[p0 + i] = 1;
        continue;
      }
    }
    best_of(mine, Best{a.peaks.sig[p0 + i], a.peaks.id[p0 + i], i}, pos);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  warp_best(mine, pos);
  if (lane == 0) K.w[w] = mine;
  __syncthreads();
  if (w == 0) {
    Best b = lane < (int)(blockDim.x >> 5) ? K.w[lane] : Best{0, 0, -1};
    warp_best(b, pos);
    if (lane == 0) K.all = b;
  }
  __syncthreads();
  return K.all.i;
}

// steps 1 and 3 for member j at squared distance d < R2: tentative membership
// or reassignment (Eq. 3)
__device__ __forceinline__ void assign_member(const LevelArgs& a, unsigned base, int* eslot, long long* edold, int j,
                                              long long d, long long R2, int nn) {
  const int s = eslot[j];
  bool take = s < 0;
  if (!take) {
    const long long R2old = __ldcg(&a.nuc_R2[base + s]);
    take = (__int128)R2 * edold[j] * a.roche_den >= (__int128)a.roche_num * R2old * d;
  }
  if (take) {
    eslot[j] = nn;
    edold[j] = d;
  }
}

__device__ __forceinline__ Tiles group_tiles(const LevelArgs& a, int seg, unsigned base, int n, int rank, int cs) {
  // tiles of different groups never share a slot: a group of n members takes
  // at most n / TILE + 1 of them
  const size_t at = base / TILE + (size_t)seg;
  return Tiles{(n + TILE - 1) / TILE, rank, cs, a.tlo + at, a.thi + at, make_int4(0, 0, 0, 0), nullptr, -1};
}

// the runs' boxes from the tiles' (complete and visible to the block)
__device__ void super_boxes(const Tiles& T, SuperBoxes& B) {
  const int per = 32 * ((T.nt + 32 * SUPERS - 1) / (32 * SUPERS));
  const int ns = T.nt <= 2 * (int)blockDim.x ? 0 : (T.nt + per - 1) / per;
  if (threadIdx.x == 0) {
    B.n = ns;
    B.per = per;
  }
  const int lane = threadIdx.x & 31;
  for (int s = threadIdx.x >> 5; s < ns; s += blockDim.x >> 5) {
    int a[3] = {INT_MAX, INT_MAX, INT_MAX}, b[3] = {INT_MIN, INT_MIN, INT_MIN};
    for (int t = s * per + lane; t < min((s + 1) * per, T.nt); t += 32) {
      const int4 l = T.lo[t], h = T.hi[t];
      a[0] = min(a[0], l.x), a[1] = min(a[1], l.y), a[2] = min(a[2], l.z);
      b[0] = max(b[0], h.x), b[1] = max(b[1], h.y), b[2] = max(b[2], h.z);
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      a[x] = __reduce_min_sync(0xffffffffu, a[x]);
      b[x] = __reduce_max_sync(0xffffffffu, b[x]);
    }
    if (lane == 0)
      for (int x = 0; x < 3; ++x) B.lo[x][s] = a[x], B.hi[x][s] = b[x];
  }
  __syncthreads();
}

__device__ __forceinline__ int4 tile_origin(const int4* epos, int4 pc) {
  const int4 ref = epos[0];
  return make_int4(fold21(pc.x - ref.x), fold21(pc.y - ref.y), fold21(pc.z - ref.z), 0);
}

struct BlockShared {
  SelShared S;
  PickShared K;
  uint32_t tiles[TILE_LIST];
  int ntiles;
  unsigned h[LEVELS];
  int hbest;
};

template <int NT>
__device__ void level_block(const LevelArgs& a, const int seg, BlockShared& B) {
  const unsigned p0 = a.peaks.off[seg];
  const int m = (int)(a.peaks.off[seg + 1] - p0);
  const int tid = threadIdx.x;
  if (m == 0) {
    if (tid == 0) a.nnuc[seg] = 0;
    return;
  }
  const unsigned base = a.seg_off[seg];
  const int n = (int)(a.seg_off[seg + 1] - base);
  const int4* epos = a.epos + base;
  int* eslot = a.eslot + base;
  long long* edold = a.edold + base;
  long long* ed = a.ed + base;
  Tiles T = group_tiles(a, seg, base, n, 0, 1);
  const bool boxes = m > 1 && n > a.small_n;
  if (boxes) tile_boxes(T, epos, n, a.tlo + (T.lo - a.tlo), a.thi + (T.hi - a.thi));
  unsigned long long gone = 0;
  int cur = next_nucleus(a, p0, m, -1, make_int4(0, 0, 0, 0), 0, gone, B.K);
  int nn = 0;
  while (cur >= 0) {
    const int4 pc = a.peaks.pos[p0 + cur];
    long long R2 = -1;
    if (boxes && nn > 0) {
      T.q = tile_origin(epos, pc);
      for (int k = 0; k <= TRIES && R2 < 0; ++k) {
        const unsigned long long lim = k < TRIES ? try_bound(k, a.pc) : search_bound(T, n, a.pc, B.h, &B.hbest);
        T.nlist = -1;
        if (lim) list_tiles(T, lim, B.tiles, &B.ntiles);
        R2 = r_search<NT>(epos, ed, n, pc, a.pc, B.S, a.small_n, a.cap, a.nb, T, lim, k == TRIES);
      }
    } else {
      R2 = r_search<NT>(epos, ed, n, pc, a.pc, B.S, a.small_n, a.cap, a.nb, T, 0, true);
    }
    if (n <= a.small_n) {
      for (int j = tid; j < n; j += NT)
        if (ed[j] < R2) assign_member(a, base, eslot, edold, j, ed[j], R2, nn);
    } else {
      for_members(T, n, boxes && nn > 0 ? (unsigned long long)R2 : 0, [&](int j) {
        const long long d = ed[j];
        if (d < R2) assign_member(a, base, eslot, edold, j, d, R2, nn);
      });
    }
    if (tid == 0) {
      a.nuc_member[base + nn] = (uint32_t)pc.w;
      a.nuc_R2[base + nn] = R2;
    }
    ++nn;
    if (m == 1) break;
    __syncthreads();
    cur = next_nucleus(a, p0, m, cur, pc, R2, gone, B.K);
  }
  if (tid == 0) {
    a.nnuc[seg] = (uint32_t)nn;
    if (a.work) atomicAdd(a.work, (unsigned long long)nn * (unsigned long long)n);
  }
}

// The plain schedule: a block per group, of 1024 threads for groups above
// PLAIN_BIG members and of 256 for the rest (each launch skips the other's): the
// groups above small_n, whose members are walked in tiles.  The line is not sharp;
// both levels together with 512 / 1,024 / 2,048 / 4,096 / 8,192, ms: 262,144
// particles 0.51 / 0.54 / 0.57 / 0.58 / 0.58, 2.1M 1.90 / 1.94 / 2.03 / 2.04 / 2.06,
// 16.8M 4.43 / 4.41 / 4.45 / 4.45 / 4.43.
constexpr int PLAIN_BIG = 2048;

template <int NT>
__global__ void __launch_bounds__(NT) k_level(LevelArgs a) {
  __shared__ BlockShared B;
  const int seg = (int)blockIdx.x;
  if ((a.seg_off[seg + 1] - a.seg_off[seg] > PLAIN_BIG) == (NT == 1024)) level_block<NT>(a, seg, B);
}

// ---------------------------------------------------------------------------
// Groups of up to 512 members: 128 threads, members, distances and slots in
// registers (four per thread), every member's strictly enclosed count counted
// directly: n(<d_i) = #{j : d_j < d_i}, R^2 the smallest d_i whose count
// satisfies the predicate.  4 KB of shared memory instead of the histogram's
// 40, so sixteen such groups are in flight on an SM instead of four.
// ---------------------------------------------------------------------------
constexpr int SM_NT = 128;
constexpr int SM_PER = COUNT_N / SM_NT;

struct SmallShared {
  long long d[COUNT_N];
  PickShared K;
  unsigned long long r;     // smallest qualifying distance
  unsigned long long dmax;  // farthest member
};

__device__ void level_small(const LevelArgs& a, const int seg, SmallShared& B) {
  const int tid = threadIdx.x;
  const unsigned base = a.seg_off[seg];
  const int n = (int)(a.seg_off[seg + 1] - base);
  const unsigned p0 = a.peaks.off[seg];
  const int m = (int)(a.peaks.off[seg + 1] - p0);
  int4 p[SM_PER];
  long long d[SM_PER], dold[SM_PER];
  int slot[SM_PER];
#pragma unroll
  for (int k = 0; k < SM_PER; ++k) {
    const int j = tid + k * SM_NT;
    p[k] = j < n ? a.epos[base + j] : make_int4(0, 0, 0, 0);
    slot[k] = -1;
    dold[k] = 0;
  }
  unsigned long long gone = 0;
  int cur = next_nucleus(a, p0, m, -1, make_int4(0, 0, 0, 0), 0, gone, B.K);
  int nn = 0;
  while (cur >= 0) {
    const int4 pc = a.peaks.pos[p0 + cur];
    unsigned long long dmax = 0;
#pragma unroll
    for (int k = 0; k < SM_PER; ++k) {
      const int j = tid + k * SM_NT;
      d[k] = j < n ? dist2(pc, p[k]) : LLONG_MAX;
      if (j < n) {
        B.d[j] = d[k];
        dmax = max(dmax, (unsigned long long)d[k]);
      }
    }
    if (tid == 0) {
      B.r = ~0ull;
      B.dmax = 0;
    }
    __syncthreads();
    unsigned cnt[SM_PER] = {};
    for (int j = 0; j < n; ++j) {
      const long long v = B.d[j];
#pragma unroll
      for (int k = 0; k < SM_PER; ++k) cnt[k] += v < d[k];
    }
    unsigned long long best = ~0ull;
#pragma unroll
    for (int k = 0; k < SM_PER; ++k)
      if (tid + k * SM_NT < n && (unsigned long long)d[k] < best && pred(cnt[k], (unsigned long long)d[k], a.pc))
        best = (unsigned long long)d[k];
    if (best != ~0ull) atomicMin(&B.r, best);
    dmax = warp_max_u64(dmax);
    if ((tid & 31) == 0) atomicMax(&B.dmax, dmax);
    __syncthreads();
    if (B.r == ~0ull) {
      __syncthreads();
      if (tid == 0) B.r = (unsigned long long)exhaust_radius((unsigned long long)n, (long long)B.dmax, a.pc);
      __syncthreads();
    }
    const long long R2 = (long long)B.r;
#pragma unroll
    for (int k = 0; k < SM_PER; ++k) {
      if (d[k] >= R2) continue;  // past the end: LLONG_MAX
      bool take = slot[k] < 0;
      if (!take) {
        const long long R2old = __ldcg(&a.nuc_R2[base + slot[k]]);
        take = (__int128)R2 * dold[k] * a.roche_den >= (__int128)a.roche_num * R2old * d[k];
      }
      if (take) {
        slot[k] = nn;
        dold[k] = d[k];
      }
    }
    if (tid == 0) {
      a.nuc_member[base + nn] = (uint32_t)pc.w;
      a.nuc_R2[base + nn] = R2;
    }
    ++nn;
    if (m == 1) break;
    __syncthreads();
    cur = next_nucleus(a, p0, m, cur, pc, R2, gone, B.K);
  }
#pragma unroll
  for (int k = 0; k < SM_PER; ++k)
    if (tid + k * SM_NT < n) a.eslot[base + tid + k * SM_NT] = slot[k];
  if (tid == 0) {
    a.nnuc[seg] = (uint32_t)nn;
    if (a.work) atomicAdd(a.work, (unsigned long long)nn * (unsigned long long)n);
  }
}

// ---------------------------------------------------------------------------
// Giant groups: one thread-block cluster of CS CTAs per group.  CTA r owns
// the tiles r, r + CS, ... for the distance, histogram, gather and assignment
// passes (interleaved, so that the tiles in reach of a nucleus spread over the
// CTAs); CTA 0 (the leader) takes the select's decisions and broadcasts them
// through its shared memory, which the other CTAs read over DSMEM.  A phase
// of the select is: own work, barrier, the leader's decision from everyone's
// shares, barrier.  Every CTA passes every cluster barrier, in the same order:
// all control decisions are read from the leader after a barrier, or computed
// by every CTA from the same data.
// ---------------------------------------------------------------------------
namespace cg = cooperative_groups;

constexpr int CL_CS = 8;      // CTAs per cluster (giant groups)
constexpr int CL_HUGE_CS = 16;  // CTAs per cluster for huge groups (non-portable size, where it fits)
constexpr int CL_NT = 1024;   // threads per CTA

enum : int { OP_DONE = 0, OP_HIST = 1, OP_GATHER = 2, OP_RESTART = 3 };

struct ClusterCtl {
  int op;
  Window W;
  long long R2;
  unsigned long long cb;    // enclosed count of the bin to gather
  int bin, last;            // bins to gather, or the one to find the extent of
  int listed;               // its members are listed (they fit)
  unsigned in_window;
};

// leader only: decide the next step of the select from bin `from` of the
// merged histogram (S.cnt / S.clo, window in Ctl)
__device__ void leader_decide(ClusterCtl& C, SelShared& S, int from, int nb, int cap, int n, const PredConst& c,
                              float scale0, unsigned long long lim) {
  const int tid = threadIdx.x;
  if (tid == 0) S.best = NB;
  __syncthreads();
  const unsigned long long dtop = S.dmax_all < C.W.whi ? S.dmax_all : C.W.whi;
  for (int b = from + tid; b < NB; b += blockDim.x)
    if (S.cnt[b] && pred(C.W.base + S.clo[b], bin_top(C.W, b, c, scale0, nb, dtop), c)) atomicMin(&S.best, b);
  __syncthreads();
  if (tid == 0) {
    const int b = S.best;
    if (b < NB) {
      C.op = OP_GATHER;
      C.cb = C.W.base + S.clo[b];
      C.bin = b;
      C.last = S.cnt[b] <= (unsigned)min(cap, RANGE) ? range_end(S, b) : b;
      C.listed = S.cnt[b] <= (unsigned)cap;
    } else {  // nothing in the window: move past it
      const unsigned long long top = lim ? lim - 1 : S.dmax_all;
      if (C.W.whi < top) {
        C.op = OP_HIST;
        C.W = Window{C.W.whi + 1, top, C.W.base + C.in_window, 1};
      } else if (lim) {  // nothing below the bound: all members, from the start
        C.op = OP_RESTART;
        C.W = Window{0, ~0ull, 0, 0};
      } else {
        C.op = OP_DONE;
        C.R2 = exhaust_radius((unsigned long long)n, (long long)S.dmax_all, c);
      }
    }
  }
  __syncthreads();
}

// R^2 of nucleus pc over the group, computed by the whole cluster.  Every CTA
// builds its histogram (and, for a gather, its list) in its own shared
// memory; after the barrier the leader reads the others' with plain DSMEM
// loads and combines them.
__device__ long long cluster_r_search(cg::cluster_group& cluster, const int4* __restrict__ epos,
                                      long long* __restrict__ ed, int n, Tiles& T, int4 pc, const PredConst& c,
                                      SelShared& S, ClusterCtl& C, int cap, int nb, unsigned long long lim) {
  const int tid = threadIdx.x;
  const bool leader = cluster.block_rank() == 0;
  const int cs = (int)cluster.num_blocks();
  ClusterCtl* LC = cluster.map_shared_rank(&C, 0);
  float scale0 = bin_scale(n, lim, c, nb);
  // the first pass: threshold-count bins over every distance below the bound
  Window W{0, lim ? lim - 1 : ~0ull, 0, 0};
  bool first = true;
  int op = OP_HIST;
  while (true) {
    if (op != OP_GATHER) {
      if (op == OP_RESTART) {
        first = true;
        lim = 0;
        T.nlist = -1;
        scale0 = bin_scale(n, 0, c, nb);
      }
      for (int b = tid; b < NB; b += blockDim.x) S.cnt[b] = 0;
      if (tid == 0 && first) S.dmax_all = 0;
      __syncthreads();
      unsigned long long dmax = 0;  // this thread's farthest member (first pass)
      for_members(T, n, lim, [&](int j) {
        unsigned long long d;
        if (first) {
          d = (unsigned long long)dist2(pc, epos[j]);
          ed[j] = (long long)d;
          dmax = d > dmax ? d : dmax;
        } else {
          d = (unsigned long long)ed[j];
        }
        if (d >= W.wlo && d <= W.whi) atomicAdd(&S.cnt[window_bin(W, d, c, scale0, nb)], 1u);
      });
      if (first) {
        const unsigned long long m = warp_max_u64(dmax);
        if ((tid & 31) == 0) atomicMax(&S.dmax_all, m);
      }
      cluster.sync();  // every CTA's histogram of its members is complete
      if (leader) {
        if (tid == 0) C.W = W;
        // combine the CTAs' histograms (the leader's own is the first share)
        static_assert(NB == CL_NT, "one bin per thread");
        unsigned cn = S.cnt[tid];
        for (int r = 1; r < cs; ++r) cn += cluster.map_shared_rank(&S, r)->cnt[tid];
        S.cnt[tid] = cn;
        if (first && tid < 32) {
          unsigned long long m = tid < cs ? cluster.map_shared_rank(&S, tid)->dmax_all : 0;
          m = warp_max_u64(m);
          if (tid == 0) S.dmax_all = m;
        }
        __syncthreads();
        unsigned excl;
        const unsigned tot = block_scan<CL_NT>(cn, excl, S.sw);
        S.clo[tid] = excl;
        if (tid == 0) C.in_window = tot;
        __syncthreads();
        leader_decide(C, S, 0, nb, cap, n, c, scale0, lim);
      }
      first = false;
    } else {  // OP_GATHER: every CTA lists its members of the bin (or finds their extent), the leader collects them
      const int bin = LC->bin, last = LC->last;
      const bool listed = LC->listed;
      if (tid == 0) {
        S.nlist = 0;
        S.pick = ~0ull;
        S.lo = ~0ull;
        S.hi = 0;
      }
      __syncthreads();
      unsigned long long lo = ~0ull, hi = 0;
      for_members(T, n, lim, [&](int j) {
        const unsigned long long d = (unsigned long long)ed[j];
        if (d < W.wlo || d > W.whi) return;
        const int x = window_bin(W, d, c, scale0, nb);
        if (x < bin || x > last) return;
        if (listed) {
          S.list[atomicAdd(&S.nlist, 1)] = (long long)d;
        } else {
          lo = d < lo ? d : lo;
          hi = d > hi ? d : hi;
        }
      });
      if (!listed) {
        hi = warp_max_u64(hi);
        lo = ~warp_max_u64(~lo);
        if ((tid & 31) == 0) {
          atomicMin(&S.lo, lo);
          atomicMax(&S.hi, hi);
        }
      }
      cluster.sync();  // every CTA's list is complete
      if (leader && listed) {
        int off = S.nlist;
        for (int r = 1; r < cs; ++r) {
          const SelShared* R = cluster.map_shared_rank(&S, r);
          const int mr = R->nlist;
          for (int j = tid; j < mr; j += blockDim.x) S.list[off + j] = R->list[j];
          off += mr;
        }
        __syncthreads();
        const int m = off;
        long long r = -1;
        if (m <= RANGE) {
          r = (long long)pick_listed(S.list, m, C.cb, c, S);
        } else {
          const int p2 = pow2_at_least(m);
          for (int j = m + tid; j < p2; j += blockDim.x) S.list[j] = LLONG_MAX;
          __syncthreads();
          bitonic_sort(S.list, p2);
          const int k = scan_sorted(S.list, m, C.cb, c, &S.best);
          if (k < m) r = S.list[k];
        }
        if (r >= 0) {
          if (tid == 0) {
            C.op = OP_DONE;
            C.R2 = r;
          }
          __syncthreads();
        } else {
          leader_decide(C, S, C.last + 1, nb, cap, n, c, scale0, lim);
        }
      } else if (leader) {
        lo = ~0ull;
        hi = 0;
        if (tid < cs) {
          const SelShared* R = cluster.map_shared_rank(&S, tid);
          lo = R->lo;
          hi = R->hi;
        }
        if (tid < 32) {
          hi = warp_max_u64(hi);
          lo = ~warp_max_u64(~lo);
        }
        if (tid == 0) {
          S.best = 0;
          if (lo == hi) {  // one distinct value: its enclosed count is cb
            if (pred(C.cb, lo, c)) {
              C.op = OP_DONE;
              C.R2 = (long long)lo;
            } else {
              S.best = 1;
            }
          } else {  // narrow the window to the bin
            C.op = OP_HIST;
            C.W = Window{lo, hi, C.cb, 1};
          }
        }
        __syncthreads();
        const bool next_bin = S.best == 1;
        __syncthreads();
        if (next_bin) leader_decide(C, S, C.bin + 1, nb, cap, n, c, scale0, lim);
      }
    }
    // the leader's decision is published, and it has read everyone's shares;
    // it writes the next one only after the next phase's first barrier, which
    // no CTA reaches before it has read this one
    cluster.sync();
    op = LC->op;
    if (op == OP_DONE) break;
    W = LC->W;
  }
  return LC->R2;
}

struct ClusterShared {
  SelShared S;
  ClusterCtl C;
  PickShared K;
  uint32_t tiles[TILE_LIST];
  int ntiles;
  SuperBoxes sup;
  unsigned h[LEVELS];
  int hbest;
};

template <int CS>
__device__ void cluster_level(const LevelArgs& a, const int seg, ClusterShared& B) {
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const bool leader = rank == 0;
  const unsigned base = a.seg_off[seg];
  const int n = (int)(a.seg_off[seg + 1] - base);
  const unsigned p0 = a.peaks.off[seg];
  const int m = (int)(a.peaks.off[seg + 1] - p0);
  const int tid = threadIdx.x;
  const int cs = (int)cluster.num_blocks();
  const int4* epos = a.epos + base;
  int* eslot = a.eslot + base;
  long long* edold = a.edold + base;
  long long* ed = a.ed + base;
  Tiles T = group_tiles(a, seg, base, n, rank, cs);
  const bool boxes = m > 1;
  if (boxes) {
    tile_boxes(T, epos, n, a.tlo + (T.lo - a.tlo), a.thi + (T.hi - a.thi));
    cluster.sync();  // every CTA reads all boxes
    if (CS == CL_HUGE_CS) super_boxes(T, B.sup);
  }
  unsigned long long gone = 0;
  int cur = next_nucleus(a, p0, m, -1, make_int4(0, 0, 0, 0), 0, gone, B.K);
  int nn = 0;
  while (cur >= 0) {
    const int4 pc = a.peaks.pos[p0 + cur];
    long long R2 = -1;
    unsigned long long lim = 0;
    bool tried = false, held = false;
    if (boxes && nn > 0) {
      T.q = tile_origin(epos, pc);
      if (private_flags(m)) {
        // the tries are small: every CTA makes them over all tiles by itself,
        // which needs no barrier of the cluster.  The CTAs may then be
        // nuclei apart until the next search of the whole cluster, so a CTA
        // reads nothing here that another one writes on the way (distances,
        // flags and earlier radii are its own).
        T.rank = 0;
        T.cs = 1;
        for (int k = 0; k < TRIES && R2 < 0; ++k) {
          const unsigned long long tl = try_bound(k, a.pc);
          list_tiles(T, tl, B.tiles, &B.ntiles, CS == CL_HUGE_CS ? &B.sup : nullptr);
          if (CS == CL_HUGE_CS && tl && held_fits<CL_NT>(T)) {
            R2 = held_search<CL_NT>(epos, n, pc, a.pc, B.S, a.nb, T, tl);
            held = R2 >= 0;
            if (R2 != -2) continue;
          }
          R2 = r_search<CL_NT>(epos, nullptr, n, pc, a.pc, B.S, 0, a.cap, a.nb, T, tl, false);
        }
        tried = R2 >= 0;
        T.rank = rank;
        T.cs = cs;
      }
      if (!held) T.nlist = -1;
      if (R2 < 0) lim = search_bound(T, n, a.pc, B.h, &B.hbest);
      if (tried && !held) list_tiles(T, (unsigned long long)R2, B.tiles, &B.ntiles);
      else if (lim) list_tiles(T, lim, B.tiles, &B.ntiles);
    }
    if (R2 < 0) R2 = cluster_r_search(cluster, epos, ed, n, T, pc, a.pc, B.S, B.C, a.cap, a.nb, lim);
    // steps 1 and 3 on this CTA's share of the members
    if (held) {
      // this CTA's among the tiles that all of them listed
      for (int i = tid >> 5; i < T.nlist; i += CL_NT / 32) {
        const int t = (int)T.list[i];
        if (t % cs == rank)
          tile_members(t, n, [&](int j) {
            const long long d = dist2(pc, epos[j]);
            if (d < R2) assign_member(a, base, eslot, edold, j, d, R2, nn);
          });
      }
    } else {
      for_members(T, n, boxes && nn > 0 ? (unsigned long long)R2 : 0, [&](int j) {
        const long long d = tried ? dist2(pc, epos[j]) : ed[j];
        if (d < R2) assign_member(a, base, eslot, edold, j, d, R2, nn);
      });
    }
    if (tid == 0) {  // every CTA: it reads the radii back in later assignments
      a.nuc_member[base + nn] = (uint32_t)pc.w;
      a.nuc_R2[base + nn] = R2;
    }
    ++nn;
    if (m == 1) break;
    __syncthreads();
    cur = next_nucleus(a, p0, m, cur, pc, R2, gone, B.K);
  }
  if (leader && tid == 0) {
    a.nnuc[seg] = (uint32_t)nn;
    if (a.work) atomicAdd(a.work, (unsigned long long)nn * (unsigned long long)n);
  }
}

// ---------------------------------------------------------------------------
// The batched schedule's work queue: the groups that have peaks, filed by
// tier and size (four bins an octave) on the device, largest first, with one
// fetch counter per tier.  Six persistent kernels pull from it concurrently:
// 16-CTA clusters take huge groups, 8-CTA clusters giants, 1024-thread blocks
// large groups, 256-thread blocks medium ones, 128-thread blocks those of up
// to 512 members and warps the smallest, each taking the next group of its
// tier when it finishes one, so no launch size depends on a count read back
// by the host.
// ---------------------------------------------------------------------------
enum : int { TIER_HUGE = 0, TIER_GIANT, TIER_LARGE, TIER_MEDIUM, TIER_SMALL, TIER_WARP, TIERS };
constexpr int SIZE_BINS = 128;
constexpr int QBINS = TIERS * SIZE_BINS;

struct TierQueue {
  unsigned count[QBINS];  // groups per bin
  unsigned next[TIERS];   // fetch counters
  unsigned first[TIERS], cnt[TIERS];
};

struct TierBounds {
  int huge, giant, large, medium, small;  // groups above `huge` members are TIER_HUGE, ...
};

// bin of every group with peaks and its rank there; groups without any have no nuclei
__global__ void __launch_bounds__(1024) k_seg_bins(const uint32_t* __restrict__ seg_off,
                                                   const uint32_t* __restrict__ peak_off, int nseg, TierBounds b,
                                                   int* __restrict__ bin, uint32_t* __restrict__ rank,
                                                   uint32_t* __restrict__ nnuc, TierQueue* q) {
  __shared__ unsigned sc[QBINS];
  for (int i = threadIdx.x; i < QBINS; i += blockDim.x) sc[i] = 0;
  __syncthreads();
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  int k = -1;
  unsigned local = 0;
  if (g < nseg) {
    if (peak_off[g + 1] == peak_off[g]) {
      nnuc[g] = 0;
    } else {
      const int n = (int)(seg_off[g + 1] - seg_off[g]);
      const int tier = n > b.huge ? TIER_HUGE : n > b.giant ? TIER_GIANT : n > b.large ? TIER_LARGE
                       : n > b.medium ? TIER_MEDIUM : n > b.small ? TIER_SMALL : TIER_WARP;
      const int msb = 31 - __clz(n);
      const int size = 4 * msb + (int)(((unsigned)n << (31 - msb)) >> 29 & 3u);
      k = tier * SIZE_BINS + SIZE_BINS - 1 - size;
      local = atomicAdd(&sc[k], 1u);
    }
    bin[g] = k;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < QBINS; i += blockDim.x)
    if (sc[i]) sc[i] = atomicAdd(&q->count[i], sc[i]);
  __syncthreads();
  if (k >= 0) rank[g] = sc[k] + local;
}

// order[position] = group, bins in order; the tiers' ranges.  With the
// default schedule only as many giants go to clusters as clusters run at a
// time, and those of 2^GIANT_ALWAYS members or more; the others follow as the
// first large groups: a 1024-thread block is slower for one such group, but
// 152 of them finish seventy sooner than 19 clusters do (side-256 box, 74
// groups above 16,384: level 1 2.05 -> 1.78 ms, level 2 1.05 -> 0.80; the
// side-128 box has ten and keeps them all on clusters, 0.39 against 0.43 ms).
// Levels 1 and 2 of the side-400 box (64M particles) with GIANT_ALWAYS of 15, 16,
// 17, 18 and 30: 8.66, 8.03, 7.68, 7.68 and 7.68 ms, of the side-256 box 2.47, 2.32,
// 2.32, 2.32, 2.32: a group has to be several times the bound before a cluster's
// eight SMs are worth its wait, and these boxes have no more groups of 2^17 than
// clusters run at once.
constexpr int GIANT_ALWAYS = 17;
__global__ void __launch_bounds__(1024) k_seg_order(const int* __restrict__ bin, const uint32_t* __restrict__ rank,
                                                    int nseg, unsigned max_giants, uint32_t* __restrict__ order,
                                                    TierQueue* q) {
  __shared__ unsigned first[QBINS + 1];
  __shared__ unsigned sw[33];
  static_assert(QBINS < 1024, "one thread per bin");
  const unsigned v = threadIdx.x < QBINS ? q->count[threadIdx.x] : 0u;
  unsigned excl;
  block_scan<1024>(v, excl, sw);
  if (threadIdx.x <= QBINS) first[threadIdx.x] = excl;
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x < TIERS) {
    unsigned f = first[threadIdx.x * SIZE_BINS], e = first[(threadIdx.x + 1) * SIZE_BINS];
    if (max_giants != UINT_MAX && (threadIdx.x == TIER_GIANT || threadIdx.x == TIER_LARGE)) {
      // the boundary between giants and large groups in the size order
      const unsigned g0 = first[TIER_GIANT * SIZE_BINS], g1 = first[(TIER_GIANT + 1) * SIZE_BINS];
      const unsigned big = first[TIER_GIANT * SIZE_BINS + SIZE_BINS - 4 * GIANT_ALWAYS] - g0;
      const unsigned cut = min(g1, g0 + max(max_giants, big));
      if (threadIdx.x == TIER_GIANT) e = cut;
      else f = cut;
    }
    q->first[threadIdx.x] = f;
    q->cnt[threadIdx.x] = e - f;
  }
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < nseg && bin[g] >= 0) order[first[bin[g]] + rank[g]] = (uint32_t)g;
}

// giants on 8-CTA clusters, huge groups on 16-CTA clusters
template <int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(CL_NT)
    k_level_cluster_q(LevelArgs a, const uint32_t* __restrict__ order, TierQueue* q, int tier) {
  __shared__ ClusterShared B;
  __shared__ unsigned item;
  cg::cluster_group cluster = cg::this_cluster();
  const bool leader = cluster.block_rank() == 0;
  const unsigned first = q->first[tier], cnt = q->cnt[tier];
  for (;;) {
    // (the first barrier also ends the previous group: its last reads of the
    // leader's shared memory are done)
    if (leader && threadIdx.x == 0) item = atomicAdd(&q->next[tier], 1u);
    cluster.sync();
    const unsigned it = *cluster.map_shared_rank(&item, 0);
    cluster.sync();  // every CTA has read the leader's item before it changes
    if (it >= cnt) return;
    cluster_level<CS>(a, (int)order[first + it], B);
  }
}

template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_level_q(LevelArgs a, const uint32_t* __restrict__ order, TierQueue* q,
                                                int tier) {
  __shared__ BlockShared B;
  __shared__ unsigned item;
  const unsigned first = q->first[tier], cnt = q->cnt[tier];
  for (;;) {
    if (threadIdx.x == 0) item = atomicAdd(&q->next[tier], 1u);
    __syncthreads();
    const unsigned it = item;
    __syncthreads();
    if (it >= cnt) return;
    level_block<NT>(a, (int)order[first + it], B);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(SM_NT, 8) k_level_small_q(LevelArgs a, const uint32_t* __restrict__ order,
                                                          TierQueue* q) {
  __shared__ SmallShared B;
  __shared__ unsigned item;
  const unsigned first = q->first[TIER_SMALL], cnt = q->cnt[TIER_SMALL];
  for (;;) {
    if (threadIdx.x == 0) item = atomicAdd(&q->next[TIER_SMALL], 1u);
    __syncthreads();
    const unsigned it = item;
    __syncthreads();
    if (it >= cnt) return;
    level_small(a, (int)order[first + it], B);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// One small group (n <= 64 members) per warp.  Members live in registers
// (lane l holds members l and l + 32).  The enclosed count n(<d_i) of every
// member is counted directly over all members (n^2 compares), so R^2 =
// min{d_i : pred(n(<d_i), d_i)} needs no sort.
// ---------------------------------------------------------------------------
constexpr long long D_INF = LLONG_MAX;

__device__ __forceinline__ long long warp_min_ll(long long v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    long long t = __shfl_xor_sync(0xffffffffu, v, o);
    v = t < v ? t : v;
  }
  return v;
}

__device__ __forceinline__ long long warp_max_ll(long long v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    long long t = __shfl_xor_sync(0xffffffffu, v, o);
    v = t > v ? t : v;
  }
  return v;
}

__device__ void level_warp(const LevelArgs& a, const int seg) {
  const int lane = threadIdx.x & 31;
  const unsigned base = a.seg_off[seg];
  const int n = (int)(a.seg_off[seg + 1] - base);
  const unsigned p0 = a.peaks.off[seg];
  const int m = (int)(a.peaks.off[seg + 1] - p0);  // at most n <= 64
  const bool v0 = lane < n, v1 = lane + 32 < n;
  const int4 p0v = v0 ? a.epos[base + lane] : make_int4(0, 0, 0, 0);
  const int4 p1v = v1 ? a.epos[base + lane + 32] : make_int4(0, 0, 0, 0);
  int slot0 = -1, slot1 = -1;
  long long do0 = 0, do1 = 0;
  const long long anum2 = (long long)a.alpha_num * a.alpha_num, aden2 = (long long)a.alpha_den * a.alpha_den;
  // the group's peaks, two per lane, and whether each may still become a nucleus
  Best k0{0, 0, -1}, k1{0, 0, -1};
  int4 c0 = make_int4(0, 0, 0, 0), c1 = make_int4(0, 0, 0, 0);
  if (lane < m) {
    k0 = Best{a.peaks.sig[p0 + lane], a.peaks.id[p0 + lane], lane};
    c0 = a.peaks.pos[p0 + lane];
  }
  if (lane + 32 < m) {
    k1 = Best{a.peaks.sig[p0 + lane + 32], a.peaks.id[p0 + lane + 32], lane + 32};
    c1 = a.peaks.pos[p0 + lane + 32];
  }
  int nn = 0;
  while (true) {
    Best b = k0;
    best_of(b, k1, a.peaks.pos + p0);
    warp_best(b, a.peaks.pos + p0);
    if (b.i < 0) break;
    const int src = b.i & 31;
    const bool hi = b.i >= 32;
    int4 pc;
    pc.x = __shfl_sync(0xffffffffu, hi ? c1.x : c0.x, src);
    pc.y = __shfl_sync(0xffffffffu, hi ? c1.y : c0.y, src);
    pc.z = __shfl_sync(0xffffffffu, hi ? c1.z : c0.z, src);
    pc.w = __shfl_sync(0xffffffffu, hi ? c1.w : c0.w, src);
    const long long d0 = v0 ? dist2(pc, p0v) : D_INF, d1 = v1 ? dist2(pc, p1v) : D_INF;
    // strictly enclosed counts
    unsigned n0 = 0, n1 = 0;
    for (int j = 0; j < n; ++j) {
      const long long dj = __shfl_sync(0xffffffffu, j >= 32 ? d1 : d0, j & 31);
      n0 += dj < d0;
      n1 += dj < d1;
    }
    const bool ok0 = v0 && pred(n0, (unsigned long long)d0, a.pc);
    const bool ok1 = v1 && pred(n1, (unsigned long long)d1, a.pc);
    long long R2 = warp_min_ll(min(ok0 ? d0 : D_INF, ok1 ? d1 : D_INF));
    if (R2 == D_INF) {
      const long long dmax = warp_max_ll(max(v0 ? d0 : 0ll, v1 ? d1 : 0ll));
      long long r = 0;
      if (lane == 0) r = exhaust_radius((unsigned long long)n, dmax, a.pc);
      R2 = __shfl_sync(0xffffffffu, r, 0);
    }
    // step 3 on the two members of this lane
    if (v0 && d0 < R2) {
      bool take = slot0 < 0;
      if (!take) {
        const long long R2old = a.nuc_R2[base + slot0];
        take = (__int128)R2 * do0 * a.roche_den >= (__int128)a.roche_num * R2old * d0;
      }
      if (take) {
        slot0 = nn;
        do0 = d0;
      }
    }
    if (v1 && d1 < R2) {
      bool take = slot1 < 0;
      if (!take) {
        const long long R2old = a.nuc_R2[base + slot1];
        take = (__int128)R2 * do1 * a.roche_den >= (__int128)a.roche_num * R2old * d1;
      }
      if (take) {
        slot1 = nn;
        do1 = d1;
      }
    }
    // step 1: peaks nearer than alpha R (and the nucleus itself) are out
    if (k0.i >= 0 && (k0.i == b.i || (__int128)aden2 * dist2(pc, c0) < (__int128)anum2 * R2)) k0.i = -1;
    if (k1.i >= 0 && (k1.i == b.i || (__int128)aden2 * dist2(pc, c1) < (__int128)anum2 * R2)) k1.i = -1;
    if (lane == 0) {
      a.nuc_member[base + nn] = (uint32_t)pc.w;
      a.nuc_R2[base + nn] = R2;
    }
    __syncwarp();
    ++nn;
    if (m == 1) break;
  }
  if (v0) a.eslot[base + lane] = slot0;
  if (v1) a.eslot[base + lane + 32] = slot1;
  if (lane == 0) {
    a.nnuc[seg] = (uint32_t)nn;
    if (a.work && nn) atomicAdd(a.work, (unsigned long long)nn * (unsigned long long)n);
  }
}

__global__ void __launch_bounds__(256) k_level_warp_q(LevelArgs a, const uint32_t* __restrict__ order, TierQueue* q) {
  const unsigned first = q->first[TIER_WARP], cnt = q->cnt[TIER_WARP];
  const int lane = threadIdx.x & 31;
  for (;;) {
    unsigned it = 0;
    if (lane == 0) it = atomicAdd(&q->next[TIER_WARP], 1u);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= cnt) return;  // whole warps leave together
    level_warp(a, (int)order[first + it]);
  }
}

// largest g with off[g] <= k (off ascending, off[0] = 0)
__device__ __forceinline__ int seg_of(const uint32_t* __restrict__ off, int nseg, unsigned k) {
  int lo = 0, hi = nseg - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= k) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// per-halo nucleus records: one thread per halo (halos of segment g start at
// hbase[g])
__global__ void k_level_halo_nuclei(const uint32_t* __restrict__ seg_off, int nseg, const uint32_t* __restrict__ hbase,
                                    const uint32_t* __restrict__ nuc_member, const long long* __restrict__ nuc_R2,
                                    uint32_t* __restrict__ hnuc, long long* __restrict__ hR2) {
  const unsigned h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h >= hbase[nseg]) return;
  const int g = seg_of(hbase, nseg, h);  // hbase ascending; segments without nuclei repeat a value
  const unsigned base = seg_off[g], q = h - hbase[g];
  hnuc[h] = nuc_member[base + q];
  hR2[h] = nuc_R2[base + q];
}

}  // namespace

// resident blocks per SM of the persistent level kernels (same for every
// device of one build; queried once)
static std::atomic<int> g_occ_l{0}, g_occ_m{0}, g_occ_s{0}, g_occ_w{0};
// 16-CTA clusters that can be resident at once (0: that size does not fit
// this device, and huge groups stay on 8-CTA clusters)
static std::atomic<int> g_cl16{0};

void level_prepare() {
  if (g_occ_l.load()) return;
  int l = 0, m = 0, s = 0, w = 0;
  int c16 = 0;
  if (cudaFuncSetAttribute(k_level_cluster_q<CL_HUGE_CS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
      cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL_HUGE_CS, 1, 1);
    cfg.blockDim = dim3(CL_NT, 1, 1);
    if (cudaOccupancyMaxActiveClusters(&c16, k_level_cluster_q<CL_HUGE_CS>, &cfg) != cudaSuccess) c16 = 0;
  }
  cudaGetLastError();  // an unsupported size leaves only the answer 0
  g_cl16.store(c16 > 0 ? c16 : 0);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&l, k_level_q<1024>, 1024, 0) != cudaSuccess || l < 1) l = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, k_level_q<256>, 256, 0) != cudaSuccess || m < 1) m = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&s, k_level_small_q, SM_NT, 0) != cudaSuccess || s < 1) s = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&w, k_level_warp_q, 256, 0) != cudaSuccess || w < 1) w = 1;
  g_occ_m.store(m);
  g_occ_s.store(s);
  g_occ_w.store(w);
  g_occ_l.store(l);
  cso_sm_count();
}

int level_run(const LevelArgs& a, cudaStream_t st) {
  if (a.nseg <= 0) return CSO_OK;
  k_level<1024><<<CL(a.nseg), 1024, 0, st>>>(a);
  k_level<256><<<CL(a.nseg), 256, 0, st>>>(a);
  CSO_CUDA(cudaGetLastError());
  return CSO_OK;
}

size_t level_tiles(long long members, long long nseg) { return (size_t)(members / TILE + nseg + 2); }

int level_run_batched(const LevelArgs& a, const LevelSchedule& sc, Workspace& ws, cudaStream_t st,
                      cudaStream_t side, cudaStream_t side2, cudaStream_t side3, cudaEvent_t fork,
                      cudaEvent_t join, cudaEvent_t join2, cudaEvent_t join3) {
  if (a.nseg <= 0) return CSO_OK;
  size_t mark = ws.off;
  int* bin = ws.get<int>(a.nseg);
  uint32_t* rank = ws.get<uint32_t>(a.nseg);
  uint32_t* order = ws.get<uint32_t>(a.nseg);
  TierQueue* q = ws.get<TierQueue>(1);
  if (!bin || !rank || !order || !q) {
    cso_set_error("workspace exhausted in the batched schedule");
    return CSO_ERR_BUDGET;
  }
  CSO_CUDA(cudaMemsetAsync(q, 0, sizeof(TierQueue), st));
  level_prepare();
  const int c16 = g_cl16;
  // groups above the huge bound (and the giant bound) run on 16-CTA clusters
  // where the device holds them; the direct count of the small tier needs
  // groups that the select would count directly too
  TierBounds b;
  b.huge = c16 > 0 ? std::max(sc.giant, sc.huge) : INT_MAX;
  b.giant = sc.giant;
  b.large = sc.large();
  b.small = sc.small;
  b.medium = a.small_n >= COUNT_N ? std::max(b.small, COUNT_N) : b.small;
  k_seg_bins<<<CL(cdiv(a.nseg, 1024)), 1024, 0, st>>>(a.seg_off, a.peaks.off, a.nseg, b, bin, rank, a.nnuc, q);
  // persistent grids sized to the device; blocks of a tier leave when its
  // queue is empty
  const int occ_l = g_occ_l, occ_m = g_occ_m, occ_s = g_occ_s, occ_w = g_occ_w;
  const int sms = cso_sm_count();
  const int n_clusters = sms / CL_CS > 0 ? sms / CL_CS : 1;
  k_seg_order<<<CL(cdiv(a.nseg, 1024)), 1024, 0, st>>>(bin, rank, a.nseg, sc.max_giants(n_clusters), order, q);
  CSO_CUDA(cudaGetLastError());
  const int nseg = a.nseg;
  // no tier can hold more groups than there are: grids never exceed nseg
  auto cap = [nseg](long long g) { return (unsigned)(g < nseg ? g : nseg); };
  CSO_CUDA(cudaEventRecord(fork, st));
  CSO_CUDA(cudaStreamWaitEvent(side, fork, 0));
  k_level_cluster_q<CL_CS><<<CL(cap(n_clusters) * CL_CS), CL_NT, 0, side>>>(a, order, q, TIER_GIANT);
  CSO_CUDA(cudaGetLastError());
  if (c16 > 0) {
    // at most two: huge groups are few, and every 16-CTA cluster holds 16 SMs
    CSO_CUDA(cudaStreamWaitEvent(side3, fork, 0));
    k_level_cluster_q<CL_HUGE_CS><<<CL(cap(c16 < 2 ? c16 : 2) * CL_HUGE_CS), CL_NT, 0, side3>>>(a, order, q, TIER_HUGE);
    CSO_CUDA(cudaGetLastError());
  }
  CSO_CUDA(cudaStreamWaitEvent(side2, fork, 0));
  k_level_q<1024><<<CL(cap((long long)sms * occ_l)), 1024, 0, side2>>>(a, order, q, TIER_LARGE);
  k_level_q<256><<<CL(cap((long long)sms * occ_m)), 256, 0, st>>>(a, order, q, TIER_MEDIUM);
  if (b.medium > b.small)
    k_level_small_q<<<CL(cap((long long)sms * occ_s)), SM_NT, 0, st>>>(a, order, q);
  k_level_warp_q<<<CL(cdiv(cap((long long)sms * occ_w * 8), 8)), 256, 0, st>>>(a, order, q);
  CSO_CUDA(cudaGetLastError());
  CSO_CUDA(cudaEventRecord(join, side));
  CSO_CUDA(cudaStreamWaitEvent(st, join, 0));
  CSO_CUDA(cudaEventRecord(join2, side2));
  CSO_CUDA(cudaStreamWaitEvent(st, join2, 0));
  if (c16 > 0) {
    CSO_CUDA(cudaEventRecord(join3, side3));
    CSO_CUDA(cudaStreamWaitEvent(st, join3, 0));
  }
  ws.off = mark;
  return CSO_OK;
}

int level_halo(int nseg, const uint32_t* seg_off, const uint32_t* hbase, const uint32_t* nuc_member,
               const long long* nuc_R2, uint32_t* hnuc, long long* hR2, long long n_halos, cudaStream_t st) {
  if (nseg <= 0 || n_halos <= 0) return CSO_OK;
  k_level_halo_nuclei<<<CL(cdiv(n_halos, 256)), 256, 0, st>>>(seg_off, nseg, hbase, nuc_member, nuc_R2, hnuc, hR2);
  CSO_CUDA(cudaGetLastError());
  return CSO_OK;
}

PredConst make_pred_const(double K, long long u) {
  PredConst c{};  // zeroed padding: level stages are cached by their argument bytes
  c.K = K;
  int E;
  double f = frexp(K, &E);
  c.Km = (unsigned long long)ldexp(f, 53);
  c.Ke = E - 53;
  c.u = (unsigned long long)u;
  double ud = (double)u;
  c.u6 = ud * ud * ud * ud * ud * ud;
  // bin of the first window: threshold count sqrt(K) d^1.5 / u^3 (before /w)
  c.bin_scale0 = (float)(sqrt(K) / (ud * ud * ud));
  c.radial = 0;
  c.rbin_inv_w = 0.0f;
  return c;
}
