// Ranks of two sets of flagged elements in one pass over the array: the
// one-sweep sort of scan_sort.cu (decoupled look-back over tiles taken from
// an atomic counter) for flags known inside the caller's kernel, so that a
// list is written by the kernel that decides who is on it, with no flag
// array, scan and second pass in between.
#pragma once
#include "cso_internal.cuh"

constexpr int R2_THREADS = 256;
constexpr int R2_WARPS = R2_THREADS / 32;
// Elements per lane (a warp holds 32 ITEMS consecutive ones, 32 per item): 16,
// or 4 for arrays of up to R2_SMALL elements, where tiles of 4,096 would leave
// most SMs without one (131,000 dense particles: k_stragglers 52 -> 21 us).  FoF and
// gather together with 16 / 4, ms: 27,000 particles 0.159 / 0.139, 512,000 0.332 /
// 0.313, 1.3M 0.513 / 0.495, 2.0M 0.630 / 0.623, 4.1M 1.026 / 1.062, 8.0M 1.803 / 1.864.
constexpr int R2_BIG = 16, R2_FEW = 4;
constexpr long long R2_SMALL = 1ll << 21;

// A status word: state << 62 | first count << 31 | second count (counts below
// 2^31).  States: 0 not published, 1 the tile's own counts, 2 inclusive prefix.
struct Rank2Shared {
  uint32_t wa[R2_WARPS], wb[R2_WARPS];
  uint32_t a0, b0;
  long long tile;
};

static inline long long rank2_tiles(long long n) {
  return cdiv(n, R2_THREADS * (n > R2_SMALL ? R2_BIG : R2_FEW));
}
// status words needed for n elements or fewer (tiles, then the tile counter), zeroed by the caller
static inline long long rank2_words(long long n) {
  const long long few = n < R2_SMALL ? n : R2_SMALL, a = cdiv(few, R2_THREADS * R2_FEW), b = cdiv(n, R2_THREADS * R2_BIG);
  return (a > b ? a : b) + 1;
}

// launches KERNEL<ITEMS> over n elements; the variadic arguments end in ..., status, tiles, ...
#define RANK2_LAUNCH(KERNEL, n, st, ...)                                                             \
  do {                                                                                               \
    const unsigned tiles_ = (unsigned)rank2_tiles(n);                                                \
    if ((n) > R2_SMALL) KERNEL<R2_BIG><<<CL(tiles_), R2_THREADS, 0, st>>>(__VA_ARGS__);              \
    else KERNEL<R2_FEW><<<CL(tiles_), R2_THREADS, 0, st>>>(__VA_ARGS__);                             \
  } while (0)

__device__ __forceinline__ long long rank2_tile(Rank2Shared& S, unsigned long long* status, long long ntiles) {
  if (threadIdx.x == 0) S.tile = (long long)atomicAdd(&status[ntiles], 1ull);
  __syncthreads();
  return S.tile;
}

// Both counts of a whole tile from its elements, by the calling warp: flags(i) has
// bit 0 set if element i is in the first set, bit 1 if it is in the second.
template <int ITEMS, class F>
__device__ __forceinline__ uint2 rank2_count(long long tile, F flags) {
  const long long base = tile * (R2_THREADS * ITEMS) + (threadIdx.x & 31);
  uint2 c = make_uint2(0, 0);
#pragma unroll 1
  for (int q = 0; q < R2_THREADS * ITEMS; q += 32) {
    const unsigned f = flags(base + q);
    c.x += __popc(__ballot_sync(0xffffffffu, f & 1u));
    c.y += __popc(__ballot_sync(0xffffffffu, f & 2u));
  }
  return c;
}

// wa, wb: the calling warp's counts (the same on every lane).  On return they
// are the numbers of flagged elements before the warp's first one; ta, tb the
// inclusive totals up to the end of this tile.  recount(t), called by one warp,
// gives both counts of the whole tile t < tile (rank2_count).
template <class R>
__device__ __forceinline__ void rank2_prefix(Rank2Shared& S, unsigned long long* status, long long tile, uint32_t& wa,
                                             uint32_t& wb, uint32_t& ta, uint32_t& tb, long long patience, R recount) {
  constexpr unsigned long long M31 = (1ull << 31) - 1;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) {
    S.wa[w] = wa;
    S.wb[w] = wb;
  }
  __syncthreads();
  uint32_t suma = 0, sumb = 0, befa = 0, befb = 0;
#pragma unroll
  for (int k = 0; k < R2_WARPS; ++k) {
    if (k == w) {
      befa = suma;
      befb = sumb;
    }
    suma += S.wa[k];
    sumb += S.wb[k];
  }
  if (w == 0) {
    uint32_t pa = 0, pb = 0;
    if (tile > 0) {
      auto put = [&](unsigned long long state, uint32_t a, uint32_t b) {
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(status + tile),
                     "l"(state << 62 | (unsigned long long)a << 31 | b)
                     : "memory");
      };
      if (lane == 0) put(1, suma, sumb);
      long long top = tile - 1, spins = 0;
      for (;;) {
        const long long j = top - lane;
        unsigned long long v = 2ull << 62;  // before tile 0: prefix 0
        if (j >= 0) asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(status + j) : "memory");
        const unsigned pmask = __ballot_sync(0xffffffffu, v >> 62 == 2);
        const unsigned xmask = __ballot_sync(0xffffffffu, v >> 62 == 0);
        const int first = pmask ? __ffs(pmask) - 1 : 31;
        const unsigned need = first == 31 ? 0xffffffffu : (2u << first) - 1u;
        if (xmask & need) {  // a predecessor has not published yet
          if (spins++ < patience) continue;
          // count the nearest such tile here and go on behind it
          const int q = __ffs(xmask & need) - 1;
          const uint2 c = recount(top - q);
          pa += c.x + __reduce_add_sync(0xffffffffu, lane < q ? (uint32_t)(v >> 31 & M31) : 0u);
          pb += c.y + __reduce_add_sync(0xffffffffu, lane < q ? (uint32_t)(v & M31) : 0u);
          top -= q + 1;
          continue;
        }
        pa += __reduce_add_sync(0xffffffffu, lane <= first ? (uint32_t)(v >> 31 & M31) : 0u);
        pb += __reduce_add_sync(0xffffffffu, lane <= first ? (uint32_t)(v & M31) : 0u);
        if (pmask) break;
        top -= 32;
      }
      if (lane == 0) put(2, pa + suma, pb + sumb);
    } else if (lane == 0) {
      asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(status),
                   "l"(2ull << 62 | (unsigned long long)suma << 31 | sumb)
                   : "memory");
    }
    if (lane == 0) {
      S.a0 = pa;
      S.b0 = pb;
    }
  }
  __syncthreads();
  wa = S.a0 + befa;
  wb = S.b0 + befb;
  ta = S.a0 + suma;
  tb = S.b0 + sumb;
}
