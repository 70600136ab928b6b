// Device-wide exclusive scan and stable LSD radix sorts (8-bit digits).
//
// Both sorts rank elements inside a tile with warp-level matching
// (__match_any_sync): warp w owns a contiguous run of the tile and keeps a
// running per-digit counter in shared memory, so ranks are stable; per-warp
// counts are then prefixed across warps.  Keys of up to 64 bits go through
// the one-sweep sort (one kernel per digit, tile offsets by look-back); keys
// wider than 64 bits (two words) through a histogram / scan / scatter
// sequence per digit whose tile offsets come from the scanned [digit][tile]
// histogram.
#include <algorithm>

#include "cso_internal.cuh"

namespace {

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
  int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// block-wide exclusive scan of one value per thread; returns the block total
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* smem_warp, uint32_t& excl) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t inc = warp_incl_scan(v);
  if (lane == 31) smem_warp[w] = inc;
  __syncthreads();
  if (w == 0) {
    uint32_t s = lane < nw ? smem_warp[lane] : 0;
    uint32_t si = warp_incl_scan(s);
    if (lane < nw) smem_warp[lane] = si - s;
    if (lane == 31) smem_warp[32] = si;
  }
  __syncthreads();
  excl = inc - v + smem_warp[w];
  uint32_t total = smem_warp[32];
  __syncthreads();
  return total;
}

// Look-back status words of the one-sweep sort (the decoupled look-back of
// Merrill and Garland, "Single-pass Parallel Prefix Scan with Decoupled
// Look-back", 2016).
__device__ __forceinline__ unsigned long long sp_load(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void sp_store(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Exclusive scan of a large array in two passes over it: sums of every warp's
// run (k_scan_sums), the blocks' sums in one block (k_scan_small), then the runs
// again with their bases (k_scan_apply).  Bound by its bytes: the second read
// costs less than the waits of a single pass with look-back did, and no warp
// waits for another.  Of 262M values 0.52 -> 0.47 ms against tiles of 32,768 by
// look-back, of 2M to 4M 21-25 -> 15 us (with the clearing of its status words).
// A run is `rounds` times 128 values (a multiple of 4 rounds, so that four loads
// a lane are in flight, and eight of the 16-bit values' half as wide ones in the
// sums: binning with 262M cells 0.673 -> 0.656 ms); a block is 8 runs.
constexpr int SC_WARPS = 8;

struct ScanIn {
  const uint32_t* w;     // the values,
  const uint16_t* half;  // or (not null, and *over 0) the same in 16 bits
  const int* over;
  __device__ __forceinline__ bool narrow() const { return half && *over == 0; }
};

// values i .. i+3 (i a multiple of 4), zero past n
template <bool HALF>
__device__ __forceinline__ uint4 scan_load(const ScanIn& in, long long i, long long n) {
  if (i + 4 <= n) {
    if (HALF) {
      const uint2 v = *reinterpret_cast<const uint2*>(in.half + i);
      return make_uint4(v.x & 0xffffu, v.x >> 16, v.y & 0xffffu, v.y >> 16);
    }
    return *reinterpret_cast<const uint4*>(in.w + i);
  }
  uint32_t t[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) t[k] = i + k < n ? (HALF ? (uint32_t)in.half[i + k] : in.w[i + k]) : 0u;
  return make_uint4(t[0], t[1], t[2], t[3]);
}

template <bool HALF, int U>
__device__ __forceinline__ uint32_t scan_run_sum(const ScanIn& in, long long at, long long n, int rounds) {
  uint32_t sum = 0;
  for (int r = 0; r < rounds; r += U) {
    uint4 v[U];
#pragma unroll
    for (int k = 0; k < U; ++k) v[k] = scan_load<HALF>(in, at + (long long)(r + k) * 128, n);
#pragma unroll
    for (int k = 0; k < U; ++k) sum += v[k].x + v[k].y + v[k].z + v[k].w;
  }
  return __reduce_add_sync(0xffffffffu, sum);
}

// run_base[block * 8 + w]: the values of the block before warp w's run
__global__ void __launch_bounds__(SC_WARPS * 32)
    k_scan_sums(ScanIn in, long long n, int rounds, uint32_t* __restrict__ run_base, uint32_t* __restrict__ block_sum) {
  __shared__ uint32_t sw[SC_WARPS];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long run = (long long)blockIdx.x * SC_WARPS + w;
  const long long at = run * rounds * 128 + lane * 4;
  const uint32_t sum = in.narrow() ? (rounds % 8 ? scan_run_sum<true, 4>(in, at, n, rounds)
                                                 : scan_run_sum<true, 8>(in, at, n, rounds))
                                   : scan_run_sum<false, 4>(in, at, n, rounds);
  if (lane == 0) sw[w] = sum;
  __syncthreads();
  uint32_t before = 0;
  for (int k = 0; k < w; ++k) before += sw[k];
  if (lane == 0) run_base[run] = before;
  if (w == SC_WARPS - 1 && lane == 0) block_sum[blockIdx.x] = before + sum;
}

template <bool HALF>
__device__ __forceinline__ void scan_run(const ScanIn& in, uint32_t* d, long long at, long long n, int rounds,
                                         uint32_t carry) {
  for (int r = 0; r < rounds; r += 4) {
    uint4 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = scan_load<HALF>(in, at + (long long)(r + k) * 128, n);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long i = at + (long long)(r + k) * 128;
      const uint32_t sum = v[k].x + v[k].y + v[k].z + v[k].w;
      const uint32_t inc = warp_incl_scan(sum);
      const uint32_t b0 = carry + inc - sum, b1 = b0 + v[k].x, b2 = b1 + v[k].y, b3 = b2 + v[k].z;
      carry += __shfl_sync(0xffffffffu, inc, 31);
      if (i + 4 <= n) {
        *reinterpret_cast<uint4*>(d + i) = make_uint4(b0, b1, b2, b3);
      } else {
        if (i < n) d[i] = b0;
        if (i + 1 < n) d[i + 1] = b1;
        if (i + 2 < n) d[i + 2] = b2;
      }
    }
  }
}

// A lane reads its four values before it writes them and no other lane touches
// them, so d may be in.w.
__global__ void __launch_bounds__(SC_WARPS * 32)
    k_scan_apply(ScanIn in, uint32_t* d, long long n, int rounds, const uint32_t* __restrict__ run_base,
                 const uint32_t* __restrict__ block_base) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = blockIdx.x;
  const long long run = (long long)b * SC_WARPS + w;
  const long long at = run * rounds * 128 + lane * 4;
  const uint32_t base = block_base[b] + run_base[run];
  if (in.narrow())
    scan_run<true>(in, d, at, n, rounds, base);
  else
    scan_run<false>(in, d, at, n, rounds, base);
}

// --------------------------------------------------------------------------
// radix sort
// --------------------------------------------------------------------------
constexpr int RS_WARPS = 8;
constexpr int RS_THREADS = RS_WARPS * 32;
constexpr int RS_ITEMS = 8;                       // per lane
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;    // 2048
constexpr int RS_RADIX = 256;

struct Key128 {
  const uint64_t* hi;
  const uint64_t* lo;
  // shifts are multiples of 8, so a digit never straddles the two words
  __device__ __forceinline__ uint32_t digit(long long i, int shift) const {
    if (shift < 64) return (uint32_t)(lo[i] >> shift) & 0xffu;
    return (uint32_t)(hi[i] >> (shift - 64)) & 0xffu;
  }
};


template <class K>
__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(K key, long long n, int shift, uint32_t* __restrict__ hist,
                                                      int ntiles) {
  __shared__ uint32_t h[RS_RADIX];
  for (int t = threadIdx.x; t < RS_RADIX; t += RS_THREADS) h[t] = 0;
  __syncthreads();
  long long base = (long long)blockIdx.x * RS_TILE;
#pragma unroll
  for (int k = 0; k < RS_ITEMS; ++k) {
    long long i = base + (long long)k * RS_THREADS + threadIdx.x;
    if (i < n) atomicAdd(&h[key.digit(i, shift)], 1u);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < RS_RADIX; t += RS_THREADS) hist[(long long)t * ntiles + blockIdx.x] = h[t];
}

template <class K, class MoveFn>
__device__ __forceinline__ void rs_scatter_body(K key, long long n, int shift, const uint32_t* __restrict__ hist,
                                                int ntiles, MoveFn move) {
  __shared__ uint32_t wh[RS_WARPS][RS_RADIX];
  __shared__ uint32_t gb[RS_RADIX];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int t = threadIdx.x; t < RS_WARPS * RS_RADIX; t += RS_THREADS) (&wh[0][0])[t] = 0;
  for (int t = threadIdx.x; t < RS_RADIX; t += RS_THREADS) gb[t] = hist[(long long)t * ntiles + blockIdx.x];
  __syncthreads();
  long long base = (long long)blockIdx.x * RS_TILE + (long long)w * 32 * RS_ITEMS;
  uint32_t dig[RS_ITEMS], rk[RS_ITEMS];
  unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int k = 0; k < RS_ITEMS; ++k) {
    long long i = base + k * 32 + lane;
    uint32_t d = i < n ? key.digit(i, shift) : RS_RADIX;  // RS_RADIX: past the end
    unsigned peers = __match_any_sync(0xffffffffu, d);
    uint32_t before = 0;
    if (d < RS_RADIX) before = wh[w][d];
    __syncwarp();
    int leader = __ffs(peers) - 1;
    if (d < RS_RADIX && lane == leader) wh[w][d] = before + __popc(peers);
    __syncwarp();
    dig[k] = d;
    rk[k] = before + __popc(peers & lt);
  }
  __syncthreads();
  // exclusive prefix across warps, per digit
  for (int t = threadIdx.x; t < RS_RADIX; t += RS_THREADS) {
    uint32_t run = 0;
#pragma unroll
    for (int q = 0; q < RS_WARPS; ++q) {
      uint32_t c = wh[q][t];
      wh[q][t] = run;
      run += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < RS_ITEMS; ++k) {
    long long i = base + k * 32 + lane;
    if (i < n) move(i, (long long)gb[dig[k]] + wh[w][dig[k]] + rk[k]);
  }
}

__global__ void __launch_bounds__(RS_THREADS)
    k_rs_scatter128(const uint64_t* __restrict__ hi, const uint64_t* __restrict__ lo, const uint32_t* __restrict__ v,
                    uint64_t* __restrict__ hi2, uint64_t* __restrict__ lo2, uint32_t* __restrict__ v2, long long n,
                    int shift, const uint32_t* __restrict__ hist, int ntiles) {
  Key128 key{hi, lo};
  rs_scatter_body(key, n, shift, hist, ntiles, [&](long long i, long long dst) {
    if (hi) hi2[dst] = hi[i];
    lo2[dst] = lo[i];
    v2[dst] = v[i];
  });
}

// --------------------------------------------------------------------------
// one-sweep radix sort (keys of up to 64 bits)
//
// In the spirit of Adinets and Merrill, "Onesweep: A Faster Least Significant
// Digit Radix Sort for GPUs" (2022): the digit histograms of every pass come
// from one upfront read of the keys, and each pass is a single kernel.  Its
// tiles take their index from an atomic counter (every predecessor of a tile
// is already running), rank their elements per 8-bit digit with warp-level
// matching (stable), publish per-digit counts and find each digit's
// exclusive prefix over the earlier tiles by a decoupled look-back (one
// thread per digit), then stage the tile in digit order in shared memory so
// that the writes to each digit's run are coalesced.  Status words are
// flag << 32 | count; the flags carry the pass number (2p + 1: tile count,
// 2p + 2: inclusive prefix), so one clearing serves every pass of a sort.
// --------------------------------------------------------------------------
constexpr int OS_THREADS = 256;
constexpr int OS_WARPS = OS_THREADS / 32;
constexpr int OS_RADIX = 256;
constexpr int OS_MAX_PASSES = 8;
constexpr int OS_LB = 8;  // predecessors read per look-back round trip

template <class K>
struct OsItems;
template <>
struct OsItems<uint64_t> {  // 3072-element tiles: 36 KB of staging
  static constexpr int v = 12;
};
template <>
struct OsItems<uint32_t> {  // 4096-element tiles: 32 KB of staging
  static constexpr int v = 16;
};

template <class K>
__global__ void __launch_bounds__(OS_THREADS) k_os_hist(const K* __restrict__ key, long long n, int passes,
                                                      uint32_t* __restrict__ ghist) {
  __shared__ uint32_t h[OS_MAX_PASSES][OS_RADIX];
  for (int t = threadIdx.x; t < OS_MAX_PASSES * OS_RADIX; t += OS_THREADS) (&h[0][0])[t] = 0;
  __syncthreads();
  for (long long i = (long long)blockIdx.x * OS_THREADS + threadIdx.x; i < n; i += (long long)gridDim.x * OS_THREADS) {
    const K k = key[i];
    for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(uint32_t)(k >> (8 * p)) & 255u], 1u);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < passes * OS_RADIX; t += OS_THREADS) {
    const uint32_t v = (&h[0][0])[t];
    if (v) atomicAdd(&ghist[t], v);
  }
}

// each pass's histogram to exclusive digit bases (one block per pass)
__global__ void __launch_bounds__(OS_RADIX) k_os_bases(uint32_t* __restrict__ ghist) {
  __shared__ uint32_t sw[33];
  uint32_t* h = ghist + (size_t)blockIdx.x * OS_RADIX;
  uint32_t excl;
  block_excl_scan(h[threadIdx.x], sw, excl);
  h[threadIdx.x] = excl;
}

template <class K>
__global__ void __launch_bounds__(OS_THREADS, 4) k_os_pass(const K* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                      K* __restrict__ kout, uint32_t* __restrict__ vout, long long n,
                                                      int pass, const uint32_t* __restrict__ gbase,
                                                      unsigned long long* __restrict__ status,
                                                      unsigned* __restrict__ ctr, long long patience) {
  constexpr int ITEMS = OsItems<K>::v;
  constexpr int TILE = OS_THREADS * ITEMS;
  __shared__ K skey[TILE];
  __shared__ uint32_t sval[TILE];
  __shared__ uint32_t wh[OS_WARPS][OS_RADIX];
  __shared__ uint32_t dpre[OS_RADIX];
  __shared__ long long gofs[OS_RADIX];
  __shared__ uint32_t sw[33];
  __shared__ unsigned tile_sh;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) tile_sh = atomicAdd(ctr, 1u);
  for (int t = threadIdx.x; t < OS_WARPS * OS_RADIX; t += OS_THREADS) (&wh[0][0])[t] = 0;
  __syncthreads();
  const long long tile = tile_sh;
  const int shift = 8 * pass;
  // warp w holds a contiguous run of the tile, 32 consecutive elements per item
  const long long base = tile * TILE + (long long)w * 32 * ITEMS;
  K key[ITEMS];
  uint32_t val[ITEMS], dr[ITEMS];  // dr: rank in the warp's run << 9 | digit (256: past the end)
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const long long e = base + k * 32 + lane;
    const bool v = e < n;
    key[k] = v ? kin[e] : K(0);
    val[k] = v ? vin[e] : 0u;
    const uint32_t d = v ? ((uint32_t)(key[k] >> shift) & 255u) : (uint32_t)OS_RADIX;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    uint32_t before = 0;
    if (d < OS_RADIX) before = wh[w][d];
    __syncwarp();
    if (d < OS_RADIX && lane == __ffs(peers) - 1) wh[w][d] = before + __popc(peers);
    __syncwarp();
    dr[k] = ((before + __popc(peers & lt)) << 9) | d;
  }
  __syncthreads();
  // thread d: digit d's per-warp prefix and the tile's count
  const int d = threadIdx.x;
  uint32_t cnt = 0;
#pragma unroll
  for (int q = 0; q < OS_WARPS; ++q) {
    const uint32_t c = wh[q][d];
    wh[q][d] = cnt;
    cnt += c;
  }
  // publish the tile's count of digit d, then stage the tile in digit order
  // (tile-local offsets only) before the look-back, so the keys leave the
  // registers before the wait
  const unsigned long long FA = (unsigned long long)(2 * pass + 1) << 32;
  const unsigned long long FP = (unsigned long long)(2 * pass + 2) << 32;
  if (tile > 0) sp_store(&status[tile * OS_RADIX + d], FA | cnt);
  uint32_t dex;
  block_excl_scan(cnt, sw, dex);
  dpre[d] = dex;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const uint32_t dk = dr[k] & 511u;
    if (dk < OS_RADIX) {
      const uint32_t pos = dpre[dk] + wh[w][dk] + (dr[k] >> 9);
      skey[pos] = key[k];
      sval[pos] = val[k];
    }
  }
  // decoupled look-back over the earlier tiles' counts of digit d: OS_LB
  // predecessors per round trip, nearest first, adding counts up to the first
  // inclusive prefix; a predecessor that has not published yet is read again,
  // and counted here when the patience is used up
  uint32_t excl = 0;
  if (tile > 0) {
    long long j = tile - 1, spins = 0;
    while (j >= 0) {
      unsigned long long wv[OS_LB];
#pragma unroll
      for (int q = 0; q < OS_LB; ++q) wv[q] = j - q >= 0 ? sp_load(&status[(j - q) * OS_RADIX + d]) : FP;
      int used = 0;
      bool done = false, wait = false;
#pragma unroll
      for (int q = 0; q < OS_LB; ++q) {
        if (done || wait) continue;
        const unsigned long long f = wv[q] & 0xffffffff00000000ull;
        if (f < FA) {  // not yet published in this pass
          wait = true;
          continue;
        }
        excl += (uint32_t)wv[q];
        ++used;
        done = f == FP;
      }
      if (done) break;
      j -= used;
      if (wait && spins++ >= patience) {
        const K* at = kin + j * TILE;
        uint32_t c = 0;
#pragma unroll 1
        for (int e = 0; e < TILE; ++e) c += ((uint32_t)(at[e] >> shift) & 255u) == (uint32_t)d;
        excl += c;
        --j;
      }
    }
  }
  sp_store(&status[tile * OS_RADIX + d], FP | (excl + cnt));
  gofs[d] = (long long)gbase[d] + excl - dex;
  __syncthreads();
  const long long left = n - tile * TILE;
  const int tn = left < TILE ? (int)left : TILE;
  for (int pos = threadIdx.x; pos < tn; pos += OS_THREADS) {
    const K kk = skey[pos];
    const long long dst = gofs[(uint32_t)(kk >> shift) & 255u] + pos;
    kout[dst] = kk;
    vout[dst] = sval[pos];
  }
}

// Small arrays by one block: the whole scan and the whole sort in one launch
// each, where the general kernels need a clearing, a launch per digit and two
// more (a launch costs 2-4 us beside others; the work itself less).
constexpr int SMALL_SCAN = 8192;
constexpr int SMALL_SORT = 2048;

__global__ void __launch_bounds__(1024) k_scan_small(uint32_t* __restrict__ d, int n, uint32_t* __restrict__ total) {
  __shared__ uint32_t sw[33];
  uint32_t carry = 0;
  for (int base = 0; base < n; base += 4096) {
    const int i = base + threadIdx.x * 4;
    uint32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = i + k < n ? d[i + k] : 0u;
    uint32_t excl;
    const uint32_t sum = block_excl_scan(v[0] + v[1] + v[2] + v[3], sw, excl);
    uint32_t at = carry + excl;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (i + k < n) d[i + k] = at;
      at += v[k];
    }
    carry += sum;
  }
  if (total && threadIdx.x == 0) *total = carry;
}

// Sorts (key, position) by the masked key in shared memory: bitonic over
// twice as many elements as threads; the position makes it stable.
template <class K>
__global__ void __launch_bounds__(SMALL_SORT / 2) k_sort_small(const K* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                             K* __restrict__ kout, uint32_t* __restrict__ vout, int n,
                                                             int m, K mask) {
  __shared__ K sk[SMALL_SORT];
  __shared__ uint16_t sp[SMALL_SORT];
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    sk[i] = i < n ? kin[i] & mask : K(~K(0));
    sp[i] = (uint16_t)i;  // past the end: behind every element of the same key
  }
  __syncthreads();
  for (int k = 2; k <= m; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < m / 2; t += blockDim.x) {
        const int i = 2 * t - (t & (j - 1)), l = i + j;
        const K a = sk[i], b = sk[l];
        const uint16_t pa = sp[i], pb = sp[l];
        const bool gt = a > b || (a == b && pa > pb);
        if (gt == ((i & k) == 0)) {
          sk[i] = b;
          sk[l] = a;
          sp[i] = pb;
          sp[l] = pa;
        }
      }
      __syncthreads();
    }
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    kout[i] = kin[sp[i]];
    vout[i] = vin[sp[i]];
  }
}

}  // namespace

int scan_u32(uint32_t* data, long long n, uint32_t* total, Workspace& ws, cudaStream_t st, const uint16_t* half,
             const int* over) {
  if (n <= 0) {
    if (total) CSO_CUDA(cudaMemsetAsync(total, 0, sizeof(uint32_t), st));
    return CSO_OK;
  }
  if (n <= SMALL_SCAN && !half) {
    k_scan_small<<<CL(1), 1024, 0, st>>>(data, (int)n, total);
    CSO_CUDA(cudaGetLastError());
    return CSO_OK;
  }
  // at most SMALL_SCAN blocks, so that one block scans their sums
  const int rounds = 4 * (int)cdiv(n, (long long)SMALL_SCAN * SC_WARPS * 128 * 4);
  const int nb = (int)cdiv(n, (long long)SC_WARPS * 128 * rounds);
  const size_t mark = ws.off;
  uint32_t* run_base = ws.get<uint32_t>((size_t)nb * SC_WARPS);
  uint32_t* block_sum = ws.get<uint32_t>(nb);
  if (!run_base || !block_sum) {
    cso_set_error("workspace exhausted in scan");
    return CSO_ERR_BUDGET;
  }
  const ScanIn in{data, half, over};
  k_scan_sums<<<CL(nb), SC_WARPS * 32, 0, st>>>(in, n, rounds, run_base, block_sum);
  k_scan_small<<<CL(1), 1024, 0, st>>>(block_sum, nb, total);
  k_scan_apply<<<CL(nb), SC_WARPS * 32, 0, st>>>(in, data, n, rounds, run_base, block_sum);
  CSO_CUDA(cudaGetLastError());
  ws.off = mark;
  return CSO_OK;
}

template <class K>
static int onesweep(K** key, uint32_t** val, K* key_alt, uint32_t* val_alt, long long n, int bits, Workspace& ws,
                    cudaStream_t st) {
  if (n <= SMALL_SORT) {
    int m = 2;
    while (m < n) m <<= 1;
    const int b8 = (bits + 7) / 8 * 8;  // whole digits, as the passes below
    const K mask = b8 >= (int)(8 * sizeof(K)) ? K(~K(0)) : K((K(1) << b8) - 1);
    k_sort_small<K><<<CL(1), m / 2 < 32 ? 32 : m / 2, 0, st>>>(*key, *val, key_alt, val_alt, (int)n, m, mask);
    CSO_CUDA(cudaGetLastError());
    std::swap(*key, key_alt);
    std::swap(*val, val_alt);
    return CSO_OK;
  }
  constexpr int TILE = OS_THREADS * OsItems<K>::v;
  const int passes = (bits + 7) / 8;
  const long long ntiles = cdiv(n, TILE);
  const size_t mark = ws.off;
  unsigned long long* status = ws.get<unsigned long long>((size_t)ntiles * OS_RADIX);
  uint32_t* aux = ws.get<uint32_t>((size_t)passes * OS_RADIX + passes);  // histograms, then tile counters
  if (!status || !aux) {
    cso_set_error("workspace exhausted in radix sort");
    return CSO_ERR_BUDGET;
  }
  CSO_CUDA(cudaMemsetAsync(status, 0, sizeof(unsigned long long) * ntiles * OS_RADIX, st));
  CSO_CUDA(cudaMemsetAsync(aux, 0, sizeof(uint32_t) * ((size_t)passes * OS_RADIX + passes), st));
  const long long hb = std::min<long long>(cdiv(n, (long long)OS_THREADS * 16), (long long)cso_sm_count() * 8);
  k_os_hist<K><<<CL((unsigned)hb), OS_THREADS, 0, st>>>(*key, n, passes, aux);
  k_os_bases<<<passes, OS_RADIX, 0, st>>>(aux);
  for (int p = 0; p < passes; ++p) {
    k_os_pass<K><<<CL((unsigned)ntiles), OS_THREADS, 0, st>>>(*key, *val, key_alt, val_alt, n, p,
                                                               aux + (size_t)p * OS_RADIX, status,
                                                               aux + (size_t)passes * OS_RADIX + p, ws.patience);
    K* t1 = *key;
    *key = key_alt;
    key_alt = t1;
    uint32_t* t2 = *val;
    *val = val_alt;
    val_alt = t2;
  }
  CSO_CUDA(cudaGetLastError());
  ws.off = mark;
  return CSO_OK;
}

int radix_sort_128(uint64_t** khi, uint64_t** klo, uint32_t** val, uint64_t* khi_alt, uint64_t* klo_alt,
                   uint32_t* val_alt, long long n, int bits, Workspace& ws, cudaStream_t st) {
  if (n <= 1 || bits <= 0) return CSO_OK;
  // keys of up to 64 bits: the low word alone, one kernel per pass
  if (bits <= 64) return onesweep<uint64_t>(klo, val, klo_alt, val_alt, n, bits, ws, st);
  int ntiles = (int)cdiv(n, RS_TILE);
  size_t mark = ws.off;
  uint32_t* hist = ws.get<uint32_t>((size_t)ntiles * RS_RADIX);
  if (!hist) {
    cso_set_error("workspace exhausted in radix sort");
    return CSO_ERR_BUDGET;
  }
  bool with_hi = bits > 64;
  for (int shift = 0; shift < bits; shift += 8) {
    Key128 key{with_hi ? *khi : nullptr, *klo};
    k_rs_hist<<<CL(ntiles), RS_THREADS, 0, st>>>(key, n, shift, hist, ntiles);
    CSO_TRY(scan_u32(hist, (long long)ntiles * RS_RADIX, nullptr, ws, st));
    k_rs_scatter128<<<CL(ntiles), RS_THREADS, 0, st>>>(with_hi ? *khi : nullptr, *klo, *val, khi_alt, klo_alt, val_alt, n,
                                                   shift, hist, ntiles);
    CSO_CUDA(cudaGetLastError());
    uint64_t* t1 = *khi; *khi = khi_alt; khi_alt = t1;
    uint64_t* t2 = *klo; *klo = klo_alt; klo_alt = t2;
    uint32_t* t3 = *val; *val = val_alt; val_alt = t3;
  }
  ws.off = mark;
  return CSO_OK;
}

int radix_sort_32(uint32_t** key, uint32_t** val, uint32_t* key_alt, uint32_t* val_alt, long long n, int bits,
                  Workspace& ws, cudaStream_t st) {
  if (n <= 1 || bits <= 0) return CSO_OK;
  return onesweep<uint32_t>(key, val, key_alt, val_alt, n, bits, ws, st);
}
