// Local density peaks (Sec. 2.2.2 step 2): the nucleus candidates of a level.
//
// A nucleus must be denser than every other particle of its group within b.
// That does not change while nuclei are accepted, so all peaks are found
// once, by the whole GPU, before the nucleus loops run, and those only choose
// among the few peaks of their group; no loop waits for peak tests, and the
// members of a group need no order by density.  (Tests inside the loops, in
// batches of eligible candidates, were the larger part of the biggest groups'
// serial chain.)
//
// Almost every member has a denser neighbour close by, and cells are sorted
// by x, so a lane first looks at the slots next to its own in the sorted
// order; the few members left (about one per warp) get a warp each over the
// 27-cell stencil, own row first, 128 neighbours a step; a test still open
// after PEAK_STEPS steps (a true peak, mostly) goes to a block of its own.
// Three kernels, so that the first, which sees every member, runs at full
// occupancy.
#include <limits.h>

#include "peaks.cuh"

namespace {

constexpr int NEAR = 16;        // slots looked at on either side
constexpr int PEAK_U = 4;       // neighbours per lane and step
constexpr int PEAK_STEPS = 4;   // steps before a test goes to a block
constexpr int OPEN_NT = 256;

// The neighbours are the runs of the 27-cell stencil, nine rows (own row
// first, where a denser neighbour usually sits), each one run plus one where
// the row wraps; rows and end cells that cannot reach within b are dropped.
struct PeakRows {
  uint32_t lo0, hi0, lo1, hi1;  // lanes 0-8: row lane's runs (rows in walk order)
  int qx1, qy, qz;              // the query in that row's image
  uint32_t pre;                 // lanes 0-9: neighbours in the rows before this one
};

__device__ __forceinline__ int peak_row_of(int o) { return o == 0 ? 4 : (o <= 4 ? o - 1 : o); }

__device__ PeakRows peak_rows(const PeakArgs& a, int4 p) {
  const int lane = threadIdx.x & 31;
  const CellGrid& g = a.grid;
  const int nc = g.nc;
  const int cy = cell_coord(p.y, nc), cz = cell_coord(p.z, nc);
  const int tc = grid_col(g, p.x);
  const XCells X = x_cells(g, tc);
  PeakRows R{0, 0, 0, 0, p.x, p.y, p.z, 0};
  if (lane < 9) {
    const int r = peak_row_of(lane);
    const int dz = r / 3 - 1, dy = r % 3 - 1;
    const int gx = (p.x + g.x0) & (CSO_BOX - 1), gcx = cell_coord(gx, nc);
    const long long zl = p.z - cell_lo(cz, nc) + 1, zr = cell_lo(cz + 1, nc) - p.z;
    const long long yl = p.y - cell_lo(cy, nc) + 1, yr = cell_lo(cy + 1, nc) - p.y;
    const long long xl = gx - cell_lo(gcx, nc) + 1, xr = cell_lo(gcx + 1, nc) - gx;
    const long long m = (dz < 0 ? zl * zl : (dz > 0 ? zr * zr : 0)) + (dy < 0 ? yl * yl : (dy > 0 ? yr * yr : 0));
    if (m < (long long)a.b2) {
      int sz, sy;
      const int zz = wrap_yz(cz + dz, nc, sz), yy = wrap_yz(cy + dy, nc, sy);
      R.qz += sz;
      R.qy += sy;
      const uint32_t* row = grid_row(g, zz, yy);
      const bool left = m + xl * xl < (long long)a.b2, right = m + xr * xr < (long long)a.b2;
      const int ca = left ? X.a : tc, cb = right ? X.b : tc;
      if (left && X.wl >= 0) { R.lo1 = row[X.wl]; R.hi1 = row[X.wl + 1]; R.qx1 = p.x + CSO_BOX; }
      if (right && X.wr >= 0) { R.lo1 = row[X.wr]; R.hi1 = row[X.wr + 1]; R.qx1 = p.x - CSO_BOX; }
      R.lo0 = row[ca];
      R.hi0 = row[cb + 1];
    }
  }
  // exclusive prefix of the rows' neighbour counts (lane 9 holds the total)
  const uint32_t cnt = lane < 9 ? (R.hi0 - R.lo0) + (R.hi1 - R.lo1) : 0u;
  uint32_t inc = cnt;
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  R.pre = inc - cnt;
  return R;
}

// One step of the test: neighbours f0 + k * 32 + lane (k < PEAK_U) of the
// flattened rows; returns a particle that beats se, or -1.  Every load of the
// step is issued before any comparison, so a step costs one memory round trip.
__device__ __forceinline__ int peak_step(const PeakArgs& a, const PeakRows& R, uint32_t f0, uint32_t total, uint32_t se,
                                         int glabel, int4 p, long long sp, uint64_t idp) {
  const int lane = threadIdx.x & 31;
  int4 q[PEAK_U];
  int lab[PEAK_U];
  long long st[PEAK_U];
  uint32_t tt[PEAK_U];
  int ow[PEAK_U];  // row (walk order) | 16 for the wrapped run
#pragma unroll
  for (int k = 0; k < PEAK_U; ++k) {
    const uint32_t f = f0 + k * 32 + lane;
    // the row holding f: the last o with pre[o] <= f
    int o = 0;
#pragma unroll
    for (int oo = 1; oo < 9; ++oo)
      if (__shfl_sync(0xffffffffu, R.pre, oo) <= f) o = oo;
    const uint32_t r = f - __shfl_sync(0xffffffffu, R.pre, o);
    const uint32_t l0 = __shfl_sync(0xffffffffu, R.lo0, o), n0 = __shfl_sync(0xffffffffu, R.hi0, o) - l0;
    const uint32_t l1 = __shfl_sync(0xffffffffu, R.lo1, o);
    tt[k] = f < total ? (r < n0 ? l0 + r : l1 + (r - n0)) : se;
    ow[k] = o | (r < n0 ? 0 : 16);
    q[k] = a.spos[tt[k]];
    lab[k] = a.slab[tt[k]];
    st[k] = a.ssig[tt[k]];
  }
  int beat = -1;
#pragma unroll
  for (int k = 0; k < PEAK_U; ++k) {
    const int o = ow[k] & 15;
    const int x1 = __shfl_sync(0xffffffffu, R.qx1, o), yq = __shfl_sync(0xffffffffu, R.qy, o),
              zq = __shfl_sync(0xffffffffu, R.qz, o);
    if (tt[k] == se || lab[k] != glabel) continue;  // past the end (tt = se), self, or another group
    const int dx = (ow[k] & 16 ? x1 : p.x) - q[k].x, dy = yq - q[k].y, dz = zq - q[k].z;
    const uint32_t d = (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
    if (d < a.b2 && (st[k] > sp || (st[k] == sp && a.sid[tt[k]] < idp))) beat = (int)tt[k];
  }
  const unsigned any = __ballot_sync(0xffffffffu, beat >= 0);
  return any ? __shfl_sync(0xffffffffu, beat, __ffs(any) - 1) : -1;
}

constexpr int BEAT_NONE = -1;  // no beater: a peak
constexpr int BEAT_OPEN = -2;  // not finished

// The test by one warp, at most `steps` steps.
__device__ int warp_peak(const PeakArgs& a, uint32_t se, int glabel, int steps) {
  const int4 p = a.spos[se];
  const long long sp = a.ssig[se];
  const uint64_t idp = a.sid[se];
  const PeakRows R = peak_rows(a, p);
  const uint32_t total = __shfl_sync(0xffffffffu, R.pre, 9);
  for (uint32_t f0 = 0; f0 < total; f0 += 32 * PEAK_U) {
    if (steps-- <= 0) return BEAT_OPEN;
    const int b = peak_step(a, R, f0, total, se, glabel, p, sp, idp);
    if (b >= 0) return b;
  }
  return BEAT_NONE;
}

struct PeakOut {
  uint2* found;        // (segment, cell-sorted index) of every peak, unordered
  uint2* left;         // members for a warp's test
  uint2* open;         // tests for a block
  unsigned m;          // members in all (room in each list)
  unsigned* counts;    // [0] found, [1] left for a warp, [2] left for a block
  uint32_t* seg_count; // peaks per segment
};

// the calling thread's peak
__device__ __forceinline__ void add_peak(const PeakOut& o, uint32_t seg, uint32_t s) {
  o.found[atomicAdd(&o.counts[0], 1u)] = make_uint2(seg, s);
  atomicAdd(&o.seg_count[seg], 1u);
}

__global__ void __launch_bounds__(256) k_peak_near(PeakArgs a, const uint32_t* __restrict__ gs,
                                                   const uint32_t* __restrict__ seg, long long T_min, long long T_test,
                                                   int first, int* __restrict__ beater, PeakOut out) {
  const unsigned k = blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = k < out.m;
  const uint32_t s = in ? gs[k] : 0u;
  const long long sp = in ? a.ssig[s] : LLONG_MIN;
  const bool test = in && sp > T_test;
  bool todo = test;
  int beat = BEAT_OPEN, lab = -1;
  if (!first) {
    if (todo) {
      beat = beater[s];
      lab = a.slab[s];
      // known: a peak, or beaten inside its segment
      if (beat != BEAT_NONE && a.slab[beat] != lab) beat = BEAT_OPEN;
    }
  } else {
    // the slots next to its own: any particle of the group there that is
    // within b and denser settles it
    int4 p = make_int4(0, 0, 0, 0);
    uint64_t id = 0;
    if (todo) {
      p = a.spos[s];
      id = a.sid[s];
      lab = a.slab[s];
    }
    for (int o0 = 1; o0 <= NEAR; o0 += 4) {
      if (!__any_sync(0xffffffffu, todo)) break;
      long long st[8];  // eight loads in flight
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const long long t = (long long)s + (u & 1 ? -(o0 + u / 2) : o0 + u / 2);
        st[u] = todo && t >= 0 && t < a.n ? a.ssig[t] : LLONG_MIN;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = (int)s + (u & 1 ? -(o0 + u / 2) : o0 + u / 2);
        if (!todo || st[u] < sp || a.slab[t] != lab) continue;
        const int4 q = a.spos[t];
        // nearest image by sign extension from 21 bits; a slot next to this
        // one may be anywhere, so each offset is bounded before it is squared
        const int dx = (int)((unsigned)(p.x - q.x) << 11) >> 11, dy = (int)((unsigned)(p.y - q.y) << 11) >> 11,
                  dz = (int)((unsigned)(p.z - q.z) << 11) >> 11;
        if (max(abs(dx), max(abs(dy), abs(dz))) > 16384) continue;  // b <= 16,384 grid units
        const uint32_t d = (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
        if (d >= a.b2 || (st[u] == sp && a.sid[t] >= id)) continue;
        beat = t;
        todo = false;
      }
    }
  }
  if (!test) return;
  if (beat == BEAT_OPEN) {
    out.left[atomicAdd(&out.counts[1], 1u)] = make_uint2(seg[k], s);
  } else {
    if (first) beater[s] = beat;
    else if (beat == BEAT_NONE && sp > T_min) add_peak(out, seg[k], s);
  }
}

// the members left, a warp each for at most PEAK_STEPS steps
__global__ void __launch_bounds__(256) k_peak_warp(PeakArgs a, long long T_min, int first, int* __restrict__ beater,
                                                   PeakOut out) {
  const int lane = threadIdx.x & 31;
  const unsigned m = out.counts[1];
  for (unsigned i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < m; i += gridDim.x * blockDim.x >> 5) {
    const uint2 o = out.left[i];
    const int b = warp_peak(a, o.y, a.slab[o.y], PEAK_STEPS);
    if (lane != 0) continue;
    if (b == BEAT_OPEN) {
      out.open[atomicAdd(&out.counts[2], 1u)] = o;
    } else {
      if (first) beater[o.y] = b;
      if (b == BEAT_NONE && a.ssig[o.y] > T_min) add_peak(out, o.x, o.y);
    }
  }
}

// the tests left open, a block each: its warps share the neighbours step by step
__global__ void __launch_bounds__(OPEN_NT) k_peak_open(PeakArgs a, long long T_min, int first,
                                                       int* __restrict__ beater, PeakOut out) {
  __shared__ int hit;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned m = out.counts[2];
  for (unsigned i = blockIdx.x; i < m; i += gridDim.x) {
    const uint2 o = out.open[i];
    if (threadIdx.x == 0) hit = BEAT_NONE;
    __syncthreads();
    const int4 p = a.spos[o.y];
    const long long sp = a.ssig[o.y];
    const uint64_t idp = a.sid[o.y];
    const int lab = a.slab[o.y];
    const PeakRows R = peak_rows(a, p);
    const uint32_t total = __shfl_sync(0xffffffffu, R.pre, 9);
    for (uint32_t f0 = (uint32_t)warp * 32 * PEAK_U; f0 < total; f0 += OPEN_NT * PEAK_U) {
      const int b = peak_step(a, R, f0, total, o.y, lab, p, sp, idp);
      if (b >= 0) {
        if (lane == 0) atomicExch(&hit, b);
        break;
      }
      // another warp's beater ends the test (one lane reads, so that the warp agrees)
      if (__shfl_sync(0xffffffffu, *(volatile int*)&hit, 0) >= 0) break;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      if (first) beater[o.y] = hit;
      if (hit == BEAT_NONE && sp > T_min) add_peak(out, o.x, o.y);
    }
    __syncthreads();
  }
}

// the peaks into their segments' places
__global__ void k_peak_place(PeakArgs a, const uint2* __restrict__ found, const unsigned* __restrict__ counts,
                             uint32_t* __restrict__ cursor, PeakList P) {
  const unsigned m = counts[0];
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const uint2 f = found[i];
    const uint32_t d = P.off[f.x] + atomicAdd(&cursor[f.x], 1u);
    int4 p = a.spos[f.y];
    p.w = (int)f.y;
    P.pos[d] = p;
    P.sig[d] = a.ssig[f.y];
    P.id[d] = a.sid[f.y];
    P.out[d] = 0;
  }
}

}  // namespace

int peaks_find(const PeakArgs& a, const uint32_t* gs, const uint32_t* seg, int m, int nseg, long long T_min,
               long long T_test, bool first, int* beater, PeakList& P, Workspace& ws, cudaStream_t st) {
  P.off = ws.get<uint32_t>((size_t)nseg + 1);
  if (!P.pos) {
    P.pos = ws.get<int4>(m);
    P.sig = ws.get<long long>(m);
    P.id = ws.get<uint64_t>(m);
    P.out = ws.get<uint8_t>(m);
  }
  const size_t mark = ws.off;
  PeakOut o;
  o.found = ws.get<uint2>(m);
  o.left = ws.get<uint2>(m);
  o.open = ws.get<uint2>(m);
  o.m = (unsigned)m;
  uint32_t* cursor = ws.get<uint32_t>((size_t)nseg + 3);
  if (!P.off || !P.pos || !P.sig || !P.id || !P.out || !o.found || !o.left || !o.open || !cursor) {
    cso_set_error("workspace exhausted in the peak search");
    return CSO_ERR_BUDGET;
  }
  o.counts = cursor + nseg;
  o.seg_count = P.off;
  CSO_CUDA(cudaMemsetAsync(P.off, 0, sizeof(uint32_t) * ((size_t)nseg + 1), st));
  CSO_CUDA(cudaMemsetAsync(cursor, 0, sizeof(uint32_t) * ((size_t)nseg + 3), st));
  if (m > 0) {
    k_peak_near<<<CL(cdiv(m, 256)), 256, 0, st>>>(a, gs, seg, T_min, T_test, first, beater, o);
    k_peak_warp<<<CL(cso_sm_count() * 8), 256, 0, st>>>(a, T_min, first, beater, o);
    k_peak_open<<<CL(cso_sm_count() * 8), OPEN_NT, 0, st>>>(a, T_min, first, beater, o);
    CSO_TRY(scan_u32(P.off, nseg, P.off + nseg, ws, st));
    k_peak_place<<<CL(cso_sm_count()), 256, 0, st>>>(a, o.found, o.counts, cursor, P);
    CSO_CUDA(cudaGetLastError());
  }
  ws.off = mark;
  return CSO_OK;
}
