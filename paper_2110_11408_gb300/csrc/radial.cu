// Radial statistics of L1 haloes (Table 1: r_XX_L2com, vcirc_max_L2com,
// rvcirc_max_L2com; Sec. 4).
//
// Every member's squared distance to its halo's centre (the grid point
// nearest the L2max centre of mass) is an exact integer, so the statistics are
// order statistics of integers: the members of all haloes are sorted once by
// (halo, d) with the device radix sort, which leaves each halo's distances
// ascending in the halo's own segment.  A block per halo then reads the four
// enclosed-fraction radii by index and finds the circular-velocity peak
// max N(<= r) / r with an exact 128-bit comparison.
#include <cooperative_groups.h>

#include "radial.cuh"

namespace {

__device__ __forceinline__ long long min_image(int dx) {
  long long d = dx;
  if (d >= (1ll << 20)) d -= CSO_BOX;
  else if (d < -(1ll << 20)) d += CSO_BOX;
  return d;
}

// centre of halo h: nearest grid point of the L2max com (L1 com without L2
// haloes); cen holds it in stored coordinates (x relative to x0)
__global__ void k_radial_centre(const cso_halo* __restrict__ rows, int H, int x0, int4* __restrict__ cen,
                                cso_radial* __restrict__ out) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h >= H) return;
  const cso_halo r = rows[h];
  const double* com = r.n_l2 > 0 ? r.l2max_com : r.com;
  int c[3];
  for (int k = 0; k < 3; ++k) {
    c[k] = (int)(llround(com[k]) & (CSO_BOX - 1));
    out[h].centre[k] = c[k];
  }
  cen[h] = make_int4((c[0] - x0) & (CSO_BOX - 1), c[1], c[2], 0);
}

__global__ void k_radial_dist(const int4* __restrict__ epos, const uint32_t* __restrict__ ehal, long long na,
                              const int4* __restrict__ cen, uint64_t* __restrict__ d,
                              unsigned long long* __restrict__ dmax) {
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long v = 0;
  if (j < na) {
    const int4 q = epos[j];
    const int4 c = cen[ehal[j]];
    const long long dx = min_image(q.x - c.x), dy = min_image(q.y - c.y), dz = min_image(q.z - c.z);
    v = (unsigned long long)(dx * dx + dy * dy + dz * dz);
    d[j] = v;
  }
  unsigned long long best = v;
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, best, o);
    best = t > best ? t : best;
  }
  if ((threadIdx.x & 31) == 0 && best) atomicMax(dmax, best);
}

__global__ void k_radial_pack(uint64_t* __restrict__ key, const uint32_t* __restrict__ ehal, long long na,
                              int dbits) {
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < na) key[j] |= (unsigned long long)ehal[j] << dbits;
}

__global__ void k_radial_hi(uint64_t* __restrict__ hi, const uint32_t* __restrict__ ehal, long long na) {
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < na) hi[j] = ehal[j];
}

// (n_a, d_a) beats (n_b, d_b) when n_a^2 / d_a > n_b^2 / d_b, or the values
// are equal and d_a is smaller; n_b = 0 marks "none yet"
__device__ __forceinline__ bool vbetter(unsigned long long na_, unsigned long long da, unsigned long long nb,
                                        unsigned long long db) {
  if (na_ == 0) return false;
  if (nb == 0) return true;
  const unsigned __int128 l = (unsigned __int128)(na_ * na_) * db;
  const unsigned __int128 r = (unsigned __int128)(nb * nb) * da;
  return l > r || (l == r && da < db);
}

// Haloes by the work they need: a halo below SS_N_MIN members stops at its
// first shrinking sphere; the others take a 256-thread block, a 1024-thread
// block from SS_LARGE members and a cluster of such blocks from SS_BIG.
constexpr long long SS_N_MIN = 700;
constexpr long long SS_LARGE = 4096;
constexpr long long SS_BIG = 16384;
enum : int { SS_MID = 0, SS_LRG, SS_CLU, SS_KINDS };

struct SsLists {  // listed haloes of each kind and their fetch counters
  unsigned n[SS_KINDS], next[SS_KINDS];
};

// Quantiles and the circular-velocity peak from a halo's sorted distances, a
// block per halo: 256 threads, or 1024 for the listed big ones.  The exact
// 128-bit comparison is made only for members whose n^2 / d comes within 1e-5
// of the thread's best in float (relative error below 1e-6), which leaves out
// almost all of them.
template <int NT>
__device__ void radial_stats(const uint64_t* __restrict__ key, unsigned long long dmask, uint32_t b, uint32_t n, double u,
                             cso_radial& r, unsigned long long* sn, unsigned long long* sd) {
  const uint64_t* D = key + b;
  unsigned long long bn = 0, bd = 0;
  float fn2 = 0.f, fd = 1.f;  // the best so far in float
  for (uint32_t i0 = threadIdx.x; i0 < n; i0 += 4 * NT) {
    unsigned long long dq[4];  // four loads in flight
#pragma unroll
    for (int k = 0; k < 4; ++k) dq[k] = i0 + k * NT < n ? D[i0 + k * NT] & dmask : 0ull;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t i = i0 + k * NT;
      const unsigned long long di = dq[k];
      if (di == 0) continue;
      const float cn = (float)(i + 1), cd = (float)di;
      if (cn * cn * fd < fn2 * cd * (1.f - 1e-5f)) continue;
      if (i + 1 < n && (D[i + 1] & dmask) == di) continue;  // N(<= r) takes the whole shell
      if (vbetter(i + 1, di, bn, bd)) {
        bn = i + 1;
        bd = di;
        fn2 = cn * cn;
        fd = cd;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long tn = __shfl_xor_sync(0xffffffffu, bn, o);
    const unsigned long long td = __shfl_xor_sync(0xffffffffu, bd, o);
    if (vbetter(tn, td, bn, bd)) {
      bn = tn;
      bd = td;
    }
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) {
    sn[w] = bn;
    sd[w] = bd;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int k = 1; k < NT / 32; ++k)
    if (vbetter(sn[k], sd[k], bn, bd)) {
      bn = sn[k];
      bd = sd[k];
    }
  const int pct[4] = {25, 50, 75, 98};
  for (int q = 0; q < 4; ++q) {
    long long m = ((long long)pct[q] * n + 99) / 100;
    if (m < 1) m = 1;
    const unsigned long long dq = n > 0 ? (D[m - 1] & dmask) : 0;
    r.d_q[q] = (int64_t)dq;
    r.r_q[q] = sqrt((double)dq) / u;
  }
  r.vmax_n = (int64_t)bn;
  r.vmax_d2 = (int64_t)bd;
  r.r_vmax = sqrt((double)bd) / u;
  r.vmax = bn > 0 ? sqrt((double)bn / r.r_vmax) : 0.0;
}

__global__ void __launch_bounds__(256) k_radial_stats(const uint64_t* __restrict__ key, unsigned long long dmask,
                                                      const uint32_t* __restrict__ seg, double u,
                                                      cso_radial* __restrict__ out) {
  __shared__ unsigned long long sn[8], sd[8];
  const int h = blockIdx.x;
  const uint32_t b = seg[h], n = seg[h + 1] - b;
  if (n < SS_BIG) radial_stats<256>(key, dmask, b, n, u, out[h], sn, sd);
}

__global__ void __launch_bounds__(1024) k_radial_stats_big(const uint64_t* __restrict__ key, unsigned long long dmask,
                                                           const uint32_t* __restrict__ seg, double u,
                                                           const uint32_t* __restrict__ list, const SsLists* L,
                                                           cso_radial* __restrict__ out) {
  __shared__ unsigned long long sn[32], sd[32];
  for (unsigned it = blockIdx.x; it < L->n[SS_CLU]; it += gridDim.x) {
    const uint32_t h = list[it], b = seg[h], n = seg[h + 1] - b;
    radial_stats<1024>(key, dmask, b, n, u, out[h], sn, sd);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Shrinking-sphere centre.  A halo below SS_N_MIN members stops at its first
// sphere, so a warp counts it.  For the others every step is one pass over
// the members that can lie in the sphere (count and summed minimum-image
// offsets of those inside), then the centre moves to the rounded centre of
// mass and the radius shrinks, or the loop stops.  The sums are exact
// integers, so neither the order nor the split of the members matters.
//
// A pass also lists the members it finds inside.  Where the next sphere lies
// within the one just counted (the centre moved by no more than the radius
// shrank, the usual case), that list is all the next pass needs; otherwise the
// list before it serves if the next sphere lies within its sphere, and the
// whole halo if not.  The lists shrink with the sphere, so a halo costs about
// twenty passes over its members instead of eighty.  The blocks of a cluster
// each have their own share of the members and add up their sums in one
// another's shared memory.  The three kinds run at the same time, beside the
// distances' sort (the loops are eighty dependent steps of a microsecond or
// two, which leave the GPU idle).  One block per halo and a pass over all its
// members per step took 4.1 ms for a halo of 150,000 members.
// ---------------------------------------------------------------------------
namespace cg = cooperative_groups;

constexpr int SS_CS = 8;
constexpr int SS_U = 4;  // members a lane loads before it looks at the first

__global__ void __launch_bounds__(256) k_ss_small(const int4* __restrict__ epos, const uint32_t* __restrict__ seg,
                                                  int H, const int4* __restrict__ nuc_pos,
                                                  const uint32_t* __restrict__ hnuc,
                                                  const cso_halo* __restrict__ rows, int x0, uint32_t* __restrict__ list,
                                                  SsLists* L,
                                                  cso_radial* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int h = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (h >= H) return;
  const uint32_t b = seg[h];
  const long long N = seg[h + 1] - b;
  if (N >= SS_N_MIN) {
    const int kind = N >= SS_BIG ? SS_CLU : N >= SS_LARGE ? SS_LRG : SS_MID;
    if (lane == 0) list[(size_t)kind * H + atomicAdd(&L->n[kind], 1u)] = (uint32_t)h;
    return;
  }
  const int4 c = nuc_pos[hnuc[h]];
  const long long R2 = rows[h].R2;
  unsigned cnt = 0;
  for (long long j = lane; j < N; j += 32) {
    const int4 q = epos[b + j];
    const long long dx = min_image(q.x - c.x), dy = min_image(q.y - c.y), dz = min_image(q.z - c.z);
    cnt += dx * dx + dy * dy + dz * dz < R2;
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) {
    cso_radial& r = out[h];
    r.ss_centre[0] = (c.x + x0) & (CSO_BOX - 1);
    r.ss_centre[1] = c.y;
    r.ss_centre[2] = c.z;
    r.ss_n = cnt;
    r.ss_R2 = R2;
    r.ss_iter = 0;
  }
}

struct Sphere {
  int c[3];
  long long R2;
};

// sphere a within sphere b, in float with a margin far above its rounding
// (radii are at most 2^21 grid units and shrink by 5% a step)
__device__ __forceinline__ bool within(const Sphere& a, const Sphere& b) {
  float m = 0;
  for (int k = 0; k < 3; ++k) {
    const float d = (float)min_image(a.c[k] - b.c[k]);
    m += d * d;
  }
  return (sqrtf(m) + sqrtf((float)a.R2)) * (1.f + 1e-5f) + 2.f <= sqrtf((float)b.R2);
}

struct SsShared {
  long long w[32][4];   // the warps' sums
  long long tot[2][4];  // the block's sums, by step parity (read by the cluster's other blocks)
  Sphere s;             // the sphere to count next
  int src;              // which list it is counted in: 0, 1, or 2 for the whole halo
  int go;
};

// One halo by one block (CS = 1) or a cluster: the ns members at `share` are
// this block's, listed at l0 and l1.  Every warp keeps lists of its own part
// of them, so a pass needs no counter the warps share, and a step two
// barriers: after the sums, and after the first warp's decision.
template <int CS>
__device__ void shrink_halo(const int4* __restrict__ share, unsigned ns, int4* __restrict__ l0, int4* __restrict__ l1,
                            long long N, int4 start, long long R2start, int x0, cso_radial* __restrict__ out,
                            SsShared& B) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const long long stop = (N + 99) / 100 > SS_N_MIN ? (N + 99) / 100 : SS_N_MIN;
  // this warp's part, and the members of its two lists
  const unsigned w0 = (unsigned)((unsigned long long)ns * w / nw), w1 = (unsigned)((unsigned long long)ns * (w + 1) / nw);
  share += w0;
  l0 += w0;
  l1 += w0;
  unsigned m0 = 0, m1 = 0;
  if (threadIdx.x == 0) {
    B.s = Sphere{{start.x, start.y, start.z}, R2start};
    B.src = 2;
  }
  __syncthreads();
  Sphere cover0, cover1;  // (first warp) what the lists hold: every member inside this sphere
  bool have0 = false, have1 = false;
  for (long long iter = 0;; ++iter) {
    const Sphere s = B.s;
    const int src = B.src;
    const int4* from = src == 2 ? share : src ? l1 : l0;
    int4* to = src == 0 ? l1 : l0;
    const unsigned m = src == 2 ? w1 - w0 : src ? m1 : m0;
    long long v[4] = {0, 0, 0, 0};  // count, summed dx, dy, dz
    unsigned kept = 0;
    for (unsigned j0 = 0; j0 < m; j0 += 32 * SS_U) {
      int4 q[SS_U];
#pragma unroll
      for (int u = 0; u < SS_U; ++u) {
        const unsigned j = j0 + u * 32 + lane;
        q[u] = j < m ? from[j] : make_int4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < SS_U; ++u) {
        const long long dx = min_image(q[u].x - s.c[0]), dy = min_image(q[u].y - s.c[1]),
                        dz = min_image(q[u].z - s.c[2]);
        const bool in = j0 + u * 32 + lane < m && dx * dx + dy * dy + dz * dz < s.R2;
        const unsigned mask = __ballot_sync(0xffffffffu, in);
        if (in) {
          v[1] += dx;
          v[2] += dy;
          v[3] += dz;
          to[kept + __popc(mask & ((1u << lane) - 1u))] = q[u];
        }
        kept += __popc(mask);
      }
    }
    if (src == 0) m1 = kept;
    else m0 = kept;
#pragma unroll
    for (int k = 1; k < 4; ++k)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane < 4) B.w[w][lane] = lane == 0 ? (long long)kept : lane == 1 ? v[1] : lane == 2 ? v[2] : v[3];
    __syncthreads();  // (also: the warp's own list is written)
    long long t = 0;  // value lane & 3 of the sums
    if (w == 0) {
      // the block's sums: eight lanes per value, then across them
      for (int x = lane >> 2; x < nw; x += 8) t += B.w[x][lane & 3];
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (CS > 1 && lane < 4) B.tot[iter & 1][lane] = t;
    }
    if (CS > 1) {
      // every block's sums; a block writes the other slot in the next step,
      // and this one again only after that step's barrier
      cg::cluster_group cluster = cg::this_cluster();
      cluster.sync();
      if (w == 0) {
        static_assert(CS == 1 || CS == 8, "eight lanes per value");
        t = cluster.map_shared_rank(&B, lane >> 2)->tot[iter & 1][lane & 3];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      }
    }
    if (w == 0) {
      // the first warp of every block takes the same decision from the same sums
      const long long cnt = __shfl_sync(0xffffffffu, t, 0);
      // lanes 1-3: the centre's coordinates
      const int a = (lane & 3) > 0 ? (lane & 3) - 1 : 0;
      double f = (double)s.c[a] + (double)t / (double)cnt;
      if (f < 0) f += (double)CSO_BOX;
      if (f >= (double)CSO_BOX) f -= (double)CSO_BOX;
      const int c = (int)(llround(f) & (CSO_BOX - 1));
      Sphere nx;
#pragma unroll
      for (int k = 0; k < 3; ++k) nx.c[k] = __shfl_sync(0xffffffffu, c, k + 1);
      nx.R2 = s.R2 * 9025 / 10000;
      if (src == 0) {
        cover1 = s;
        have1 = true;
      } else {
        cover0 = s;
        have0 = true;
      }
      if (lane == 0) {
        B.go = cnt >= stop;
        if (cnt < stop) {
          if (out) {
            out->ss_centre[0] = (s.c[0] + x0) & (CSO_BOX - 1);
            out->ss_centre[1] = s.c[1];
            out->ss_centre[2] = s.c[2];
            out->ss_n = cnt;
            out->ss_R2 = s.R2;
            out->ss_iter = iter;
          }
        } else {
          const int dst = src == 0 ? 1 : 0;
          const bool again = src == 0 ? have0 && within(nx, cover0) : src == 1 && have1 && within(nx, cover1);
          B.src = within(nx, s) ? dst : again ? src : 2;
          B.s = nx;
        }
      }
    }
    __syncthreads();
    if (!B.go) break;
  }
  __syncthreads();
}

template <int NT, int KIND>
__global__ void __launch_bounds__(NT) k_ss_block(const int4* __restrict__ epos, const uint32_t* __restrict__ seg,
                                                 const int4* __restrict__ nuc_pos, const uint32_t* __restrict__ hnuc,
                                                 const cso_halo* __restrict__ rows, int x0,
                                                 const uint32_t* __restrict__ list, SsLists* L, int4* __restrict__ l0,
                                                 int4* __restrict__ l1, cso_radial* __restrict__ out) {
  __shared__ SsShared B;
  __shared__ unsigned item;
  for (;;) {
    if (threadIdx.x == 0) item = atomicAdd(&L->next[KIND], 1u);
    __syncthreads();
    const unsigned it = item;
    __syncthreads();
    if (it >= L->n[KIND]) return;
    const uint32_t h = list[it], b = seg[h], n = seg[h + 1] - b;
    shrink_halo<1>(epos + b, n, l0 + b, l1 + b, n, nuc_pos[hnuc[h]], rows[h].R2, x0, out + h, B);
  }
}

__global__ void __cluster_dims__(SS_CS, 1, 1) __launch_bounds__(1024)
    k_ss_big(const int4* __restrict__ epos, const uint32_t* __restrict__ seg, const int4* __restrict__ nuc_pos,
             const uint32_t* __restrict__ hnuc, const cso_halo* __restrict__ rows, int x0,
             const uint32_t* __restrict__ list, SsLists* L, int4* __restrict__ l0, int4* __restrict__ l1,
             cso_radial* __restrict__ out) {
  __shared__ SsShared B;
  __shared__ unsigned item;
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned rank = cluster.block_rank();
  for (;;) {
    if (rank == 0 && threadIdx.x == 0) item = atomicAdd(&L->next[SS_CLU], 1u);
    cluster.sync();
    const unsigned it = *cluster.map_shared_rank(&item, 0);
    cluster.sync();  // read by all before it changes
    if (it >= L->n[SS_CLU]) return;
    const uint32_t h = list[it], b = seg[h], n = seg[h + 1] - b;
    const uint32_t lo = (uint32_t)((unsigned long long)n * rank / SS_CS);
    const uint32_t hi = (uint32_t)((unsigned long long)n * (rank + 1) / SS_CS);
    shrink_halo<SS_CS>(epos + b + lo, hi - lo, l0 + b + lo, l1 + b + lo, n, nuc_pos[hnuc[h]], rows[h].R2, x0,
                       rank == 0 ? out + h : nullptr, B);
  }
}

}  // namespace

int radial_run(const uint32_t* seg, const uint32_t* ehal, const int4* epos, long long na, const cso_halo* rows,
               int H, int x0, double u, const uint32_t* hnuc, const int4* nuc_pos, cso_radial* out, void* pinned,
               Workspace& ws, cudaStream_t st, const SideStreams& side) {
  if (H <= 0) return CSO_OK;
  const size_t mark = ws.off;
  SsLists* lists = ws.get<SsLists>(1);
  uint32_t* list = ws.get<uint32_t>((size_t)SS_KINDS * H);
  int4* l0 = ws.get<int4>(na);
  int4* l1 = ws.get<int4>(na);
  int4* cen = ws.get<int4>(H);
  uint64_t* key = ws.get<uint64_t>(na);
  uint64_t* key2 = ws.get<uint64_t>(na);
  uint32_t* val = ws.get<uint32_t>(na);
  uint32_t* val2 = ws.get<uint32_t>(na);
  unsigned long long* dmax = ws.get<unsigned long long>(1);
  if (!lists || !list || !l0 || !l1 || !cen || !key || !key2 || !val || !val2 || !dmax) {
    cso_set_error("workspace exhausted in the radial statistics");
    return CSO_ERR_BUDGET;
  }
  // the shrinking spheres on the side streams; no return leaves one running
  struct Join {
    const SideStreams& s;
    bool on = false;
    ~Join() {
      if (on)
        for (int k = 0; k < 3; ++k) cudaStreamSynchronize(s.stream[k]);
    }
  } join{side};
  CSO_CUDA(cudaMemsetAsync(lists, 0, sizeof(SsLists), st));
  k_ss_small<<<CL(cdiv(H, 8)), 256, 0, st>>>(epos, seg, H, nuc_pos, hnuc, rows, x0, list, lists, out);
  CSO_CUDA(cudaEventRecord(side.fork, st));
  join.on = true;
  for (int k = 0; k < 3; ++k) CSO_CUDA(cudaStreamWaitEvent(side.stream[k], side.fork, 0));
  const int sms = cso_sm_count();
  const unsigned clusters = (unsigned)(sms / SS_CS > 0 ? sms / SS_CS : 1);
  if (na >= SS_BIG)
    k_ss_big<<<CL(clusters * SS_CS), 1024, 0, side.stream[0]>>>(epos, seg, nuc_pos, hnuc, rows, x0,
                                                               list + (size_t)SS_CLU * H, lists, l0, l1, out);
  if (na >= SS_LARGE)
    k_ss_block<1024, SS_LRG><<<CL(sms), 1024, 0, side.stream[1]>>>(epos, seg, nuc_pos, hnuc, rows, x0,
                                                                 list + (size_t)SS_LRG * H, lists, l0, l1, out);
  if (na >= SS_N_MIN)
    k_ss_block<256, SS_MID><<<CL(sms * 8), 256, 0, side.stream[2]>>>(epos, seg, nuc_pos, hnuc, rows, x0,
                                                                   list + (size_t)SS_MID * H, lists, l0, l1, out);
  CSO_CUDA(cudaGetLastError());
  for (int k = 0; k < 3; ++k) CSO_CUDA(cudaEventRecord(side.join[k], side.stream[k]));
  // distances to the centre, sorted by (halo, distance)
  k_radial_centre<<<CL(cdiv(H, 256)), 256, 0, st>>>(rows, H, x0, cen, out);
  CSO_CUDA(cudaMemsetAsync(dmax, 0, sizeof(unsigned long long), st));
  if (na > 0) {
    k_radial_dist<<<CL(cdiv(na, 256)), 256, 0, st>>>(epos, ehal, na, cen, key, dmax);
    CSO_CUDA(cudaMemsetAsync(val, 0, sizeof(uint32_t) * na, st));
  }
  CSO_CUDA(cudaMemcpyAsync(pinned, dmax, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
  CSO_CUDA(cudaStreamSynchronize(st));
  const unsigned long long dm = *(unsigned long long*)pinned;
  const int dbits = bit_length_u64(dm) > 0 ? bit_length_u64(dm) : 1;
  const int hbits = bit_length_u64((unsigned long long)(H - 1));
  const uint64_t* sorted = key;
  unsigned long long dmask = ~0ull;
  if (na > 0) {
    uint32_t* pv = val;
    if (dbits + hbits <= 64) {
      // one 64-bit key: halo above the distance
      k_radial_pack<<<CL(cdiv(na, 256)), 256, 0, st>>>(key, ehal, na, dbits);
      uint64_t* ph = nullptr;
      uint64_t* pl = key;
      CSO_TRY(radix_sort_128(&ph, &pl, &pv, nullptr, key2, val2, na, dbits + hbits, ws, st));
      sorted = pl;
      dmask = dbits == 64 ? ~0ull : ((1ull << dbits) - 1);
    } else {
      uint64_t* hi = ws.get<uint64_t>(na);
      uint64_t* hi2 = ws.get<uint64_t>(na);
      if (!hi || !hi2) {
        cso_set_error("workspace exhausted in the radial statistics");
        return CSO_ERR_BUDGET;
      }
      k_radial_hi<<<CL(cdiv(na, 256)), 256, 0, st>>>(hi, ehal, na);
      uint64_t* ph = hi;
      uint64_t* pl = key;
      CSO_TRY(radix_sort_128(&ph, &pl, &pv, hi2, key2, val2, na, 64 + hbits, ws, st));
      sorted = pl;
    }
  }
  if (na >= SS_BIG)
    k_radial_stats_big<<<CL(sms), 1024, 0, st>>>(sorted, dmask, seg, u, list + (size_t)SS_CLU * H, lists, out);
  k_radial_stats<<<CL(H), 256, 0, st>>>(sorted, dmask, seg, u, out);
  CSO_CUDA(cudaGetLastError());
  for (int k = 0; k < 3; ++k) CSO_CUDA(cudaStreamWaitEvent(st, side.join[k], 0));
  join.on = false;
  ws.off = mark;
  return CSO_OK;
}
