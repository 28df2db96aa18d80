// Core numbers.  Graphs of up to kLocalMaxNnz entries: kcore_local_kernel
// (below); larger ones, and small ones of few levels or of long cascades:
// a bucketed parallel peel (Section 3: K(v) is the largest k
// such that v lies in the k-core; the peel removes, level by level, every
// vertex whose remaining degree is at most k).
//
// One cooperative persistent launch processes all levels:
//   scan    every live vertex with remaining degree == k joins the level-k
//           frontier; vertices of larger degree are compacted into the next
//           live list, so later scans only touch what is left; if nothing
//           joins, k jumps to the smallest remaining degree.  A warp reads
//           kScanSlices slices of 32 live entries at once (one atomic for
//           their place in the next list).  Up to kScanLocalLive live
//           vertices, each block peels the frontier its warps found right
//           after its scan, from lists in shared memory that all its warps
//           share: rows of at most 32 edges one lane each, the 128-edge
//           chunks of rows of up to kLocalRow edges one warp each, the
//           cascade they start as further generations of the same lists, up
//           to kBlockDrainEdges edges; everything else becomes work items,
//           one per 128-edge chunk;
//   process after a grid barrier, the work items appended so far are split
//           statically over all warps (rows under 32 edges one lane per
//           item, longer chunks one warp per item, coalesced); every
//           neighbour whose degree is still above k is decremented, and one
//           whose degree falls to k joins the frontier: onto its block's
//           lists (walked by that block in the same phase) or as items of the
//           next sub-round, until a sub-round appends nothing.
// In the scan phase a vertex joins by claiming its core number
// (compare-and-swap from -1), so one that a scan reads at degree k just after
// a decrement made it k joins once; where decrements skip the read of the
// degree (degree arrays that fit in L2), a decrement from k also claims, for a
// vertex still at k that the scan has not reached.  In the sub-rounds only the
// decrement that takes a degree from k + 1 to k finds a vertex, and a plain
// store does.  The
// append order is a degeneracy order: when a vertex joins, every neighbour
// that joins later is still counted in its remaining degree, which is at most
// k.  It becomes the search's vertex ranking.
#include "mc_internal.cuh"

#include <algorithm>
#include <climits>
#include <cmath>
#include <mutex>

namespace mc {

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kChunk = 128;  // edges per work item
constexpr int kPer = 4;      // edges per lane in flight
constexpr int kLocalRow = 4096;  // rows of at most this many edges may go onto the block lists
constexpr int kPoolShort = 4096;  // block list of rows of 1..32 edges (one lane per row)
constexpr int kPoolLong = 2048;   // block list of 128-edge chunks of rows of 33..kLocalRow edges (a warp each)
constexpr long long kBlockDrainEdges = 65536;  // edges a block walks from its lists per phase (then it spills)
constexpr int64_t kScanLocalLive = (int64_t)1 << 21;  // live vertices up to which the scan peels locally
constexpr int kScanSlices = 8;  // slices of 32 live entries a warp's scan reads at once
constexpr int64_t kNoCheckMaxN = (int64_t)1 << 24;  // degree arrays up to 64 MB stay in L2: decrements unread

struct KcoreCtl {
  unsigned bar_count, bar_gen;
  int otail;          // vertices appended to the peel order
  int live_n[2];      // live-list sizes (ping-pong)
  int pad;
  long long wtail;    // work items appended
  int minrem[3];      // smallest remaining degree, rotated per level scan
  long long snap[2][3];  // (otail, wtail, live) captured by the last block into each barrier
};

__device__ __forceinline__ long long ld_vol64(const long long *p) { return *(const volatile long long *)p; }

// Grid barrier number gen + 1 (every block counts them) that also snapshots
// (otail, wtail) when every block has arrived.  Bounded spin: on timeout the
// error word is set.
__device__ __forceinline__ void barrier_snap(KcoreCtl *ctl, unsigned nblocks, unsigned &gen, int32_t *err,
                                             long long spin_limit, long long *otail_out, long long *wtail_out,
                                             const int *live_src, long long *live_out) {
  __shared__ long long s_o, s_w, s_l;
  __syncthreads();
  gen++;
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&ctl->bar_count, 1u) == nblocks - 1) {
      __threadfence();
      ctl->snap[gen & 1][0] = *(volatile int *)&ctl->otail;
      ctl->snap[gen & 1][1] = ld_vol64(&ctl->wtail);
      ctl->snap[gen & 1][2] = live_src ? *(volatile const int *)live_src : 0;
      *(volatile unsigned *)&ctl->bar_count = 0;
      __threadfence();
      *(volatile unsigned *)&ctl->bar_gen = gen;
    } else {
      long long it = 0;
      while (*(volatile unsigned *)&ctl->bar_gen != gen) {
        if (++it > spin_limit) { atomicExch(err, kDevTimeout); break; }
        __nanosleep(16);
      }
    }
    __threadfence();
    s_o = ld_vol64(&ctl->snap[gen & 1][0]);
    s_w = ld_vol64(&ctl->snap[gen & 1][1]);
    s_l = ld_vol64(&ctl->snap[gen & 1][2]);
  }
  __syncthreads();
  *otail_out = s_o;
  *wtail_out = s_w;
  if (live_out) *live_out = s_l;
}

__global__ void degree_init_kernel(int64_t n, const int64_t *__restrict__ rp, int32_t *__restrict__ deg,
                                   int32_t *__restrict__ core, int32_t *__restrict__ maxdeg, const int32_t *skip) {
  if (skip && *skip) return;
  int local = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    int d = (int)(rp[v + 1] - rp[v]);
    deg[v] = d;
    core[v] = -1;  // not yet in the peel order
    local = max(local, d);
  }
  local = dev::warp_max(local);
  if ((threadIdx.x & 31) == 0) atomicMax(maxdeg, local);
}

// The rows a block peels within one phase: two generations of two lists
// (rows of 1..32 edges, walked one lane per row; the 128-edge chunks of rows
// of 33..kLocalRow edges, encoded like work items and walked by one warp
// each).  The new frontier found while one generation is walked goes to the
// other, so the block's 32 warps share its cascade.  A counter may run past
// its list's capacity: the entries beyond it were not stored (those rows or
// chunks became work items instead).
struct BlockPool {
  int s[2][kPoolShort];
  long long l[2][kPoolLong];
  int ns[2], nl[2];
  long long edges;  // edges walked from the lists in this phase
  int fscan[kWarps][32 * kScanSlices];  // a warp's scanned frontier, compacted
};

// Append the lanes' new frontier vertices (flag nf, vertex u): core and
// peel order; then their rows' work.  With a block pool (bp, generation
// gen), rows of 1..kLocalRow edges go onto its lists while there is room,
// to be walked by this block in the same phase; the others become one work
// item per chunk of their row, walked in the next sub-round.  All lanes
// call.
template <bool CLAIM>
__device__ __forceinline__ void append_frontier(bool nf, int u, int k, const int64_t *__restrict__ rp, int32_t *core,
                                                int32_t *order, long long *wq, KcoreCtl *ctl,
                                                BlockPool *bp = nullptr, int gen = 0) {
  const int lane = threadIdx.x & 31;
  if (!__any_sync(0xffffffffu, nf)) return;
  // claim: a vertex found by a scan and by a decrement in the same phase
  // joins once; after the scan only decrements find vertices, each exactly
  // once (the one that takes its degree from k + 1 to k), so a store does
  if (CLAIM) {
    if (nf) nf = atomicCAS(core + u, -1, k) == -1;
  } else if (nf) {
    core[u] = k;
  }
  const unsigned m = __ballot_sync(0xffffffffu, nf);
  if (!m) return;
  const unsigned lt = (1u << lane) - 1u;
  int64_t d = 0;
  if (nf) d = rp[u + 1] - rp[u];
  // chunks [c0, c0 + nch) of the lane's row become work items
  int c0 = 0, nch = (nf && d > 0) ? (int)((d + kChunk - 1) / kChunk) : 0;
  if (bp) {
    const bool sh = nf && d > 0 && d <= 32;
    const bool lg = nf && d > 32 && d <= kLocalRow;
    const unsigned ms = __ballot_sync(0xffffffffu, sh);
    int lincl = lg ? nch : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, lincl, o);
      if (lane >= o) lincl += y;
    }
    const int ltot = __shfl_sync(0xffffffffu, lincl, 31);
    int bs = 0, bl = 0;
    if (lane == 0) {
      if (ms) bs = atomicAdd(&bp->ns[gen], __popc(ms));
      if (ltot) bl = atomicAdd(&bp->nl[gen], ltot);
    }
    bs = __shfl_sync(0xffffffffu, bs, 0);
    bl = __shfl_sync(0xffffffffu, bl, 0);
    if (sh) {
      const int at = bs + __popc(ms & lt);
      if (at < kPoolShort) {
        bp->s[gen][at] = u;
        nch = 0;
      }
    }
    if (lg) {
      // the chunks that fit go onto the list, the rest become work items
      const int at = bl + lincl - nch;
      const int fit = max(0, min(nch, kPoolLong - at));
      for (int c = 0; c < fit; c++) bp->l[gen][at + c] = ((long long)u << 32) | (unsigned)c;
      c0 = fit;
      nch -= fit;
    }
  }
  int incl = nch;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int tot = __shfl_sync(0xffffffffu, incl, 31);
  int ob = 0;
  long long wb = 0;
  if (lane == 0) {
    ob = atomicAdd(&ctl->otail, __popc(m));
    if (tot) wb = (long long)atomicAdd((unsigned long long *)&ctl->wtail, (unsigned long long)tot);
  }
  ob = __shfl_sync(0xffffffffu, ob, 0);
  wb = __shfl_sync(0xffffffffu, wb, 0);
  if (nf) {
    order[ob + __popc(m & lt)] = u;
    long long at = wb + incl - nch;
    for (int c = 0; c < nch; c++) wq[at + c] = ((long long)u << 32) | (unsigned)(c0 + c);
  }
  __syncwarp();
}

// One work item per lane that has one (a chunk entry of a block list).
__device__ __forceinline__ void push_entry(bool has, long long e, long long *wq, KcoreCtl *ctl) {
  const int lane = threadIdx.x & 31;
  const unsigned m = __ballot_sync(0xffffffffu, has);
  if (!m) return;
  long long wb = 0;
  if (lane == 0) wb = (long long)atomicAdd((unsigned long long *)&ctl->wtail, (unsigned long long)__popc(m));
  wb = __shfl_sync(0xffffffffu, wb, 0);
  if (has) wq[wb + __popc(m & ((1u << lane) - 1u))] = e;
}

// Work items (one per chunk) for lanes' vertices already in the peel order:
// what is left on a block's lists at the end of its budget.
__device__ __forceinline__ void push_items(bool has, int u, const int64_t *__restrict__ rp, long long *wq,
                                           KcoreCtl *ctl) {
  const int lane = threadIdx.x & 31;
  const int nch = has ? (int)((rp[u + 1] - rp[u] + kChunk - 1) / kChunk) : 0;
  int incl = nch;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int tot = __shfl_sync(0xffffffffu, incl, 31);
  if (!tot) return;
  long long wb = 0;
  if (lane == 0) wb = (long long)atomicAdd((unsigned long long *)&ctl->wtail, (unsigned long long)tot);
  wb = __shfl_sync(0xffffffffu, wb, 0);
  long long at = wb + incl - nch;
  for (int c = 0; c < nch; c++) wq[at + c] = ((long long)u << 32) | (unsigned)c;
}

// One decrement of neighbour u at level k; true when u joins the level-k
// frontier through it.  With chk the degree is read first and only a degree
// above k is decremented, so the decrement that takes it from k + 1 to k is
// the one that finds u.  Without chk the read is skipped: a peeled
// neighbour's degree (at most k, no longer read) just goes lower.  In the
// sub-rounds every vertex at degree k or below is already peeled, so again
// only k + 1 -> k finds one; while a scan may still read the degrees
// (CLAIM), a vertex still at exactly k may not have been reached by it yet,
// so the decrement from k claims it too (the claim's compare-and-swap keeps
// each vertex to one join).
template <bool CLAIM>
__device__ __forceinline__ bool decrement(int32_t *deg, int u, int k, bool chk) {
  if (u < 0) return false;
  if (chk && __ldcg(deg + u) <= k) return false;
  const int old = atomicSub(deg + u, 1);
  return old == k + 1 || (CLAIM && !chk && old == k);
}

// Walk one row (b0, len) with the whole warp (coalesced), kPer edges per
// lane in flight before the frontier appends.
template <bool CLAIM>
__device__ __forceinline__ void walk_row(int64_t b0, int len, int k, bool chk, const int64_t *__restrict__ rp,
                                         const int32_t *__restrict__ ci, int32_t *deg, int32_t *core, int32_t *order,
                                         long long *wq, KcoreCtl *ctl, BlockPool *bp, int gen) {
  const int lane = threadIdx.x & 31;
  for (int eb = 0; eb < len; eb += 32 * kPer) {
    int u[kPer];
    bool nf[kPer];
#pragma unroll
    for (int q = 0; q < kPer; q++) {
      const int e = eb + q * 32 + lane;
      u[q] = e < len ? ci[b0 + e] : -1;
    }
#pragma unroll
    for (int q = 0; q < kPer; q++) nf[q] = decrement<CLAIM>(deg, u[q], k, chk);
#pragma unroll
    for (int q = 0; q < kPer; q++) append_frontier<CLAIM>(nf[q], u[q], k, rp, core, order, wq, ctl, bp, gen);
  }
}

// Walk rows of at most 32 edges, one lane per row (b0, len; len 0 for idle
// lanes), decrementing every neighbour whose degree is still above k; new
// frontier vertices are appended (to the block's lists when given).
template <bool CLAIM>
__device__ __forceinline__ void walk_short_rows(int64_t b0, int len, int k, bool chk, const int64_t *__restrict__ rp,
                                                const int32_t *__restrict__ ci, int32_t *deg, int32_t *core,
                                                int32_t *order, long long *wq, KcoreCtl *ctl, BlockPool *bp,
                                                int gen) {
  const int maxlen = dev::warp_max(len);
  for (int j0 = 0; j0 < maxlen; j0 += kPer) {
    int u[kPer];
    bool nf[kPer];
#pragma unroll
    for (int q = 0; q < kPer; q++) u[q] = (j0 + q < len) ? ci[b0 + j0 + q] : -1;
#pragma unroll
    for (int q = 0; q < kPer; q++) nf[q] = decrement<CLAIM>(deg, u[q], k, chk);
#pragma unroll
    for (int q = 0; q < kPer; q++) append_frontier<CLAIM>(nf[q], u[q], k, rp, core, order, wq, ctl, bp, gen);
  }
}

// The block's own cascade: the rows on its lists of generation gen, walked
// by all its warps (short rows 32 to a warp, one lane each; chunks of long
// rows one warp each), the new frontier going to the other generation, until the
// lists are empty or kBlockDrainEdges edges were walked; what is left
// becomes work items of the next sub-round.  Every thread of the block
// calls; the lists are empty on return.
template <bool CLAIM>
__device__ void block_drain(int k, bool chk, const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
                            int32_t *deg, int32_t *core, int32_t *order, long long *wq, KcoreCtl *ctl, BlockPool *bp,
                            int gen) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  for (;;) {
    __syncthreads();  // the generation's rows are in place, its edges counted
    const int ns = min(bp->ns[gen], kPoolShort), nl = min(bp->nl[gen], kPoolLong);
    const long long walked = bp->edges;
    __syncthreads();  // every thread has read the counters before they change
    if (ns + nl == 0) break;
    if (walked >= kBlockDrainEdges) {
      for (int j0 = wib * 32; j0 < ns; j0 += kThreads) {
        const int j = j0 + lane;
        push_items(j < ns, j < ns ? bp->s[gen][j] : 0, rp, wq, ctl);
      }
      for (int j0 = wib * 32; j0 < nl; j0 += kThreads) {
        const int j = j0 + lane;
        push_entry(j < nl, j < nl ? bp->l[gen][j] : 0, wq, ctl);
      }
      break;
    }
    if (threadIdx.x == 0) {
      bp->ns[gen ^ 1] = 0;
      bp->nl[gen ^ 1] = 0;
    }
    __syncthreads();
    int mine = 0;
    for (int j0 = wib * 32; j0 < ns; j0 += kThreads) {
      const int j = j0 + lane;
      const int u = j < ns ? bp->s[gen][j] : -1;
      const int64_t b0 = u >= 0 ? rp[u] : 0;
      const int len = u >= 0 ? (int)(rp[u + 1] - b0) : 0;
      mine += len;
      walk_short_rows<CLAIM>(b0, len, k, chk, rp, ci, deg, core, order, wq, ctl, bp, gen ^ 1);
    }
    for (int j = wib; j < nl; j += kWarps) {
      const long long e = bp->l[gen][j];
      const int u = (int)(e >> 32), c = (int)(e & 0xffffffff);
      const int64_t b0 = rp[u] + (int64_t)c * kChunk;
      const int len = (int)(min(rp[u + 1], b0 + kChunk) - b0);
      if (lane == 0) mine += len;
      walk_row<CLAIM>(b0, len, k, chk, rp, ci, deg, core, order, wq, ctl, bp, gen ^ 1);
    }
    mine = dev::warp_sum(mine);
    if (lane == 0 && mine) atomicAdd((unsigned long long *)&bp->edges, (unsigned long long)mine);
    gen ^= 1;
  }
  if (threadIdx.x == 0) {
    bp->ns[0] = bp->ns[1] = 0;
    bp->nl[0] = bp->nl[1] = 0;
    bp->edges = 0;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kThreads, 1) kcore_peel_kernel(int64_t n, const int64_t *__restrict__ rp,
                                                                 const int32_t *__restrict__ ci, int32_t *deg,
                                                                 int32_t *core, int32_t *order, int32_t *live0,
                                                                 int32_t *live1, long long *wq, KcoreCtl *ctl,
                                                                 int32_t *err, long long spin_limit, int nocheck,
                                                                 const int32_t *skip) {
  if (skip && *skip) return;  // the order is made already
  unsigned gen = 0;           // grid barriers passed
  __shared__ int bmin;
  extern __shared__ __align__(16) unsigned char s_pool[];
  BlockPool *bp = (BlockPool *)s_pool;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t gwarp = (int64_t)blockIdx.x * kWarps + wib;
  const int64_t nwarps = (int64_t)gridDim.x * kWarps;
  const unsigned nblocks = gridDim.x;
  const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
  const unsigned lt = (1u << lane) - 1u;
  const bool chk = nocheck == 0;
  if (threadIdx.x == 0) {
    bp->ns[0] = bp->ns[1] = 0;
    bp->nl[0] = bp->nl[1] = 0;
    bp->edges = 0;
  }

  int k = 0;
  unsigned level = 0;
  long long otail_now = 0, otail_prev = 0, wtail_now = 0, wstart = 0;
  int64_t live_count = n;  // level 0 scans every vertex (identity list)
  int32_t *lin = live0, *lout = live1;

  for (;;) {
    // ---------------- scan: frontier of level k, compaction of the rest ----
    if (threadIdx.x == 0) bmin = INT_MAX;
    if (leader) {
      ctl->minrem[(level + 1) % 3] = INT_MAX;
      ctl->live_n[(level + 1) & 1] = 0;
    }
    __syncthreads();
    int lmin = INT_MAX;
    int *lout_n = &ctl->live_n[level & 1];
    const bool scan_local = live_count <= kScanLocalLive;  // the same in every block
    // groups of kScanSlices slices of 32 live entries go round-robin over the
    // blocks first, so a run of frontier vertices in the list is spread over
    // many blocks; a warp reads a group's entries and degrees at once, takes
    // its place in the next live list with one atomic, and appends the
    // group's frontier 32 vertices at a time
    int *fw = bp->fscan[wib];
    constexpr int kGroup = 32 * kScanSlices;
    for (int64_t sg = blockIdx.x + (int64_t)nblocks * wib; sg * kGroup < live_count; sg += nwarps) {
      int v[kScanSlices], d[kScanSlices];
#pragma unroll
      for (int q = 0; q < kScanSlices; q++) {
        const int64_t i = sg * kGroup + q * 32 + lane;
        v[q] = -1;
        if (i < live_count) v[q] = (level == 0) ? (int)i : lin[i];
      }
#pragma unroll
      for (int q = 0; q < kScanSlices; q++) d[q] = v[q] >= 0 ? __ldcg(deg + v[q]) : INT_MIN;
      int ktot = 0;
#pragma unroll
      for (int q = 0; q < kScanSlices; q++) {
        if (d[q] > k) lmin = min(lmin, d[q]);
        ktot += __popc(__ballot_sync(0xffffffffu, d[q] > k));
      }
      int ob = 0;
      if (lane == 0 && ktot) ob = atomicAdd(lout_n, ktot);
      ob = __shfl_sync(0xffffffffu, ob, 0);
      int ftot = 0;
#pragma unroll
      for (int q = 0; q < kScanSlices; q++) {
        const unsigned km = __ballot_sync(0xffffffffu, d[q] > k);
        if (d[q] > k) lout[ob + __popc(km & lt)] = v[q];
        ob += __popc(km);
        const unsigned fm = __ballot_sync(0xffffffffu, d[q] == k);
        if (d[q] == k) fw[ftot + __popc(fm & lt)] = v[q];
        ftot += __popc(fm);
      }
      __syncwarp();
      for (int f0 = 0; f0 < ftot; f0 += 32) {
        const bool has = f0 + lane < ftot;
        const int u = has ? fw[f0 + lane] : -1;
        if (scan_local)
          append_frontier<true>(has, u, k, rp, core, order, wq, ctl, bp, 0);
        else
          append_frontier<false>(has, u, k, rp, core, order, wq, ctl);
      }
      __syncwarp();
    }
    // the frontier a block found (up to its lists) is peeled at once by that
    // block, while others may still be scanning: a vertex they read at
    // degree k after a decrement here is claimed once; one kept at k + 1 and
    // then peeled here is dropped by the next scan, its degree being <= k.
    // Above kScanLocalLive live vertices the frontier is large enough to
    // keep every warp busy in the sub-rounds: the scan only lists it (no
    // decrement runs during the scan, so each vertex joins once without a
    // claim)
    if (scan_local) block_drain<true>(k, chk, rp, ci, deg, core, order, wq, ctl, bp, 0);
    lmin = -dev::warp_max(-lmin);
    if (lane == 0 && lmin != INT_MAX) atomicMin(&bmin, lmin);
    __syncthreads();
    if (threadIdx.x == 0 && bmin != INT_MAX) atomicMin(&ctl->minrem[level % 3], bmin);
    long long live_next = 0;
    barrier_snap(ctl, nblocks, gen, err, spin_limit, &otail_now, &wtail_now, lout_n, &live_next);
    if (*(volatile int32_t *)err) return;
    live_count = live_next;
    { int32_t *t = lin; lin = lout; lout = t; }

    if (otail_now >= n) break;
    if (otail_now == otail_prev) {
      // nothing at level k: no decrement happened, so the smallest kept
      // degree is exact
      int mk = *(volatile int *)&ctl->minrem[level % 3];
      level++;
      if (mk == INT_MAX) break;  // unreachable while vertices remain
      k = mk;
      continue;
    }

    // ---------------- process: sub-rounds over fixed item ranges ----------
    // Items [s0, e0) were appended before the last barrier; those appended
    // while processing them form the next sub-round.  Warps take groups of
    // 32 items statically: rows shorter than 32 edges are walked one lane per
    // item (lanes in step, so appends stay warp-aggregated), longer chunks by
    // the whole warp.  The frontier they find goes to the block's lists.
    long long s0 = wstart, e0 = wtail_now;
    while (s0 < e0) {
      // pass A: items of fewer than 32 edges, 32 per warp, one lane each
      for (long long gb = s0 + gwarp * 32; gb < e0; gb += nwarps * 32) {
        const long long t = gb + lane;
        const bool valid = t < e0;
        const long long item = valid ? __ldcg(wq + t) : -1LL;
        int64_t b0 = 0;
        int len = 0;
        if (valid) {
          const int v = (int)(item >> 32), c = (int)(item & 0xffffffff);
          b0 = rp[v] + (int64_t)c * kChunk;
          len = (int)(min(rp[v + 1], b0 + kChunk) - b0);
        }
        walk_short_rows<false>(b0, (valid && len < 32) ? len : 0, k, chk, rp, ci, deg, core, order, wq, ctl, bp,
                               0);
      }
      // pass B: longer chunks, one warp each (coalesced row reads)
      for (long long t = s0 + gwarp; t < e0; t += nwarps) {
        const long long item = __ldcg(wq + t);
        const int v = (int)(item >> 32), c = (int)(item & 0xffffffff);
        const int64_t b0 = rp[v] + (int64_t)c * kChunk;
        const int len = (int)(min(rp[v + 1], b0 + kChunk) - b0);
        if (len < 32) continue;
        walk_row<false>(b0, len, k, chk, rp, ci, deg, core, order, wq, ctl, bp, 0);
      }
      block_drain<false>(k, chk, rp, ci, deg, core, order, wq, ctl, bp, 0);
      long long e1 = 0;
      barrier_snap(ctl, nblocks, gen, err, spin_limit, &otail_now, &e1, nullptr, nullptr);
      if (*(volatile int32_t *)err) return;
      s0 = e0;
      e0 = e1;
      wtail_now = e1;
    }
    wstart = wtail_now;
    otail_prev = otail_now;
    level++;
    if (otail_now >= n) break;
    k++;
  }
}

// A peel that stopped early (its spin limit ran out) leaves the tail of the
// order unwritten: such entries are skipped and reported, never used as an
// index.
__global__ void peel_pos_kernel(int64_t n, const int32_t *__restrict__ order, int32_t *__restrict__ pos,
                                const int32_t *__restrict__ core, int32_t *__restrict__ maxcore, int32_t *err,
                                const int32_t *skip) {
  if (skip && *skip) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int v = order[i];
    if (v < 0 || (int64_t)v >= n) {
      atomicCAS(err, kDevOk, kDevCheck);
      continue;
    }
    pos[v] = (int32_t)i;
    if (i == n - 1) *maxcore = core[v];  // the peel order is nondecreasing in K
  }
}

// ------------------------------------------------------------------------
// Core numbers by local updates, then the order shell by shell.
//
// The level-by-level peel of a graph of many levels is bound by latency: a
// level costs a grid barrier and a chain of dependent steps per generation of
// its cascade, and graphs have hundreds of levels (258 at R-MAT scale 22).
// This kernel runs all levels at once, in two parts (the H-index operator
// converges to the core numbers: Lue, Zhou, Zhang and Stanley 2016; as a
// distributed algorithm: Montresor, De Pellegrini and Miorandi 2013):
//   values  every vertex holds an upper bound h of its core number, at first
//           min(degree, sqrt(entries)); a vertex whose support (neighbours
//           with a bound of at least h) may have fallen below h takes the
//           largest k with at least k neighbours of bound >= k.  A step
//           evaluates the listed vertices, and after a barrier the lowered
//           ones list the neighbours they no longer support.  8 to 70 steps.
//   order   with K known, the shells are peeled side by side: a vertex leaves
//           in the first round in which at most K(v) of its neighbours of core
//           number >= K(v) have not left in an earlier round; positions go by
//           shell, then by round.  Each vertex has at most K(v) neighbours
//           after it, so this is a degeneracy order.  7 to 68 rounds.
// Rows of at most 32 entries are read by a warp four at a time, rows of up to
// kLocalWarpRow by a warp, longer ones by a block; a new value is found in
// one pass over the row from a histogram of the values just below h.  A step
// of few vertices takes 4-12 us (two barriers and six dependent L2 accesses);
// in all the rows are read about 17 times.  Graphs that need more than
// kLocalSteps steps or rounds (long paths) are left to the peel.
//
// The peel / this kernel: Chung-Lu 20,000 vertices 1.42 / 0.46 ms, R-MAT scale
// 15 2.1 / 0.58, scale 18 (edge factor 12) 3.5 / 1.5, scale 20 5.7 / 5.0,
// Chung-Lu 1,000,003 vertices (35 M entries, K(G) = 438) 14.8 / 4.3.  Barriers
// that count arrivals over the launch took another 4 .. 10% off (calls of the
// first three and the last: 0.58 -> 0.55, 0.67 -> 0.63, 2.01 -> 1.92, 5.1 -> 4.6
// ms).  Above kLocalMaxNnz the repeated reads cost more than the peel's barriers,
// and so they do below it where the levels are few for the rows (local_pays).
// ------------------------------------------------------------------------

constexpr int64_t kLocalMaxNnz = 40000000;
// Steps (rounds) after which the graph is left to the peel.  R-MAT, Chung-Lu and
// G(n, p) graphs of 10^3 .. 2 x 10^6 vertices need 8 to 70; what a graph with a long
// cascade besides (a path of thousands at R-MAT scale 15: 5.7 ms by the peel
// alone) pays on top is 128 steps of 9 us, 2.4 ms with 256 of them.
constexpr int kLocalSteps = 128;
constexpr int kLocalWarpRow = 2048;
constexpr int kLocalBins = 256;                 // per warp; a block uses all its warps' bins
constexpr int kLocalBlockBins = kLocalBins * kWarps;
constexpr int kStage = 64;                      // listed vertices a warp holds back to append 32 at a time

struct LocalCtl {
  unsigned bar_count;
  int pad[31];
  int n[3][32];   // [counter set][class 0..2]: listed vertices
  int all[32];    // [0..1] vertices of class 1, 2; [2] vertices placed; [3] largest core number
  int hist[256];  // vertices by degree (degree_bin)
};

// Degrees in bins: one each below 32, then eight per power of two.
__device__ __forceinline__ int degree_bin(int d) {
  const int e = 31 - __clz(d | 1);
  return d < 32 ? d : 32 + (e - 5) * 8 + ((d >> (e - 3)) & 7);
}
__device__ __forceinline__ int bin_degree(int b) {  // the bin's smallest degree
  return b < 32 ? b : (8 + ((b - 32) & 7)) << (2 + ((b - 32) >> 3));
}

// Whether this kernel beats the peel, from the degrees alone.  The peel pays per
// level, of which there are at most H - L: no core number is above the largest H
// with H vertices of degree >= H, and few are below L, the degree that 1/64 of
// the vertices do not reach.  This kernel pays per row entry, about 17 reads
// each.  Up to 4.5 M entries the reads are in L2 and 16 levels are enough; above,
// the line of equal times is at 28 levels per million entries.  This kernel /
// the peel, in ms with loading (0.5): H - L = 15, 4.0 M entries 1.39 / 0.81;
// 16, 0.1 M 0.80 / 0.86; 29, 0.9 M 1.53 / 2.47; 35, 4.0 M 2.20 / 2.65; 19, 8.0 M
// 2.00 / 1.00; 52, 10 M 1.80 / 1.19; 251, 6.0 M 3.04 / 2.97; 333, 12 M 4.10 / 3.43;
// 596, 20 M 3.95 / 4.85; 650, 30 M 8.39 / 6.73; 1,058, 32 M 4.71 / 6.61; 1,386, 31
// M 5.75 / 6.27.  Grids, paths, trees and stars have H - L of 0 to 8: 2.5 / 1.1 (a
// 100 x 100 grid), 25.6 / 9.0 (a star of 10^7).  Dense graphs of nearly one degree
// and no hubs are decided in a step or two here (K(300, 5000) 0.65 / 0.78).
__device__ __forceinline__ bool local_pays(int high, int low, int maxdeg, int64_t nnz) {
  const int levels = high - low;
  if (levels < 16) return low >= 64 && nnz < 8000000 && maxdeg <= 8192;
  return nnz < 4500000 || levels * (int64_t)1000000 >= 28 * nnz;
}

struct LocalArgs {
  int64_t n, nnz;
  int cap;  // sqrt(entries)
  const int64_t *rp;
  const int32_t *ci;
  int32_t *h, *old, *stamp;  // h becomes the core numbers; old: the value before the last evaluation, then the support counts
  int32_t *order, *pos;
  int32_t *list[2][3], *all[2];  // listed vertices by row class; all vertices of classes 1 and 2
  int32_t *start, *taken;        // per core number: first position, positions taken
  LocalCtl *ctl;
  int32_t *maxdeg, *maxcore, *done;
  int32_t *err;
  long long spin;
};

struct LocalShared {
  int bins[kLocalBlockBins];
  int stage[kWarps][kStage];
  int cnt[3], err;
  int red[4];
  unsigned barriers;  // thread 0's
};

__device__ __forceinline__ int row_class(int64_t len) { return len <= 32 ? 0 : (len <= kLocalWarpRow ? 1 : 2); }

// Short rows a warp takes at a time (four are read at once): as few as keep
// every warp busy.
__device__ __forceinline__ int short_batch(int64_t n0, int64_t nwarps) {
  return (int)min((int64_t)32, max((int64_t)4, (n0 / nwarps + 4) & ~(int64_t)3));
}

// Grid barrier; afterwards S.cnt holds the three list lengths of `src`.
// False: the error word is set.
__device__ bool local_barrier(const LocalArgs &a, LocalShared &S, const int *src) {
  __syncthreads();
  if (threadIdx.x == 0) {
    // arrivals are counted over the whole launch: the count itself says when
    // all have reached this barrier, nothing is reset and no second word read
    const unsigned all = (S.barriers += 1) * gridDim.x;
    __threadfence();
    if (atomicAdd(&a.ctl->bar_count, 1u) + 1 < all) {
      long long it = 0;
      while ((int)(*(volatile unsigned *)&a.ctl->bar_count - all) < 0) {
        if (++it > a.spin) {
          atomicExch(a.err, kDevTimeout);
          break;
        }
        __nanosleep(16);
      }
    }
    __threadfence();
    if (src) {
      S.cnt[0] = __ldcg(src);
      S.cnt[1] = __ldcg(src + 1);
      S.cnt[2] = __ldcg(src + 2);
    }
    S.err = *(volatile int32_t *)a.err;
  }
  __syncthreads();
  return S.err == 0;
}

// Append the lanes' vertices (has, u) to the lists of buffer b (counter set t)
// by row class; with PLACE they also take their positions in the order.  All
// lanes.
template <bool PLACE>
__device__ __forceinline__ void local_append(const LocalArgs &a, bool has, int u, int b, int t) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int c = has ? row_class(a.rp[u + 1] - a.rp[u]) : -1;
  unsigned m[3];
#pragma unroll
  for (int q = 0; q < 3; q++) m[q] = __ballot_sync(0xffffffffu, c == q);
  int at = 0;
  if (lane < 3) {  // the three classes' places at once
    const int k = __popc(lane == 0 ? m[0] : lane == 1 ? m[1] : m[2]);
    if (k) at = atomicAdd(&a.ctl->n[t][lane], k);
  }
#pragma unroll
  for (int q = 0; q < 3; q++) {
    const int base = __shfl_sync(0xffffffffu, at, q);
    if (c == q) a.list[b][q][base + __popc(m[q] & lt)] = u;
  }
  if (PLACE) {
    const int k = has ? a.h[u] : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, k);
    const int first = __ffs(peers) - 1;
    int to = 0;
    if (has && lane == first) to = a.start[k] + atomicAdd(a.taken + k, __popc(peers));
    to = __shfl_sync(0xffffffffu, to, first);
    if (has) {
      const int p = to + __popc(peers & lt);
      a.order[p] = u;
      a.pos[u] = p;
    }
    const unsigned any = __ballot_sync(0xffffffffu, has);
    if (lane == 0 && any) atomicAdd(&a.ctl->all[2], __popc(any));
  }
}

// Hold the lanes' vertices back until there are 32 to append.
template <bool PLACE>
__device__ __forceinline__ void local_stage(const LocalArgs &a, int *buf, int &held, bool has, int u, int b, int t) {
  const int lane = threadIdx.x & 31;
  const unsigned m = __ballot_sync(0xffffffffu, has);
  if (!m) return;
  if (has) buf[held + __popc(m & ((1u << lane) - 1u))] = u;
  held += __popc(m);
  __syncwarp();
  if (held >= 32) {
    local_append<PLACE>(a, true, buf[lane], b, t);
    held -= 32;
    const int x = lane < held ? buf[32 + lane] : 0;
    __syncwarp();
    if (lane < held) buf[lane] = x;
    __syncwarp();
  }
}
template <bool PLACE>
__device__ __forceinline__ void local_stage_end(const LocalArgs &a, int *buf, int &held, int b, int t) {
  const int lane = threadIdx.x & 31;
  if (held) local_append<PLACE>(a, lane < held, lane < held ? buf[lane] : 0, b, t);
  held = 0;
  __syncwarp();
}

// Smallest i in [0, bins) with c + bin[0] + .. + bin[i] >= h - 1 - i (the new
// value is h - 1 - i); -1 if none.  A warp, 32 bins
// at a time: values seldom fall far, so the first group mostly has it.
__device__ __forceinline__ int window_find(const int *bin, int bins, int h, int c) {
  const int lane = threadIdx.x & 31;
  for (int g = 0; g < bins; g += 32) {
    int incl = bin[g + lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, c + incl >= h - 1 - (g + lane));
    if (hit) return g + __ffs(hit) - 1;
    c += __shfl_sync(0xffffffffu, incl, 31);
  }
  return -1;
}

// New value of a row of 33..kLocalWarpRow entries whose vertex holds h.  The
// values may fall while they are read: a pass counts every entry once (at or
// above the window, or in it), so a value that is too high counts on a
// neighbour that falls below it in this step and will list the vertex again.
__device__ __forceinline__ int eval_warp(const LocalArgs &a, int64_t e0, int len, int h, int *bin) {
  const int lane = threadIdx.x & 31;
  int top = h;  // window: values top - 1 .. top - kLocalBins
  for (;;) {
    __syncwarp();
    for (int i = lane; i < kLocalBins; i += 32) bin[i] = 0;
    __syncwarp();
    int mine = 0;
    for (int b = 0; b < len; b += 32 * 8) {
      int x[8];
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int e = b + 32 * q + lane;
        x[q] = e < len ? a.ci[e0 + e] : -1;
      }
#pragma unroll
      for (int q = 0; q < 8; q++) x[q] = x[q] >= 0 ? a.h[x[q]] : INT_MIN;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        if (x[q] >= top) mine++;
        else if (x[q] >= top - kLocalBins) atomicAdd(&bin[top - 1 - x[q]], 1);
      }
    }
    __syncwarp();
    const int c = dev::warp_sum(mine);
    if (top == h && c >= h) return h;
    const int i = window_find(bin, kLocalBins, top, c);
    if (i >= 0) return top - 1 - i;
    top -= kLocalBins;
  }
}

// The same by a block (all threads), for longer rows.
__device__ int eval_block(const LocalArgs &a, LocalShared &S, int64_t e0, int64_t len, int h) {
  const int lane = threadIdx.x & 31;
  int top = h;
  for (;;) {
    __syncthreads();
    for (int i = threadIdx.x; i < kLocalBlockBins; i += kThreads) S.bins[i] = 0;
    if (threadIdx.x == 0) S.red[0] = 0;
    __syncthreads();
    int mine = 0;
    for (int64_t b = 0; b < len; b += kThreads * 8) {
      int x[8];
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int64_t e = b + kThreads * q + threadIdx.x;
        x[q] = e < len ? a.ci[e0 + e] : -1;
      }
#pragma unroll
      for (int q = 0; q < 8; q++) x[q] = x[q] >= 0 ? a.h[x[q]] : INT_MIN;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        if (x[q] >= top) mine++;
        else if (x[q] >= top - kLocalBlockBins) atomicAdd(&S.bins[top - 1 - x[q]], 1);
      }
    }
    mine = dev::warp_sum(mine);
    if (lane == 0 && mine) atomicAdd(&S.red[0], mine);
    __syncthreads();
    const int c = S.red[0];
    if (top == h && c >= h) return h;
    if (threadIdx.x < 32) {
      const int i = window_find(S.bins, kLocalBlockBins, top, c);
      if (lane == 0) S.red[1] = i;
    }
    __syncthreads();
    if (S.red[1] >= 0) return top - 1 - S.red[1];
    top -= kLocalBlockBins;
  }
}

// Neighbour u of a vertex whose value fell from `was` to `now`: true when u
// counted on it and has to be evaluated (once per step: stamp).
__device__ __forceinline__ bool lost_support(const LocalArgs &a, int u, int now, int was, int step) {
  if (u < 0) return false;
  const int x = a.h[u];
  if (x <= now || x > was) return false;
  if (__ldcg(a.stamp + u) == step) return false;
  return atomicExch(a.stamp + u, step) != step;
}

// Neighbour u of a vertex of core number k that left: true when u leaves in
// the next round through it.
__device__ __forceinline__ bool leaves_next(const LocalArgs &a, int u, int k) {
  if (u < 0 || a.h[u] != k) return false;
  if (__ldcg(a.old + u) <= k) return false;
  return atomicSub(a.old + u, 1) == k + 1;
}

// The rows of the listed vertices, every neighbour tested; those that pass go
// to the lists of buffer b.  Values (ORDER false): of the vertices whose value
// fell in this step; order: of all.  When few rows are listed, a row is split
// over several warps (blocks).
template <bool ORDER>
__device__ __forceinline__ void local_walk(const LocalArgs &a, const int32_t *l0, const int32_t *l1, const int32_t *l2,
                                           int64_t n0, int64_t n1, int64_t n2, int step, int *buf, int b, int t) {
  const int lane = threadIdx.x & 31;
  const int64_t gwarp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int64_t nwarps = (int64_t)gridDim.x * kWarps;
  int held = 0;
  auto test = [&](int u, int p, int was) { return ORDER ? leaves_next(a, u, p) : lost_support(a, u, p, was, step); };
  auto row = [&](int64_t e0, int64_t e1, int at, int stride, int p, int was) {
    for (int64_t c = e0; c < e1; c += 8 * (int64_t)stride) {
      int u[8];
      unsigned hit = 0;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int64_t e = c + (int64_t)stride * q + at;
        u[q] = e < e1 ? a.ci[e] : -1;
      }
#pragma unroll
      for (int q = 0; q < 8; q++) hit |= test(u[q], p, was) ? 1u << q : 0u;
#pragma unroll
      for (int q = 0; q < 8; q++) local_stage<ORDER>(a, buf, held, (hit >> q) & 1u, u[q], b, t);
    }
  };
  const int s2 = n2 > 0 ? (int)max((int64_t)1, (int64_t)gridDim.x / n2) : 1;
  for (int64_t i = blockIdx.x; i < n2 * s2; i += gridDim.x) {
    const int v = l2[i / s2], p = a.h[v], was = ORDER ? 0 : __ldcg(a.old + v);
    if (ORDER || p < was) row(a.rp[v], a.rp[v + 1], (int)(i % s2) * kThreads + threadIdx.x, s2 * kThreads, p, was);
  }
  const int s1 = n1 > 0 ? (int)max((int64_t)1, min((int64_t)16, nwarps / n1)) : 1;
  for (int64_t i = gwarp; i < n1 * s1; i += nwarps) {
    const int v = l1[i / s1], p = a.h[v], was = ORDER ? 0 : __ldcg(a.old + v);
    if (ORDER || p < was) row(a.rp[v], a.rp[v + 1], (int)(i % s1) * 32 + lane, s1 * 32, p, was);
  }
  const int per = short_batch(n0, nwarps);
  for (int64_t c = gwarp * per; c < n0; c += nwarps * per) {
    const int64_t i = c + lane;
    int v = -1, len = 0, p = 0, was = 0;
    int64_t e0 = 0;
    if (lane < per && i < n0) {
      v = l0 ? l0[i] : (int)i;
      e0 = a.rp[v];
      const int64_t d = a.rp[v + 1] - e0;
      len = d <= 32 ? (int)d : 0;
      if (len) {
        p = a.h[v];
        if (!ORDER) was = __ldcg(a.old + v);
      }
    }
    unsigned m = __ballot_sync(0xffffffffu, len > 0 && (ORDER || p < was));
    while (m) {
      int u[4];
      bool hit[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int j = m ? __ffs(m) - 1 : -1;
        m &= m - 1;
        const int64_t e = __shfl_sync(0xffffffffu, e0, j & 31);
        const int L = __shfl_sync(0xffffffffu, len, j & 31);
        const int pj = __shfl_sync(0xffffffffu, p, j & 31), wj = __shfl_sync(0xffffffffu, was, j & 31);
        u[q] = (j >= 0 && lane < L) ? a.ci[e + lane] : -1;
        hit[q] = test(u[q], pj, wj);
      }
#pragma unroll
      for (int q = 0; q < 4; q++) local_stage<ORDER>(a, buf, held, hit[q], u[q], b, t);
    }
  }
  local_stage_end<ORDER>(a, buf, held, b, t);
}

__global__ void __launch_bounds__(kThreads, 1) kcore_local_kernel(LocalArgs a) {
  __shared__ LocalShared S;
  if (threadIdx.x == 0) S.barriers = 0;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t gwarp = (int64_t)wib * gridDim.x + blockIdx.x;  // neighbouring items go to different blocks
  const int64_t nwarps = (int64_t)gridDim.x * kWarps;
  const unsigned lt = (1u << lane) - 1u;
  const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
  int *bin = S.bins + wib * kLocalBins, *buf = S.stage[wib];
  const int64_t n = a.n;

  // ---- bounds, the vertices of longer rows, and the degrees
  for (int i = threadIdx.x; i < 256; i += kThreads) S.bins[i] = 0;
  __syncthreads();
  int top = 0;
  for (int64_t b = gwarp * 32; b < n; b += nwarps * 32) {
    const int64_t v = b + lane;
    int d = 0;
    if (v < n) {
      d = (int)(a.rp[v + 1] - a.rp[v]);
      const int x = min(d, a.cap);
      a.h[v] = x;
      a.stamp[v] = 0;
      top = max(top, d);
    }
    const int db = v < n ? degree_bin(d) : -1;
    if (__all_sync(0xffffffffu, db == __shfl_sync(0xffffffffu, db, 0))) {
      if (lane == 0) atomicAdd(&S.bins[db], 32);
    } else if (db >= 0) {
      atomicAdd(&S.bins[db], 1);
    }
#pragma unroll
    for (int q = 1; q < 3; q++) {
      const bool in = v < n && row_class(d) == q;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (!m) continue;
      int at = 0;
      if (lane == 0) at = atomicAdd(&a.ctl->all[q - 1], __popc(m));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (in) a.all[q - 1][at + __popc(m & lt)] = (int)v;
    }
  }
  top = dev::warp_max(top);
  if (lane == 0) atomicMax(a.maxdeg, top);
  __syncthreads();
  for (int i = threadIdx.x; i < 256; i += kThreads)
    if (S.bins[i]) atomicAdd(&a.ctl->hist[i], S.bins[i]);
  if (!local_barrier(a, S, nullptr)) return;
  if (wib == 0) {
    int c[8], sum = 0, high = 0, low = INT_MAX;
#pragma unroll
    for (int q = 0; q < 8; q++) sum += c[q] = __ldcg(&a.ctl->hist[8 * lane + q]);
    int below = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, below, o);
      if (lane >= o) below += y;
    }
    below -= sum;
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int d = 8 * lane + q < 240 ? bin_degree(8 * lane + q) : INT_MAX;
      if (n - below >= d) high = max(high, d);
      below += c[q];
      if (below > n / 64) low = min(low, d);
    }
    high = __reduce_max_sync(0xffffffffu, high);
    low = __reduce_min_sync(0xffffffffu, low);
    if (lane == 0) S.red[0] = local_pays(high, low, __ldcg(a.maxdeg), a.nnz);
  }
  __syncthreads();
  if (!S.red[0]) return;  // done stays 0: left to the peel
  const int all1 = __ldcg(&a.ctl->all[0]), all2 = __ldcg(&a.ctl->all[1]);

  // ---- values
  int64_t n0 = n, n1 = all1, n2 = all2;
  const int32_t *l0 = nullptr, *l1 = a.all[0], *l2 = a.all[1];
  int step = 0;
  for (;;) {
    const int nxt = (step + 1) & 1;
    step++;
    if (leader) a.ctl->n[nxt][0] = a.ctl->n[nxt][1] = a.ctl->n[nxt][2] = 0;
    // evaluate: long rows first
    for (int64_t i = blockIdx.x; i < n2; i += gridDim.x) {
      const int v = l2[i];
      const int64_t e0 = a.rp[v];
      const int h = __ldcg(a.h + v);
      const int x = eval_block(a, S, e0, a.rp[v + 1] - e0, h);
      if (threadIdx.x == 0) {
        a.old[v] = h;
        if (x < h) a.h[v] = x;
      }
    }
    __syncthreads();
    for (int64_t i = gwarp; i < n1; i += nwarps) {
      const int v = l1[i];
      const int64_t e0 = a.rp[v];
      const int h = __ldcg(a.h + v);
      const int x = eval_warp(a, e0, (int)(a.rp[v + 1] - e0), h, bin);
      if (lane == 0) {
        a.old[v] = h;
        if (x < h) a.h[v] = x;
      }
    }
    const int per = short_batch(n0, nwarps);
    for (int64_t b = gwarp * per; b < n0; b += nwarps * per) {
      const int64_t i = b + lane;
      int v = -1, len = 0, h = 0;
      int64_t e0 = 0;
      if (lane < per && i < n0) {
        v = l0 ? l0[i] : (int)i;
        e0 = a.rp[v];
        const int64_t d = a.rp[v + 1] - e0;
        len = d <= 32 ? (int)d : 0;
        if (len) h = __ldcg(a.h + v);
      }
      int nh = h;
      unsigned m = __ballot_sync(0xffffffffu, len > 0);
      while (m) {
        int j[4], x[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          j[q] = m ? __ffs(m) - 1 : -1;
          m &= m - 1;
          const int64_t e = __shfl_sync(0xffffffffu, e0, j[q] & 31);
          const int L = __shfl_sync(0xffffffffu, len, j[q] & 31);
          x[q] = (j[q] >= 0 && lane < L) ? a.ci[e + lane] : -1;
        }
#pragma unroll
        for (int q = 0; q < 4; q++) x[q] = x[q] >= 0 ? a.h[x[q]] : INT_MIN;
#pragma unroll
        for (int q = 0; q < 4; q++) {
          if (j[q] < 0) break;
          int k = __shfl_sync(0xffffffffu, h, j[q]);
          while (__popc(__ballot_sync(0xffffffffu, x[q] >= k)) < k) k--;
          if (lane == j[q]) nh = k;
        }
      }
      if (len) {
        a.old[v] = h;
        if (nh < h) a.h[v] = nh;
      }
    }
    if (!local_barrier(a, S, nullptr)) return;
    // push: the lowered vertices list the neighbours that counted on them
    local_walk<false>(a, l0, l1, l2, n0, n1, n2, step, buf, nxt, nxt);
    if (!local_barrier(a, S, a.ctl->n[nxt])) return;
    n0 = S.cnt[0];
    n1 = S.cnt[1];
    n2 = S.cnt[2];
    l0 = a.list[nxt][0];
    l1 = a.list[nxt][1];
    l2 = a.list[nxt][2];
    if (n0 + n1 + n2 == 0) break;
    if (step >= kLocalSteps) return;  // done stays 0: left to the peel
  }

  // ---- order.  Supports within K's own core and the shell sizes (a.taken).
  if (leader) {
    for (int t = 0; t < 3; t++) a.ctl->n[t][0] = a.ctl->n[t][1] = a.ctl->n[t][2] = 0;
  }
  __syncthreads();
  for (int64_t i = blockIdx.x; i < all2; i += gridDim.x) {
    const int v = a.all[1][i];
    const int k = __ldcg(a.h + v);
    const int64_t e0 = a.rp[v], e1 = a.rp[v + 1];
    __syncthreads();
    if (threadIdx.x == 0) S.red[0] = 0;
    __syncthreads();
    int c = 0;
#pragma unroll 4
    for (int64_t e = e0 + threadIdx.x; e < e1; e += kThreads) c += a.h[a.ci[e]] >= k ? 1 : 0;
    c = dev::warp_sum(c);
    if (lane == 0 && c) atomicAdd(&S.red[0], c);
    __syncthreads();
    if (threadIdx.x == 0) a.old[v] = S.red[0];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kLocalBlockBins; i += kThreads) S.bins[i] = 0;
  __syncthreads();
  for (int64_t i = gwarp; i < all1; i += nwarps) {
    const int v = a.all[0][i];
    const int k = __ldcg(a.h + v);
    const int64_t e0 = a.rp[v], e1 = a.rp[v + 1];
    int c = 0;
#pragma unroll 4
    for (int64_t e = e0 + lane; e < e1; e += 32) c += a.h[a.ci[e]] >= k ? 1 : 0;
    c = dev::warp_sum(c);
    if (lane == 0) a.old[v] = c;
  }
  int kmax = 0;
  for (int64_t b = gwarp * 32; b < n; b += nwarps * 32) {
    const int64_t v = b + lane;
    int len = 0, k = 0, cnt = 0;
    int64_t e0 = 0;
    if (v < n) {
      e0 = a.rp[v];
      const int64_t d = a.rp[v + 1] - e0;
      len = d <= 32 ? (int)d : -1;
      k = __ldcg(a.h + v);
      kmax = max(kmax, k);
      if (k < kLocalBlockBins) atomicAdd(&S.bins[k], 1);
      else atomicAdd(a.taken + k, 1);
    }
    unsigned m = __ballot_sync(0xffffffffu, len > 0);
    while (m) {
      int j[4], x[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        j[q] = m ? __ffs(m) - 1 : -1;
        m &= m - 1;
        const int64_t e = __shfl_sync(0xffffffffu, e0, j[q] & 31);
        const int L = __shfl_sync(0xffffffffu, len, j[q] & 31);
        x[q] = (j[q] >= 0 && lane < L) ? a.ci[e + lane] : -1;
      }
#pragma unroll
      for (int q = 0; q < 4; q++) x[q] = x[q] >= 0 ? a.h[x[q]] : INT_MIN;
#pragma unroll
      for (int q = 0; q < 4; q++) {
        if (j[q] < 0) break;
        const int kk = __shfl_sync(0xffffffffu, k, j[q]);
        const int c = __popc(__ballot_sync(0xffffffffu, x[q] >= kk));
        if (lane == j[q]) cnt = c;
      }
    }
    if (len >= 0 && v < n) a.old[v] = cnt;
  }
  kmax = dev::warp_max(kmax);
  if (lane == 0) atomicMax(&a.ctl->all[3], kmax);
  __syncthreads();
  for (int i = threadIdx.x; i < kLocalBlockBins; i += kThreads)
    if (S.bins[i]) atomicAdd(a.taken + i, S.bins[i]);
  if (!local_barrier(a, S, nullptr)) return;
  kmax = __ldcg(&a.ctl->all[3]);
  if (blockIdx.x == 0) {  // first positions; a.taken restarts at 0
    int carry = 0;
    for (int b = 0; b <= kmax; b += kThreads) {
      const int k = b + threadIdx.x;
      const int x = k <= kmax ? __ldcg(a.taken + k) : 0;
      int incl = x;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      __syncthreads();
      if (lane == 31) S.bins[wib] = incl;
      __syncthreads();
      int before = 0, tot = 0;
      for (int w = 0; w < kWarps; w++) {
        if (w < wib) before += S.bins[w];
        tot += S.bins[w];
      }
      if (k <= kmax) {
        a.start[k] = carry + before + incl - x;
        a.taken[k] = 0;
      }
      carry += tot;
    }
  }
  if (!local_barrier(a, S, nullptr)) return;
  for (int64_t b = gwarp * 32; b < n; b += nwarps * 32) {
    const int64_t v = b + lane;
    bool has = false;
    if (v < n) has = __ldcg(a.old + v) <= a.h[v];
    if (__any_sync(0xffffffffu, has)) local_append<true>(a, has, (int)v, 0, 0);
  }
  if (!local_barrier(a, S, a.ctl->n[0])) return;
  for (int r = 0;; r++) {
    const int cur = r & 1, nxt = cur ^ 1;
    n0 = S.cnt[0];
    n1 = S.cnt[1];
    n2 = S.cnt[2];
    if (n0 + n1 + n2 == 0) break;
    if (r >= kLocalSteps) return;
    // the counters of round r - 1, free since the last barrier and first used
    // again after the next one
    if (leader) a.ctl->n[(r + 2) % 3][0] = a.ctl->n[(r + 2) % 3][1] = a.ctl->n[(r + 2) % 3][2] = 0;
    local_walk<true>(a, a.list[cur][0], a.list[cur][1], a.list[cur][2], n0, n1, n2, 0, buf, nxt, (r + 1) % 3);
    if (!local_barrier(a, S, a.ctl->n[(r + 1) % 3])) return;
  }
  if (leader) {
    *a.maxcore = kmax;
    if (__ldcg(&a.ctl->all[2]) == (int)n) *a.done = 1;
  }
}

// Batches of small graphs: one block peels one whole graph at a time
// (degrees in shared memory, shared-memory atomics, block barriers between
// sub-rounds), blocks taking graphs from a counter.  The peel order of graph
// g is written to order[voff[g] ..), so each graph's segment is its own
// degeneracy order.
constexpr int kBatchCap = (int)kBatchPeelCap;  // largest graph this kernel takes
constexpr int kBatchThreads = 512;

__global__ void __launch_bounds__(kBatchThreads) kcore_batch_kernel(int32_t count, const int64_t *__restrict__ voff,
                                                                    const int64_t *__restrict__ rp,
                                                                    const int32_t *__restrict__ ci,
                                                                    int32_t *__restrict__ core,
                                                                    int32_t *__restrict__ order, int32_t *next,
                                                                    int32_t *maxdeg, int32_t *maxcore, int32_t *err) {
  __shared__ int deg[kBatchCap];
  __shared__ int q[kBatchCap];
  __shared__ int s_g, s_tail, s_min;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = kBatchThreads / 32;
  const unsigned lt = (1u << lane) - 1u;
  for (;;) {
    __syncthreads();
    if (tid == 0) s_g = atomicAdd(next, 1);
    __syncthreads();
    const int g = s_g;
    if (g >= count) break;
    const int64_t v0 = voff[g];
    const int ng = (int)(voff[g + 1] - v0);
    int lmax = 0;
    for (int i = tid; i < ng; i += kBatchThreads) {
      deg[i] = (int)(rp[v0 + i + 1] - rp[v0 + i]);
      lmax = max(lmax, deg[i]);
    }
    lmax = dev::warp_max(lmax);
    if (lane == 0) atomicMax(maxdeg, lmax);
    if (tid == 0) s_tail = 0;
    __syncthreads();
    int k = 0, head = 0, kmax_g = 0;
    while (true) {
      // scan: every unpeeled vertex with degree == k joins the level
      __syncthreads();  // everyone has read s_min / s_tail of the last level
      if (tid == 0) s_min = INT_MAX;
      __syncthreads();
      int lmin = INT_MAX;
      for (int b = wid * 32; b < ng; b += kBatchThreads) {
        const int i = b + lane;
        const int d = (i < ng) ? deg[i] : INT_MIN;
        const bool hit = d == k;
        if (d > k) lmin = min(lmin, d);
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (m) {
          int base = 0;
          if (lane == 0) base = atomicAdd(&s_tail, __popc(m));
          base = __shfl_sync(0xffffffffu, base, 0);
          if (hit) {
            q[base + __popc(m & lt)] = i;
            core[v0 + i] = k;
          }
        }
      }
      lmin = -dev::warp_max(-lmin);
      if (lane == 0 && lmin != INT_MAX) atomicMin(&s_min, lmin);
      __syncthreads();
      int tail = s_tail;
      if (tail == head) {  // nothing at level k
        if (s_min == INT_MAX) break;  // every vertex peeled
        k = s_min;
        continue;
      }
      kmax_g = k;
      // sub-rounds: warps walk the rows of q[head, tail); neighbours that fall
      // to k join q for the next sub-round
      while (head < tail) {
        for (int j = head + wid; j < tail; j += nw) {
          const int i = q[j];
          const int64_t e0 = rp[v0 + i], e1 = rp[v0 + i + 1];
          for (int64_t eb = e0; eb < e1; eb += 32) {
            const int64_t e = eb + lane;
            bool nf = false;
            int u = -1;
            if (e < e1) {
              u = (int)(ci[e] - v0);
              if ((unsigned)u >= (unsigned)ng) {  // an edge leaving the graph: not a valid batch
                atomicExch(err, kDevCheck);
                u = -1;
              } else if (deg[u] > k) {
                nf = (atomicSub(&deg[u], 1) == k + 1);
              }
            }
            const unsigned m = __ballot_sync(0xffffffffu, nf);
            if (m) {
              int base = 0;
              if (lane == 0) base = atomicAdd(&s_tail, __popc(m));
              base = __shfl_sync(0xffffffffu, base, 0);
              if (nf) {
                q[base + __popc(m & lt)] = u;
                core[v0 + u] = k;
              }
            }
          }
        }
        __syncthreads();
        head = tail;
        tail = s_tail;
        __syncthreads();
      }
      k++;
    }
    // the queue is the graph's peel order (core numbers were written on append)
    __syncthreads();
    for (int j = tid; j < ng; j += kBatchThreads) order[v0 + j] = (int32_t)(v0 + q[j]);
    if (tid == 0) atomicMax(maxcore, kmax_g);
    __syncthreads();
  }
}

__global__ void batch_pos_kernel(int64_t n, const int32_t *__restrict__ order, int32_t *__restrict__ pos) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    pos[order[i]] = (int32_t)i;
}

}  // namespace

// Enqueues kcore_local_kernel; *out: three device words (done, largest
// degree, K(G)).
static int launch_local(mc_graph *g, long long spin_limit, const int32_t **out) {
  const int64_t n = g->n;
  LocalArgs a{};
  a.n = n;
  a.nnz = g->nnz;
  a.cap = (int)std::sqrt((double)g->nnz) + 1;
  a.rp = g->row_ptr;
  a.ci = g->col_idx;
  a.h = g->core;
  a.order = g->order;
  a.pos = g->pos;
  a.err = g->err;
  a.spin = spin_limit;
  const int64_t c1 = std::min<int64_t>(n, g->nnz / 33 + 1), c2 = std::min<int64_t>(n, g->nnz / kLocalWarpRow + 1);
  void *p;
  MC_TRY(ws_get(g, "kl.v", (size_t)(4 * n + 3 * (c1 + c2) + a.cap + 2) * sizeof(int32_t), &p));
  int32_t *w = (int32_t *)p;
  auto take = [&](int64_t k) {
    int32_t *r = w;
    w += k;
    return r;
  };
  a.old = take(n);
  a.stamp = take(n);
  for (int b = 0; b < 2; b++) {
    a.list[b][0] = take(n);
    a.list[b][1] = take(c1);
    a.list[b][2] = take(c2);
  }
  a.all[0] = take(c1);
  a.all[1] = take(c2);
  a.start = take(a.cap + 2);
  const size_t ctl_bytes = sizeof(LocalCtl) + 64 + (size_t)(a.cap + 2) * sizeof(int32_t);
  MC_TRY(ws_get(g, "kl.ctl", ctl_bytes, &p));
  MC_CUDA_TRY(cudaMemsetAsync(p, 0, ctl_bytes, g->stream));
  a.ctl = (LocalCtl *)p;
  a.done = (int32_t *)((char *)p + sizeof(LocalCtl));
  a.maxdeg = a.done + 1;
  a.maxcore = a.done + 2;
  a.taken = (int32_t *)((char *)p + sizeof(LocalCtl) + 64);
  *out = a.done;
  int per_sm = 0;
  MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kcore_local_kernel, kThreads, 0));
  if (per_sm < 1) return MC_ERR_CUDA;
  const int blocks = (int)std::min<int64_t>(g->sm_count, std::max<int64_t>(1, (n + g->nnz / 2 + kThreads - 1) / kThreads));
  void *args[] = {&a};
  MC_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)kcore_local_kernel, dim3(blocks), dim3(kThreads), args, 0,
                                          g->stream));
  g_launches++;
  return MC_OK;
}

int launch_core_numbers(mc_graph *g, long long spin_limit) {
  const int64_t n = g->n;
  g->order_given = false;
  if (n == 0) {
    g->max_core = 0;
    g->cores_valid = true;
    return MC_OK;
  }
  void *p;
  if (g->count > 1 && g->max_graph_n <= kBatchCap) {
    MC_TRY(ws_get(g, "kc.bctl", 64, &p));
    int32_t *bctl = (int32_t *)p;  // [0] graph counter, [1] max degree, [2] max core
    MC_CUDA_TRY(cudaMemsetAsync(bctl, 0, 64, g->stream));
    int per_sm = 0;
    MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kcore_batch_kernel, kBatchThreads, 0));
    const int blocks = (int)std::min<int64_t>(g->count, (int64_t)g->sm_count * std::max(per_sm, 1));
    kcore_batch_kernel<<<blocks, kBatchThreads, 0, g->stream>>>(g->count, g->voff, g->row_ptr, g->col_idx, g->core,
                                                                g->order, bctl, bctl + 1, bctl + 2, g->err);
    batch_pos_kernel<<<(int)std::min<int64_t>((n + 255) / 256, (int64_t)g->sm_count * 8), 256, 0, g->stream>>>(
        n, g->order, g->pos);
    g_launches += 2;
    MC_CUDA_TRY(cudaGetLastError());
    if (g->capturing) {
      g->cores_valid = true;
      return MC_OK;
    }
    int32_t *host = (int32_t *)g->h_small;
    MC_CUDA_TRY(cudaMemcpyAsync(host, bctl + 1, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, g->stream));
    MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
    MC_TRY(check_device_error(g));
    g->max_degree = host[0];
    g->max_core = host[1];
    g->cores_valid = true;
    return MC_OK;
  }
  // mid-size graphs: all levels at once, if that pays; the peel below is
  // skipped on the device then in a captured solve and not launched otherwise
  const int32_t *skip = nullptr;
  if (g->nnz <= kLocalMaxNnz) {
    MC_TRY(launch_local(g, spin_limit, &skip));
    if (!g->capturing) {
      int32_t *host = (int32_t *)g->h_small;
      MC_CUDA_TRY(cudaMemcpyAsync(host, skip, 3 * sizeof(int32_t), cudaMemcpyDeviceToHost, g->stream));
      MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
      MC_TRY(check_device_error(g));
      if (host[0]) {
        g->max_degree = host[1];
        g->max_core = host[2];
        g->cores_valid = true;
        return MC_OK;
      }
      skip = nullptr;
    }
  }
  MC_TRY(ws_get(g, "kc.deg", n * sizeof(int32_t), &p));
  int32_t *deg = (int32_t *)p;
  MC_TRY(ws_get(g, "kc.live", 2 * n * sizeof(int32_t) + 64, &p));
  int32_t *live0 = (int32_t *)p, *live1 = live0 + n;
  const int64_t wcap = n + g->nnz / kChunk + 64;
  MC_TRY(ws_get(g, "kc.wq", wcap * sizeof(long long), &p));
  long long *wq = (long long *)p;
  MC_TRY(ws_get(g, "kc.ctl", sizeof(KcoreCtl) + 64, &p));
  KcoreCtl *ctl = (KcoreCtl *)p;
  int32_t *maxdeg = (int32_t *)((char *)p + sizeof(KcoreCtl) + 16);
  MC_CUDA_TRY(cudaMemsetAsync(ctl, 0, sizeof(KcoreCtl) + 64, g->stream));
  MC_CUDA_TRY(cudaMemsetAsync(wq, 0xff, wcap * sizeof(long long), g->stream));

  int ib = (int)std::min<int64_t>((n + 255) / 256, (int64_t)g->sm_count * 8);
  degree_init_kernel<<<ib, 256, 0, g->stream>>>(n, g->row_ptr, deg, g->core, maxdeg, skip);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());

  int per_sm = 0;
  const size_t pool = sizeof(BlockPool);
  MC_CUDA_TRY(cudaFuncSetAttribute((const void *)kcore_peel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)pool));
  MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kcore_peel_kernel, kThreads, pool));
  if (per_sm < 1) return MC_ERR_CUDA;
  int blocks = g->sm_count;
  int64_t need = (n + kThreads - 1) / kThreads;
  if (need < blocks) blocks = (int)std::max<int64_t>(1, need);
  int64_t n_arg = n;
  const int64_t *rp = g->row_ptr;
  const int32_t *ci = g->col_idx;
  int32_t *core = g->core, *order = g->order, *err = g->err;
  long long sl = spin_limit;
  int nocheck = n <= kNoCheckMaxN ? 1 : 0;
  void *args[] = {&n_arg, (void *)&rp, (void *)&ci, &deg, &core, &order, &live0, &live1, &wq, &ctl, &err, &sl,
                  &nocheck, (void *)&skip};
  MC_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)kcore_peel_kernel, dim3(blocks), dim3(kThreads), args, pool,
                                          g->stream));
  g_launches++;
  peel_pos_kernel<<<ib, 256, 0, g->stream>>>(n, g->order, g->pos, g->core, maxdeg + 1, g->err, skip);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  if (g->capturing) {  // K(G) and the degree bound are kept from the direct solve before capture
    g->cores_valid = true;
    return MC_OK;
  }
  int32_t *host = (int32_t *)g->h_small;
  MC_CUDA_TRY(cudaMemcpyAsync(host, maxdeg, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, g->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
  MC_TRY(check_device_error(g));
  g->max_degree = host[0];
  g->max_core = host[1];
  g->cores_valid = true;
  return MC_OK;
}

}  // namespace mc

// ------------------------------------------------------------------------
// Core numbers without any device allocation.
//
// Some callers cannot call cudaMalloc: allocator hooks that must not
// re-enter the allocator, or hosts that hand the library a fixed memory
// budget and own every byte of it.  For them this entry point
// runs the same peel with its working memory in a file-scope device array of
// fixed size, reserved when the library is loaded and held by every GPU that
// loads it until the process exits.
// ------------------------------------------------------------------------

namespace mc {
namespace {

constexpr int64_t kNoAllocMaxN = 1 << 20;     // vertices
constexpr int64_t kNoAllocMaxNnz = 1 << 26;   // CSR entries (2 x edges)
constexpr int64_t kNoAllocWq = kNoAllocMaxN + kNoAllocMaxNnz / kChunk + 64;
constexpr size_t kNoAllocCtlBytes = 4096;
// layout: control block | degrees | two live lists | peel order | positions | work items
constexpr size_t kNaOffDeg = kNoAllocCtlBytes;
constexpr size_t kNaOffLive = kNaOffDeg + 4 * kNoAllocMaxN;
constexpr size_t kNaOffOrder = kNaOffLive + 8 * kNoAllocMaxN;
constexpr size_t kNaOffPos = kNaOffOrder + 4 * kNoAllocMaxN;
constexpr size_t kNaOffWq = kNaOffPos + 4 * kNoAllocMaxN;
constexpr size_t kNoAllocBytes = kNaOffWq + 8 * kNoAllocWq;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// The bounds the peel's memory accesses rely on, checked before it runs:
// row_ptr[0] = 0, row_ptr nondecreasing (so every row lies inside
// [0, row_ptr[n]) = [0, nnz)), and every column index in [0, n).  Reads
// only row_ptr[0..n] and col_idx[0..nnz); a failure sets *bad.
__global__ void csr_bounds_kernel(int64_t n, int64_t nnz, const int64_t *__restrict__ rp,
                                  const int32_t *__restrict__ ci, int32_t *bad) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool ok = true;
  for (int64_t v = t0; v < n; v += stride) {
    const int64_t a = rp[v], b = rp[v + 1];
    if (b < a || (v == 0 && a != 0)) ok = false;
  }
  for (int64_t e = t0; e < nnz; e += stride) {
    const int32_t u = ci[e];
    if (u < 0 || (int64_t)u >= n) ok = false;
  }
  if (!ok) atomicExch(bad, 1);
}

// device address of g_noalloc_scratch, per device (set up on first use)
static void *g_noalloc_ptr[64];
static std::mutex g_noalloc_mu;

int noalloc_setup(int dev, unsigned char **out) {
  if (dev < 0 || dev >= 64) return MC_ERR_ARG;
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      set_last_cuda_error(e, "cudaGetSymbolAddress(g_noalloc_scratch)", __FILE__, __LINE__);
      return MC_ERR_CUDA;
    }
    g_noalloc_ptr[dev] = p;
  }
  *out = (unsigned char *)g_noalloc_ptr[dev];
  return MC_OK;
}

}  // namespace
}  // namespace mc

extern "C" int mc_core_numbers_noalloc(int64_t n, const int64_t *row_ptr, const int32_t *col_idx,
                                       int32_t *core_out, int32_t *max_core_out, void *cuda_stream) {
  using namespace mc;
  if (n < 0 || (n > 0 && (!row_ptr || !col_idx || !core_out))) return MC_ERR_ARG;
  if (n > kNoAllocMaxN) return MC_ERR_TOO_LARGE;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  if (max_core_out) *max_core_out = 0;
  if (n == 0) return MC_OK;
  int dev = 0, sms = 0;
  MC_CUDA_TRY(cudaGetDevice(&dev));
  MC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  unsigned char *base = nullptr;
  MC_TRY(noalloc_setup(dev, &base));
  int64_t nnz = 0;
  MC_CUDA_TRY(cudaMemcpyAsync(&nnz, row_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  MC_CUDA_TRY(cudaStreamSynchronize(s));
  if (nnz < 0) return MC_ERR_ARG;
  if (nnz > kNoAllocMaxNnz) return MC_ERR_TOO_LARGE;

  KcoreCtl *ctl = (KcoreCtl *)base;
  int32_t *maxdeg = (int32_t *)(base + 1024);  // [0] max degree, [1] max core
  int32_t *err = (int32_t *)(base + 2048);
  int32_t *bad = (int32_t *)(base + 3072);
  int32_t *deg = (int32_t *)(base + kNaOffDeg);
  int32_t *live0 = (int32_t *)(base + kNaOffLive), *live1 = live0 + n;
  int32_t *order = (int32_t *)(base + kNaOffOrder);
  int32_t *pos = (int32_t *)(base + kNaOffPos);
  long long *wq = (long long *)(base + kNaOffWq);
  // the array keeps the previous call's contents: clear the control block
  MC_CUDA_TRY(cudaMemsetAsync(base, 0, kNoAllocCtlBytes, s));

  // the peel indexes its arrays by row offsets and column entries, so those
  // are checked first; the caller's graph is not otherwise validated
  const int cb = (int)std::min<int64_t>((std::max(n, nnz) + 255) / 256, (int64_t)sms * 8);
  csr_bounds_kernel<<<cb, 256, 0, s>>>(n, nnz, row_ptr, col_idx, bad);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  int32_t h_bad = 0;
  MC_CUDA_TRY(cudaMemcpyAsync(&h_bad, bad, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  MC_CUDA_TRY(cudaStreamSynchronize(s));
  if (h_bad) return MC_ERR_INVALID_GRAPH;

  const int ib = (int)std::min<int64_t>((n + 255) / 256, (int64_t)sms * 8);
  degree_init_kernel<<<ib, 256, 0, s>>>(n, row_ptr, deg, core_out, maxdeg, nullptr);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  int per_sm = 0;
  const size_t pool = sizeof(BlockPool);
  MC_CUDA_TRY(cudaFuncSetAttribute((const void *)kcore_peel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)pool));
  MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kcore_peel_kernel, kThreads, pool));
  if (per_sm < 1) return MC_ERR_CUDA;
  int blocks = sms;
  const int64_t need = (n + kThreads - 1) / kThreads;
  if (need < blocks) blocks = (int)std::max<int64_t>(1, need);
  int64_t n_arg = n;
  long long sl = kDefaultSpinLimit;
  int nocheck = n <= kNoCheckMaxN ? 1 : 0;
  const int32_t *skip = nullptr;
  void *args[] = {&n_arg, (void *)&row_ptr, (void *)&col_idx, &deg, &core_out, &order, &live0, &live1, &wq, &ctl,
                  &err, &sl, &nocheck, (void *)&skip};
  MC_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)kcore_peel_kernel, dim3(blocks), dim3(kThreads), args, pool,
                                          s));
  g_launches++;
  peel_pos_kernel<<<ib, 256, 0, s>>>(n, order, pos, core_out, maxdeg + 1, err, nullptr);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  int32_t host[3] = {0, 0, 0};
  MC_CUDA_TRY(cudaMemcpyAsync(host, maxdeg, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  MC_CUDA_TRY(cudaMemcpyAsync(host + 2, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  MC_CUDA_TRY(cudaStreamSynchronize(s));
  if (host[2] == kDevTimeout) return MC_ERR_TIMEOUT;
  if (host[2] != kDevOk) return MC_ERR_DEVICE_CHECK;
  if (max_core_out) *max_core_out = host[1];
  return MC_OK;
}
