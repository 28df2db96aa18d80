// Clique-peeling vertex order (Section 6.2) and the gap cost of an order.
//
// Section 6.2 orders the vertices for compression by taking a large clique
// with the heuristic, removing it and repeating, the vertices following the
// cliques in the order found and each clique's members by degree.  Here the
// cliques are taken in rounds, all vertices at once:
//
//   grow    every alive vertex v with no valid stored clique grows Algorithm
//           1's greedy clique C(v) over the alive vertices: candidates are
//           its alive neighbours, the next member is the remaining candidate
//           of largest core number (ties: larger degree, then smaller id),
//           and the candidates are filtered to that member's neighbours.  A
//           stored clique stays valid while all its members are alive (the
//           vertices that died were rejected candidates, whose removal
//           changes no decision of the greedy scan).  A thread per vertex
//           checks that and lists the stale ones; warps grow them, whole
//           blocks those of many neighbours.
//   scatter key(v) = |C(v)| << 32 | (2^31 - 1 - rank(v)); every member u of
//           C(v) takes the largest key of the cliques holding it (atomicMax).
//   accept  C(v) is accepted iff it holds the largest key at every member;
//           accepted cliques are disjoint, and the globally largest key is
//           always accepted.
//   place   an exclusive scan over v of (1 << 32 | |C(v)|) for the accepted
//           ones gives each its group index and position; a warp per
//           accepted clique writes its members ranked by decreasing degree
//           (ties: smaller id) and marks them dead.
//
// Rounds repeat until every vertex is placed (the host queues one ahead of the
// count it looks at; a round after the last vertex changes nothing).  Cliques
// live in one arena laid out like the CSR: vertex v's candidates occupy the front
// of [rp[v], rp[v+1]) while it grows, and its members other than v end at the top
// of that range, so the arena is nnz int32 and needs no per-warp buffers or size
// limits.
//
// The gap cost relabels the graph by an order (new id = position), sorts
// every new row (bitonic networks in a warp's registers up to 1,024 entries;
// above, a block sets a bit per entry and reads the bits in order, or runs the
// network in shared memory), and sums log2(1 + gap) over the entries, the
// first gap of row p taken from p itself: 1 + gap rounded once to single
// precision, log2f (within 1 ulp), summed exactly in units of 2^-24 (in double
// for the graph as it was loaded).
#include <algorithm>
#include <climits>

#include "mc_internal.cuh"
#include "scan.cuh"

namespace mc {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kOT = 256;         // threads per block of the warp-per-vertex kernels
constexpr int kWarpSortMax = 1024;
constexpr int kBlockSortMax = 16384;
constexpr int kBigT = 1024;      // threads of the block sorter
constexpr int kGT = 256;         // threads of a growing block
constexpr int kGW = kGT / 32;
constexpr int64_t kBlockGrowMin = 4096;  // neighbours above which a block grows the clique
constexpr int64_t kMidGrowMin = 512;     // ... while few vertices have more than these
constexpr unsigned kMidPerBlock = 8;     // few: at most this many per growing block
constexpr int kTake = 4;                // listed vertices a warp takes at a time while there are many
constexpr int kNear = 256;              // candidates, and entries of a row, that a warp holds in shared memory
constexpr int64_t kManyVertices = 50000;  // ten per growing warp; above, throughput is the bound (grow_kernel)

struct OA {
  int64_t n;
  const int64_t *rp;
  const int32_t *ci, *core;
  const unsigned long long *kd;  // core number (high word) and degree per vertex
  const int32_t *rank;  // tie rank per vertex, nullptr: the vertex id
  uint8_t *alive;
  int32_t *csize;  // stored clique size; 0: grow; negative: accepted this round
  int32_t *arena;
  unsigned long long *bestkey;
  int64_t *ctl;  // [0] placed, [1] groups, [2] grows, [3] candidate tests, [4] rounds, [5] scan total,
                 // [6] the blocks' list length and next entry, [7] the warps' (two unsigned each), [8] the
                 // mid-size vertices' list length
  int64_t *goff;
  int32_t *order;
  int64_t *gstart;
  int32_t *ground;
  int32_t round;
  int32_t *err;
  int32_t *big;     // vertices for the blocks this round; from the list's end on, those of mid-size
  unsigned *nbig, *nmid;
  int32_t *stale;   // vertices for the warps this round
  unsigned *nstale, *take, *take_big;
};

struct CKey {
  int k, d, id;
};
__device__ __forceinline__ bool ahead(const CKey &a, const CKey &b) {
  if (a.k != b.k) return a.k > b.k;
  if (a.d != b.d) return a.d > b.d;
  return a.id < b.id;
}
// The warp's first key (core numbers and degrees are not negative).
__device__ __forceinline__ CKey warp_first(const CKey &x) {
  const int k = __reduce_max_sync(FULL, x.k);
  const int d = __reduce_max_sync(FULL, x.k == k ? x.d : INT_MIN);
  return CKey{k, d, __reduce_min_sync(FULL, (x.k == k && x.d == d) ? x.id : INT_MAX)};
}
__device__ __forceinline__ CKey ckey(const OA &a, int u) {
  const unsigned long long x = __ldg(a.kd + u);
  return CKey{(int)(x >> 32), (int)(x & 0xffffffffu), u};
}
__global__ void key_kernel(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ core,
                           unsigned long long *__restrict__ kd) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    kd[v] = ((unsigned long long)(unsigned)core[v] << 32) | (unsigned)(rp[v + 1] - rp[v]);
}
__device__ __forceinline__ unsigned long long key_of(const OA &a, int v, int size) {
  const int r = a.rank ? a.rank[v] : v;
  return ((unsigned long long)(unsigned)size << 32) | (unsigned)(0x7fffffff - r);
}

// Fence posts of w's row [r0, r1): every step-th entry, at most cap of them, to
// `post` (by nt threads, this one t).  A row of at most cap entries is held
// whole (step 1).
struct Fence {
  const int32_t *post, *row;
  int posts, top, len, step;
};
__device__ __forceinline__ Fence set_fence(const OA &a, int64_t r0, int64_t r1, int32_t *post, int cap, int t, int nt) {
  Fence f;
  f.row = a.ci + r0;
  f.post = post;
  f.len = (int)(r1 - r0);
  f.step = (f.len + cap - 1) / cap;
  f.posts = f.step ? (f.len + f.step - 1) / f.step : 0;
  f.top = f.posts ? 1 << (31 - __clz(f.posts)) : 0;
  for (int i = t; i < f.posts; i += nt) post[i] = f.row[(int64_t)i * f.step];
  return f;
}

// Greedy filter step of one warp: candidates in[i0, i1) other than w that are
// in w's row go to out, in order; their first key to nb.  Each lane looks up
// FLY candidates side by side: a binary search of the fence posts in shared
// memory, then of the step - 1 entries behind one.  in and out may be the same
// list (a tile is read before anything of it is written).
template <int FLY>
__device__ __forceinline__ int filter(const OA &a, const Fence &f, int w, const int32_t *in, int i0, int i1,
                                      int32_t *out, CKey &nb) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int kept = 0;
  for (int base = i0; base < i1; base += 32 * FLY) {
    int x[FLY], lo[FLY], left[FLY];
    bool keep[FLY];
#pragma unroll
    for (int q = 0; q < FLY; q++) {
      const int i = base + 32 * q + lane;
      x[q] = i < i1 ? in[i] : -1;
      lo[q] = 0;  // posts <= x
    }
    for (int st = f.top; st > 0; st >>= 1) {
#pragma unroll
      for (int q = 0; q < FLY; q++)
        if (base + 32 * q < i1 && lo[q] + st <= f.posts && f.post[lo[q] + st - 1] <= x[q]) lo[q] += st;
    }
    int any = 0;
#pragma unroll
    for (int q = 0; q < FLY; q++) {
      keep[q] = lo[q] > 0 && f.post[lo[q] - 1] == x[q];
      const int at = (lo[q] - 1) * f.step + 1;
      left[q] = (lo[q] > 0 && !keep[q]) ? min(f.step - 1, f.len - at) : 0;
      lo[q] = at;
      any |= left[q];
    }
    while (any) {
      int y[FLY];
#pragma unroll
      for (int q = 0; q < FLY; q++) y[q] = left[q] ? f.row[lo[q] + (left[q] >> 1)] : 0;
      any = 0;
#pragma unroll
      for (int q = 0; q < FLY; q++) {
        if (left[q] == 0) continue;
        const int h = left[q] >> 1;
        if (y[q] == x[q]) {
          keep[q] = true;
          left[q] = 0;
        } else if (y[q] < x[q]) {
          lo[q] += h + 1;
          left[q] -= h + 1;
        } else {
          left[q] = h;
        }
        any |= left[q];
      }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < FLY; q++) {
      keep[q] = keep[q] && x[q] != w;
      const unsigned m = __ballot_sync(FULL, keep[q]);
      if (keep[q]) {
        out[kept + __popc(m & lt)] = x[q];
        const CKey k = ckey(a, x[q]);
        if (ahead(k, nb)) nb = k;
      }
      kept += __popc(m);
    }
    __syncwarp();
  }
  return kept;
}

// A growing warp's shared memory.
struct GrowSmem {
  int32_t post[kGW][kNear], cand[kGW][kNear];
};

// Alive entries of v's row [s0, s1), one warp: to out (row order: ascending
// id), their first key to bk.
template <int FLY>
__device__ __forceinline__ int alive_of(const OA &a, int64_t s0, int64_t s1, int32_t *out, CKey &bk) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int cnt = 0;
  for (int64_t eb = s0; eb < s1; eb += 32 * FLY) {
    int u[FLY];
    bool ok[FLY];
#pragma unroll
    for (int q = 0; q < FLY; q++) {
      const int64_t e = eb + 32 * q + lane;
      u[q] = e < s1 ? a.ci[e] : -1;
    }
#pragma unroll
    for (int q = 0; q < FLY; q++) ok[q] = u[q] >= 0 && a.alive[u[q]] != 0;
#pragma unroll
    for (int q = 0; q < FLY; q++) {
      const unsigned m = __ballot_sync(FULL, ok[q]);
      if (ok[q]) {
        out[cnt + __popc(m & lt)] = u[q];
        const CKey k = ckey(a, u[q]);
        if (ahead(k, bk)) bk = k;
      }
      cnt += __popc(m);
    }
  }
  return cnt;
}

// Greedy growth of C(v) by one warp (all lanes) from cnt candidates (in
// ascending id) whose first key is bk, j members found so far: take the first
// candidate, keep the candidates adjacent to it, until none is left.  The
// candidates are in shared memory once they are at most kNear; before that at
// the front of v's arena range, where member j (from 1) goes to rp[v+1] - j
// after its filter: with cnt candidates left, cnt + j <= deg(v), so it lies
// past them.  Returns |C(v)|.
template <int FLY>
__device__ __forceinline__ int warp_steps(const OA &a, int64_t e1, int32_t *cand, int cnt, CKey bk, int j,
                                          int32_t *post, int32_t *near, unsigned long long &tests) {
  const int lane = threadIdx.x & 31;
  const CKey none{INT_MIN, INT_MIN, INT_MAX};
  while (cnt > 0) {
    if (cand != near && cnt <= kNear) {
      for (int i = lane; i < cnt; i += 32) near[i] = cand[i];
      cand = near;
    }
    const int w = bk.id;
    tests += (unsigned long long)cnt;
    int out = 0;
    CKey nb = none;
    if (cnt > 1) {
      __syncwarp();
      const Fence f = set_fence(a, a.rp[w], a.rp[w + 1], post, kNear, lane, 32);
      __syncwarp();
      out = filter<FLY>(a, f, w, cand, 0, cnt, cand, nb);
    }
    cnt = out;
    j++;
    if (lane == 0) a.arena[e1 - j] = w;
    __syncwarp();
    bk = warp_first(nb);
  }
  return 1 + j;
}

// Lane test: v's stored clique is missing or holds a placed member.
__device__ __forceinline__ bool needs_grow(const OA &a, int v) {
  const int s = a.csize[v];
  if (s <= 0) return true;
  const int64_t e1 = a.rp[v + 1];
  for (int i = 0; i < s - 1; i++)
    if (!a.alive[a.arena[e1 - 1 - i]]) return true;
  return false;
}

// check: a thread per vertex resets the alive vertices' keys and lists the
// ones that need a clique (warp-aggregated appends) by their row's length
__global__ void check_kernel(OA a) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < a.n; base += stride) {
    const int64_t vv = base + lane;
    int c = -1;  // 0: warps, 1: mid-size, 2: blocks
    if (vv < a.n && a.alive[vv]) {
      a.bestkey[vv] = 0ull;
      if (needs_grow(a, (int)vv)) {
        const int64_t d = a.rp[vv + 1] - a.rp[vv];
        c = d > kBlockGrowMin ? 2 : d > kMidGrowMin ? 1 : 0;
      }
    }
    const unsigned ms = __ballot_sync(FULL, c == 0), mm = __ballot_sync(FULL, c == 1), mb = __ballot_sync(FULL, c == 2);
    unsigned at = 0;
    if (lane == 0 && ms) at = atomicAdd(a.nstale, (unsigned)__popc(ms));
    if (lane == 1 && mm) at = atomicAdd(a.nmid, (unsigned)__popc(mm));
    if (lane == 2 && mb) at = atomicAdd(a.nbig, (unsigned)__popc(mb));
    const unsigned as = __shfl_sync(FULL, at, 0), am = __shfl_sync(FULL, at, 1), ab = __shfl_sync(FULL, at, 2);
    if (c == 0) a.stale[as + __popc(ms & lt)] = (int32_t)vv;
    if (c == 1) a.big[a.n - 1 - (am + __popc(mm & lt))] = (int32_t)vv;
    if (c == 2) a.big[ab + __popc(mb & lt)] = (int32_t)vv;
  }
}

// First candidate over the block (contains two __syncthreads).
__device__ __forceinline__ CKey block_first(CKey x, CKey *sk) {
  x = warp_first(x);
  if ((threadIdx.x & 31) == 0) sk[threadIdx.x >> 5] = x;
  __syncthreads();
  CKey r = sk[0];
#pragma unroll
  for (int i = 1; i < kGW; i++)
    if (ahead(sk[i], r)) r = sk[i];
  __syncthreads();
  return r;
}
// This warp's place among the block's counts (contains a __syncthreads before
// the read; the caller syncs before scnt is written again).
__device__ __forceinline__ int block_place(int c, int *scnt, int *tot) {
  const int wid = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) scnt[wid] = c;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int i = 0; i < kGW; i++) {
    const int x = scnt[i];
    before += i < wid ? x : 0;
    all += x;
  }
  *tot = all;
  return before;
}

// The same growth by a whole block, for vertices of many neighbours: one slice
// of the candidates per warp, filtered to a scratch row and packed back in
// order; the fence posts are the block's.  What is left goes to the first warp
// once it fits its shared memory.
template <int FLY>
__device__ int block_grow(const OA &a, int v, int32_t *B, GrowSmem &S, int *scnt, CKey *sk,
                          unsigned long long &tests) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const CKey none{INT_MIN, INT_MIN, INT_MAX};
  const int64_t e0 = a.rp[v], e1 = a.rp[v + 1], len = e1 - e0;
  int32_t *A = a.arena + e0;
  int64_t s0 = len * wid / kGW, s1 = len * (wid + 1) / kGW;
  CKey nb = none;
  int c = alive_of<FLY>(a, e0 + s0, e0 + s1, B + s0, nb);
  int cnt, j = 0;
  for (;;) {
    __syncwarp();
    const int at = block_place(c, scnt, &cnt);
    for (int i = lane; i < c; i += 32) A[at + i] = B[s0 + i];
    const CKey bk = block_first(nb, sk);
    if (cnt <= kNear) {
      int size = 0;
      if (wid == 0) size = warp_steps<FLY>(a, e1, A, cnt, bk, j, S.post[0], S.cand[0], tests);
      __syncthreads();
      return size;  // of the first warp
    }
    const int w = bk.id;
    if (threadIdx.x == 0) tests += (unsigned long long)cnt;
    const Fence f = set_fence(a, a.rp[w], a.rp[w + 1], &S.post[0][0], kGW * kNear, threadIdx.x, kGT);
    __syncthreads();
    s0 = (int64_t)cnt * wid / kGW;
    s1 = (int64_t)cnt * (wid + 1) / kGW;
    nb = none;
    c = filter<FLY>(a, f, w, A, (int)s0, (int)s1, B + s0, nb);
    j++;
    __syncthreads();  // A has been read
    // cnt + j <= deg(v): the member's slot lies past the packed candidates
    if (threadIdx.x == 0) a.arena[e1 - j] = w;
  }
}

// grow: the listed vertices of many neighbours by the first blocks (those with
// a scratch row), the others by warps, each taking the next as it frees up, so
// that a few long growths (the dense core's, every round) do not hold back the
// rest.  The longest chain of dependent loads is what a round takes: a step of
// a growth is the next member's row bounds, its fence posts, at most
// log2(length / 256) further entries of it and the kept candidates' keys.
// R-MAT scale 16, all rounds: 5.1 ms with 8 warps per SM, rows searched or
// merged in L2 and blocks only above 4,096 neighbours; 2.0 ms now.  Vertices of
// 513 .. 4,096 neighbours go to blocks while there are at most kMidPerBlock per
// block, when the longest growth decides, and to warps otherwise, when all of
// them do: whole order of scale 16 / 17 / 20 / 22 in 3.8 / 5.6 / 51 / 191 ms,
// always blocks 3.8 / 5.8 / 55 / 342, never blocks 4.8 / 7.7 / 50 / 185
// (before: 7.6 / 11.9 / 71 / 316; all on one machine, another has taken 3.6 / 5.0 /
// 43 / 218 since).
// FLY: candidates that a lane has in flight.  Four side by side, with 32 warps
// per SM, are right for the latency of long growths; where no vertex has more than
// kMidGrowMin neighbours and many are left, warps are what is short: one at a time
// with 48 warps per SM.  Whole order of 50,000 cliques of 20 in 5.0 ms (7.3 with four;
// 5.3 with 64 warps that searched the rows in L2), 50,000 of 50 in 39.9 (56.1;
// 43.9), G(10^6, 16) 2.47 (3.07; 2.74); 64 warps per SM spill (5.1, 39.8, 2.56).
// R-MAT scale 20, which has longer rows, would take 49 ms instead of 41.
template <int FLY, int BLOCKS>
__global__ void __launch_bounds__(kGT, BLOCKS) grow_kernel(OA a, int32_t *scratch, int64_t scratch_stride, int big_blocks) {
  __shared__ GrowSmem S;
  __shared__ CKey sk[kGW];
  __shared__ int scnt[kGW];
  __shared__ unsigned s_b;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const CKey none{INT_MIN, INT_MIN, INT_MAX};
  unsigned long long grows = 0, tests = 0;
  const unsigned nbig = *a.nbig, nmid = *a.nmid, nstale = *a.nstale;
  const bool mid_blocks = nmid <= kMidPerBlock * (unsigned)big_blocks;
  if ((int)blockIdx.x < big_blocks) {
    const unsigned total = nbig + (mid_blocks ? nmid : 0u);
    for (;;) {
      if (total == 0) break;
      if (threadIdx.x == 0) s_b = atomicAdd(a.take_big, 1u);
      __syncthreads();
      const unsigned b = s_b;
      __syncthreads();
      if (b >= total) break;
      const int v = b < nbig ? a.big[b] : a.big[a.n - 1 - (b - nbig)];
      const int size = block_grow<FLY>(a, v, scratch + blockIdx.x * scratch_stride, S, scnt, sk, tests);
      if (threadIdx.x == 0) {
        a.csize[v] = size;
        grows++;
      }
    }
  }
  const unsigned mids = mid_blocks ? 0u : nmid, total = mids + nstale;
  const unsigned chunk = total > 8u * kGW * gridDim.x ? (unsigned)kTake : 1u;
  for (;;) {
    unsigned idx = 0;
    if (lane == 0) idx = atomicAdd(a.take, chunk);
    idx = __shfl_sync(FULL, idx, 0);
    if (idx >= total) break;
    const unsigned end = min(total, idx + chunk);
    for (unsigned t = idx; t < end; t++) {
      const int v = t < mids ? a.big[a.n - 1 - t] : a.stale[t - mids];
      const int64_t e0 = a.rp[v], e1 = a.rp[v + 1];
      int32_t *cand = e1 - e0 <= kNear ? S.cand[wid] : a.arena + e0;
      CKey bk = none;
      __syncwarp();
      const int cnt = alive_of<FLY>(a, e0, e1, cand, bk);
      __syncwarp();
      const int size = warp_steps<FLY>(a, e1, cand, cnt, warp_first(bk), 0, S.post[wid], S.cand[wid], tests);
      if (lane == 0) {
        a.csize[v] = size;
        grows++;
      }
    }
  }
  if (lane == 0 && grows) atomicAdd((unsigned long long *)(a.ctl + 2), grows);
  if (lane == 0 && tests) atomicAdd((unsigned long long *)(a.ctl + 3), tests);
}

// scatter: every member takes the largest key of the cliques holding it
__global__ void scatter_kernel(OA a) {
  for (int64_t vv = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; vv < a.n; vv += (int64_t)gridDim.x * blockDim.x) {
    const int v = (int)vv;
    if (!a.alive[v]) continue;
    const int s = a.csize[v];
    const unsigned long long k = key_of(a, v, s);
    const int64_t e1 = a.rp[v + 1];
    atomicMax(a.bestkey + v, k);
    for (int i = 0; i < s - 1; i++) atomicMax(a.bestkey + a.arena[e1 - 1 - i], k);
  }
}

// accept: the clique holds its key at every member
__global__ void accept_kernel(OA a) {
  for (int64_t vv = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; vv < a.n; vv += (int64_t)gridDim.x * blockDim.x) {
    const int v = (int)vv;
    if (!a.alive[v]) continue;
    const int s = a.csize[v];
    const unsigned long long k = key_of(a, v, s);
    const int64_t e1 = a.rp[v + 1];
    bool ok = a.bestkey[v] == k;
    for (int i = 0; i < s - 1 && ok; i++) ok = a.bestkey[a.arena[e1 - 1 - i]] == k;
    if (ok) a.csize[v] = -s;
  }
}

struct AccF {
  const int32_t *csize;
  __device__ int64_t operator()(int64_t v) const {
    const int s = csize[v];
    return s < 0 ? ((int64_t)1 << 32) | (int64_t)(-s) : 0;
  }
};
struct AccG {
  int64_t *goff;
  __device__ void operator()(int64_t v, int64_t excl, int64_t val) const {
    if (val) goff[v] = excl;
  }
};

// place: warps take 32 vertices at a time and write each accepted clique's
// members ranked by degree (whole warp per clique)
__global__ void __launch_bounds__(kOT) place_kernel(OA a) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t placed = a.ctl[0], groups = a.ctl[1];
  for (int64_t base = gw * 32; base < a.n; base += nw * 32) {
    const int64_t vv = base + lane;
    const int sl = vv < a.n ? -a.csize[vv] : 0;
    unsigned m = __ballot_sync(FULL, sl > 0);
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      const int v = (int)base + src;
      const int s = __shfl_sync(FULL, sl, src);
      const int64_t packed = a.goff[v];
      const int64_t gi = groups + (packed >> 32), pos = placed + (packed & 0xffffffffLL);
      const int64_t e1 = a.rp[v + 1];
      // accepted cliques are disjoint sets of unplaced vertices, so they fit;
      // anything else is a broken invariant: report it, write nothing
      if (pos + s > a.n || gi >= a.n) {
        if (lane == 0) atomicExch(a.err, kDevCheck);
        continue;
      }
      for (int i = lane; i < s; i += 32) {
        const int x = i == 0 ? v : a.arena[e1 - i];
        const int64_t dx = a.rp[x + 1] - a.rp[x];
        int r = 0;
        for (int t = 0; t < s; t++) {
          const int y = t == 0 ? v : a.arena[e1 - t];
          const int64_t dy = a.rp[y + 1] - a.rp[y];
          r += (dy > dx || (dy == dx && y < x)) ? 1 : 0;
        }
        a.order[pos + r] = x;
      }
      __syncwarp();
      for (int i = lane; i < s; i += 32) a.alive[i == 0 ? v : a.arena[e1 - i]] = 0;
      if (lane == 0) {
        a.gstart[gi] = pos;
        a.ground[gi] = a.round;
        a.csize[v] = 0;
      }
    }
  }
}

// *look (host memory): this round and the vertices placed by then, in one word
__global__ void advance_kernel(int64_t *ctl, int32_t round, volatile unsigned long long *look) {
  const int64_t t = ctl[5];
  ctl[0] += t & 0xffffffffLL;
  ctl[1] += t >> 32;
  ctl[4] += t != 0;  // (a round that was queued after the last vertex was placed has none)
  ((unsigned *)(ctl + 6))[0] = 0u;  // the growers' lists, empty for the next round
  ((unsigned *)(ctl + 6))[1] = 0u;
  ((unsigned *)(ctl + 7))[0] = 0u;
  ((unsigned *)(ctl + 7))[1] = 0u;
  ((unsigned *)(ctl + 8))[0] = 0u;
  *look = ((unsigned long long)(round + 1) << 32) | (unsigned long long)ctl[0];
}

// a caller's tie rank must be a permutation of [0, n): seen[] starts at 0
__global__ void rank_check_kernel(int64_t n, const int32_t *rank, unsigned long long *seen, int32_t *bad) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int r = rank[v];
    if (r < 0 || r >= n || atomicExch(seen + r, 1ull) != 0ull) atomicExch(bad, 1);
  }
}

// ---- relabelling by an order and the gap cost ----

// pos[order[p]] = p; pos starts at -1 everywhere, a repeat or an id out of
// range sets *bad
__global__ void inverse_kernel(int64_t n, const int32_t *order, int32_t *pos, int32_t *bad) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const int v = order[p];
    if (v < 0 || v >= n || atomicCAS(pos + v, -1, (int)p) != -1) atomicExch(bad, 1);
  }
}

struct DegF {
  const int64_t *rp;
  const int32_t *order;
  __device__ int64_t operator()(int64_t p) const {
    const int v = order[p];
    return rp[v + 1] - rp[v];
  }
};
struct RowG {
  int64_t *nrp;
  __device__ void operator()(int64_t p, int64_t excl, int64_t) const { nrp[p] = excl; }
};

// One term of the gap cost: log2(1 + gap) in single precision (one rounding of
// 1 + gap, log2f within 1 ulp, so a relative error below 2^-22).
__device__ __forceinline__ float gap_term(int x, int prev, bool first) {
  const int gap = first ? abs(x - prev) : x - prev;
  return log2f((float)(gap + 1));
}

// The term in units of 2^-24: exact, since a term of a sorted row without
// repeats is log2f of at least 2, so above one half, and below 32; a repeat's
// is 0.  The integer sum is exact as well, and cheaper than doubles on this
// chip (gap cost of R-MAT scale 18: 345 us with doubles, 327 us with integers,
// everything else alike).
__device__ __forceinline__ int64_t gap_fixed(int x, int prev, bool first) {
  return (int64_t)__float2int_rn(gap_term(x, prev, first) * kGapUnit);
}

struct RA {
  int64_t n;
  const int64_t *rp;
  const int32_t *ci, *order, *pos;
  // the rows' place in nci: nrp[p] (relabelling), or nullptr: the old row's own
  // range (the gap cost, which needs memory for the long rows only)
  const int64_t *nrp;
  int32_t *nci;
  int32_t *mid, *big;  // rows of 33 .. kWarpSortMax entries, and of more
  unsigned *nmid;
  unsigned long long *nbig;
  unsigned long long *total;  // the gap cost's sum
};

// Bitonic sort of 32 R integers in a warp's registers; x[r] of lane l is item
// l R + r, so only the stages across lanes need shuffles.  The merges are a
// loop: unrolled over all sizes of R the code did not stay in the instruction
// cache (134 us instead of 70 for the rows of 33 .. 1,024 entries of R-MAT
// scale 18, 225 instead of 80 with the gap cost).
template <int R>
__device__ __forceinline__ void merge_lane(int (&x)[R], bool up) {
#pragma unroll
  for (int j = R / 2; j > 0; j >>= 1) {
#pragma unroll
    for (int r = 0; r < R; r++) {
      if (r & j) continue;
      const int lo = min(x[r], x[r | j]), hi = max(x[r], x[r | j]);
      x[r] = up ? lo : hi;
      x[r | j] = up ? hi : lo;
    }
  }
}
template <int R>
__device__ __forceinline__ void sort_regs(int (&x)[R]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 2; k < R; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
      for (int r = 0; r < R; r++) {
        if (r & j) continue;
        const int lo = min(x[r], x[r | j]), hi = max(x[r], x[r | j]);
        x[r] = (r & k) == 0 ? lo : hi;
        x[r | j] = (r & k) == 0 ? hi : lo;
      }
    }
  }
#pragma unroll 1
  for (int d = 1; d <= 32; d <<= 1) {  // sorts of d lanes' items
    const bool up = (lane & d) == 0;
#pragma unroll 1
    for (int j = d >> 1; j > 0; j >>= 1) {
      const bool keep_min = ((lane & j) == 0) == up;
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int y = __shfl_xor_sync(FULL, x[r], j);
        x[r] = keep_min ? min(x[r], y) : max(x[r], y);
      }
    }
    merge_lane<R>(x, up);
  }
}

// A row of 33 .. 32 R entries, sorted in registers and brought into row order
// through shared memory.
template <int R, bool GAP>
__device__ __forceinline__ int64_t sort_row(const RA &a, int64_t p, int64_t e0, int L, int64_t o0, int32_t *buf) {
  const int lane = threadIdx.x & 31;
  int x[R];
#pragma unroll
  for (int r = 0; r < R; r++) x[r] = 32 * r + lane < L ? a.ci[e0 + 32 * r + lane] : -1;
#pragma unroll
  for (int r = 0; r < R; r++) x[r] = x[r] >= 0 ? a.pos[x[r]] : INT_MAX;
  sort_regs<R>(x);
  __syncwarp();
#pragma unroll
  for (int r = 0; r < R; r++) {
    const int i = lane * R + r;
    buf[i + (i >> 5)] = x[r];
  }
  __syncwarp();
  int64_t s = 0;
  for (int i = lane; i < L; i += 32) {
    const int y = buf[i + (i >> 5)];
    if (GAP) s += gap_fixed(y, i ? buf[i - 1 + ((i - 1) >> 5)] : (int)p, i == 0);
    else a.nci[o0 + i] = y;
  }
  __syncwarp();
  return s;
}

__device__ __forceinline__ void block_add(int64_t s, unsigned long long *total) {
  __shared__ int64_t red[32];
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
  if (lane == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t t = 0;
    for (int w = 0; w < (int)blockDim.x / 32; w++) t += red[w];
    if (t != 0) atomicAdd(total, (unsigned long long)t);
  }
}

// The rows of at most 32 entries of the relabelled graph, written (GAP false) or
// only summed up for the gap cost: a warp holds the bounds of up to 32 rows,
// one per lane (rows far apart in the new order, which puts the long ones
// together), and sorts four at a time -- the chain entry -> position is what
// bounds them.  The longer rows are listed for the kernels below.  R-MAT scale
// 18 (7.2 M entries): 0.60 ms for rows up to 1,024 entries with one row per
// warp at a time and the sort in shared memory; now 30 us here and 70 us in
// mid_rows_kernel (with the gap cost instead of the writes 39 and 80 us; that
// was a pass of its own, 0.43 ms).  Both in one kernel took 183 us: the sort of
// 1,024 entries left the short rows 16 warps per SM.
template <bool GAP>
__global__ void __launch_bounds__(kOT) short_rows_kernel(RA a) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t s = 0;
  for (int64_t base = gw; base < a.n; base += nw * 32) {
    const int64_t mp = base + nw * lane;
    int64_t me0 = 0, mo0 = 0, ml = 0;
    if (mp < a.n) {
      const int v = a.order[mp];
      me0 = a.rp[v];
      ml = a.rp[v + 1] - me0;
      mo0 = a.nrp ? a.nrp[mp] : me0;
    }
    unsigned m = __ballot_sync(FULL, ml > 0 && ml <= 32);
    while (m) {
      int x[4], len[4], src[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        src[q] = m ? __ffs(m) - 1 : -1;
        m &= m - 1;  // (0 stays 0)
        const int64_t e0 = __shfl_sync(FULL, me0, max(src[q], 0));
        len[q] = __shfl_sync(FULL, (int)ml, max(src[q], 0));
        if (src[q] < 0) len[q] = 0;
        x[q] = lane < len[q] ? a.ci[e0 + lane] : -1;
      }
#pragma unroll
      for (int q = 0; q < 4; q++) x[q] = x[q] >= 0 ? a.pos[x[q]] : INT_MAX;
#pragma unroll
      for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
          const bool keep_min = ((lane & j) == 0) == ((lane & k) == 0);
#pragma unroll
          for (int q = 0; q < 4; q++) {
            const int y = __shfl_xor_sync(FULL, x[q], j);
            x[q] = keep_min ? min(x[q], y) : max(x[q], y);
          }
        }
#pragma unroll
      for (int q = 0; q < 4; q++) {
        if (GAP) {
          const int y = __shfl_up_sync(FULL, x[q], 1);
          if (lane < len[q]) s += gap_fixed(x[q], lane ? y : (int)(base + nw * src[q]), lane == 0);
        } else {
          const int64_t o0 = __shfl_sync(FULL, mo0, max(src[q], 0));
          if (lane < len[q]) a.nci[o0 + lane] = x[q];
        }
      }
    }
    // the longer ones are listed
    const unsigned mid = __ballot_sync(FULL, ml > 32 && ml <= kWarpSortMax);
    unsigned at = 0;
    if (lane == 0 && mid) at = atomicAdd(a.nmid, (unsigned)__popc(mid));
    at = __shfl_sync(FULL, at, 0);
    if (ml > 32) {
      if (ml <= kWarpSortMax) a.mid[at + __popc(mid & ((1u << lane) - 1u))] = (int32_t)mp;
      else a.big[atomicAdd(a.nbig, 1ull)] = (int32_t)mp;
    }
  }
  if (GAP) block_add(s, a.total);
}

// The listed rows of 33 to kWarpSortMax entries, a warp each.
template <bool GAP>
__global__ void __launch_bounds__(kOT, 3) mid_rows_kernel(RA a) {
  __shared__ int32_t sm[kOT / 32][kWarpSortMax + kWarpSortMax / 32];
  int32_t *buf = sm[threadIdx.x >> 5];
  const unsigned gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
  const unsigned total = *a.nmid;
  int64_t s = 0;
  for (unsigned t = gw; t < total; t += nw) {
    const int64_t p = a.mid[t];
    const int v = a.order[p];
    const int64_t e0 = a.rp[v], o0 = a.nrp ? a.nrp[p] : e0;
    const int L = (int)(a.rp[v + 1] - e0);
    if (L <= 64) s += sort_row<2, GAP>(a, p, e0, L, o0, buf);
    else if (L <= 128) s += sort_row<4, GAP>(a, p, e0, L, o0, buf);
    else if (L <= 256) s += sort_row<8, GAP>(a, p, e0, L, o0, buf);
    else if (L <= 512) s += sort_row<16, GAP>(a, p, e0, L, o0, buf);
    else s += sort_row<32, GAP>(a, p, e0, L, o0, buf);
  }
  if (GAP) block_add(s, a.total);
}

// compare-exchange stages (k, j >= jlo) of a bitonic sort over buf[0..P) by
// the whole block; global index base + i decides the direction
__device__ __forceinline__ void bitonic_stages(int32_t *buf, int P, int64_t base, int k, int jhi, int jlo) {
  for (int j = jhi; j >= jlo; j >>= 1) {
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
      const int l = i ^ j;
      if (l > i) {
        const int x = buf[i], y = buf[l];
        const bool up = ((base + i) & k) == 0;
        if ((x > y) == up) {
          buf[i] = y;
          buf[l] = x;
        }
      }
    }
    __syncthreads();
  }
}

// Row [e0, e0 + L) of new ids sorted to out by bitonic stages (row: the block's
// scratch row).
__device__ void bitonic_row(const RA &a, int64_t e0, int64_t L, int32_t *out, int32_t *sbuf, int32_t *row) {
  int64_t P = 1;
  while (P < L) P <<= 1;
  if (P <= kBlockSortMax) {
    for (int64_t i = threadIdx.x; i < P; i += blockDim.x) sbuf[i] = i < L ? a.pos[a.ci[e0 + i]] : INT_MAX;
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1) bitonic_stages(sbuf, (int)P, 0, k, k >> 1, 1);
    for (int64_t i = threadIdx.x; i < L; i += blockDim.x) out[i] = sbuf[i];
    __syncthreads();
    return;
  }
  for (int64_t i = threadIdx.x; i < P; i += blockDim.x) row[i] = i < L ? a.pos[a.ci[e0 + i]] : INT_MAX;
  __syncthreads();
  const int C = kBlockSortMax;
  // every stage with k <= C stays inside a chunk
  for (int64_t c = 0; c < P; c += C) {
    for (int i = threadIdx.x; i < C; i += blockDim.x) sbuf[i] = row[c + i];
    __syncthreads();
    for (int k = 2; k <= C; k <<= 1) bitonic_stages(sbuf, C, c, k, k >> 1, 1);
    for (int i = threadIdx.x; i < C; i += blockDim.x) row[c + i] = sbuf[i];
    __syncthreads();
  }
  for (int64_t k = 2 * (int64_t)C; k <= P; k <<= 1) {
    for (int64_t j = k >> 1; j >= C; j >>= 1) {
      for (int64_t i = threadIdx.x; i < P; i += blockDim.x) {
        const int64_t l = i ^ j;
        if (l > i) {
          const int x = row[i], y = row[l];
          const bool up = (i & k) == 0;
          if ((x > y) == up) {
            row[i] = y;
            row[l] = x;
          }
        }
      }
      __syncthreads();
    }
    for (int64_t c = 0; c < P; c += C) {
      for (int i = threadIdx.x; i < C; i += blockDim.x) sbuf[i] = row[c + i];
      __syncthreads();
      bitonic_stages(sbuf, C, c, (int)k, C >> 1, 1);
      for (int i = threadIdx.x; i < C; i += blockDim.x) row[c + i] = sbuf[i];
      __syncthreads();
    }
  }
  for (int64_t i = threadIdx.x; i < L; i += blockDim.x) out[i] = row[i];
  __syncthreads();
}

// Row [e0, e0 + L) of distinct new ids, sorted to out, by the bits of a window of
// 32 words new ids at a time: every entry sets its bit, and the set bits are
// written in order.  words of shared memory to clear and read instead of
// log^2 L passes over the row.  Returns whether all L entries were distinct
// (else what is in out does not count).
__device__ bool bitmap_row(const RA &a, int64_t e0, int64_t L, int32_t *out, unsigned *bm, int words, int *wsum) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t span = 32ll * words;
  const int per = ((words + kBigT / 32 - 1) / (kBigT / 32) + 31) & ~31;  // words per warp
  const int b0 = min(words, wid * per), b1 = min(words, b0 + per);
  int64_t done = 0;
  for (int64_t first = 0; first < a.n; first += span) {
    for (int i = threadIdx.x; i < words; i += kBigT) bm[i] = 0u;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < L; i += kBigT) {
      const int64_t x = a.pos[a.ci[e0 + i]] - first;
      if (x >= 0 && x < span) atomicOr(bm + (x >> 5), 1u << (x & 31));
    }
    __syncthreads();
    int c = 0;
    for (int i = b0 + lane; i < b1; i += 32) c += __popc(bm[i]);
    c = __reduce_add_sync(FULL, c);
    if (lane == 0) wsum[wid] = c;
    __syncthreads();
    int64_t at = done;
    for (int w = 0; w < kBigT / 32; w++) {
      at += w < wid ? wsum[w] : 0;
      done += wsum[w];
    }
    for (int i = b0; i < b1; i += 32) {
      unsigned y = i + lane < b1 ? bm[i + lane] : 0u;
      int incl = __popc(y);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int z = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += z;
      }
      int32_t *o = out + at + incl - __popc(y);
      while (y) {
        *o++ = (int32_t)(first + 32ll * (i + lane) + __ffs(y) - 1);
        y &= y - 1;
      }
      at += __shfl_sync(FULL, incl, 31);
    }
    __syncthreads();  // bm and wsum are free
  }
  return done == L;
}

// A block per long row: by bits where the words of all new ids are few for the
// row (at most kBitWords per entry: equal there, 0.80 and 0.85 ms for 600 rows
// of 4,100 entries among 4.2 M ids; at 64 words 0.61 against 0.45 ms, at 8 1.09
// against 1.35 ms); otherwise, and for rows with an entry twice, a bitonic sort
// in shared memory, above kBlockSortMax entries over a scratch row of the next
// power of two in global memory whose stages with j below kBlockSortMax run
// chunk by chunk in shared memory.  R-MAT scale 18: 0.50 ms with the bitonic
// sort alone, 0.07 ms now.
constexpr int kBitWords = 32;
template <bool GAP>
__global__ void __launch_bounds__(kBigT) long_rows_kernel(RA a, int words, int32_t *scratch, int64_t scratch_stride) {
  extern __shared__ int32_t sbuf[];
  __shared__ int wsum[kBigT / 32];
  const int64_t cnt = (int64_t)*a.nbig;
  int64_t s = 0;
  for (int64_t b = blockIdx.x; b < cnt; b += gridDim.x) {
    const int64_t p = a.big[b], e0 = a.rp[a.order[p]], L = a.rp[a.order[p] + 1] - e0;
    const int64_t o0 = a.nrp ? a.nrp[p] : e0;
    const bool bits = (a.n + 31) / 32 <= kBitWords * L;
    if (!bits || !bitmap_row(a, e0, L, a.nci + o0, (unsigned *)sbuf, words, wsum))
      bitonic_row(a, e0, L, a.nci + o0, sbuf, scratch + blockIdx.x * scratch_stride);
    if (GAP) {
      __syncthreads();
      const int32_t *row = a.nci + o0;
      for (int64_t i = threadIdx.x; i < L; i += kBigT)
        s += gap_fixed(row[i], i ? row[i - 1] : (int)p, i == 0);
    }
  }
  if (GAP) block_add(s, a.total);
}

// The gap cost of the graph as it is: sum over the entries of log2(1 + gap),
// the sum in double.
__global__ void __launch_bounds__(kOT) gap_kernel(int64_t n, const int64_t *nrp, const int32_t *nci, double *total) {
  __shared__ double red[kOT / 32];
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  double s = 0.0;
  for (int64_t p = gw; p < n; p += nw) {
    const int64_t e0 = nrp[p], e1 = nrp[p + 1];
    for (int64_t e = e0 + lane; e < e1; e += 32) s += (double)gap_term(nci[e], e == e0 ? (int)p : nci[e - 1], e == e0);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
  if (lane == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kOT / 32; w++) t += red[w];
    atomicAdd(total, t);
  }
}

int grid_of(mc_graph *g, int64_t items, int per_block, int per_sm) {
  const int64_t want = (items + per_block - 1) / per_block;
  return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)g->sm_count * per_sm));
}

}  // namespace

int clique_order(mc_graph *g, const int32_t *rank, int32_t *d_order, int64_t *d_gstart, int32_t *d_ground,
                 int64_t *groups_out, int32_t *rounds_out, int64_t *work_out) {
  const int64_t n = g->n;
  *groups_out = 0;
  *rounds_out = 0;
  if (n == 0) return MC_OK;
  if (!g->cores_valid) MC_TRY(launch_core_numbers(g, kDefaultSpinLimit));
  void *p;
  OA a{};
  a.n = n;
  a.rp = g->row_ptr;
  a.ci = g->col_idx;
  a.core = g->core;
  MC_TRY(ws_get(g, "co.alive", (size_t)n, &p));
  a.alive = (uint8_t *)p;
  MC_TRY(ws_get(g, "co.csize", (size_t)n * 4, &p));
  a.csize = (int32_t *)p;
  MC_TRY(ws_get(g, "co.arena", (size_t)std::max<int64_t>(g->nnz, 1) * 4, &p));
  a.arena = (int32_t *)p;
  MC_TRY(ws_get(g, "co.key", (size_t)n * 8, &p));
  a.bestkey = (unsigned long long *)p;
  MC_TRY(ws_get(g, "co.goff", (size_t)n * 8, &p));
  a.goff = (int64_t *)p;
  MC_TRY(ws_get(g, "co.ctl", 128, &p));
  a.ctl = (int64_t *)p;
  a.err = g->err;
  a.order = d_order;
  a.gstart = d_gstart;
  a.ground = d_ground;
  MC_CUDA_TRY(cudaMemsetAsync(a.ctl, 0, 128, g->stream));
  if (rank) {
    MC_TRY(ws_get(g, "co.rank", (size_t)n * 4, &p));
    MC_CUDA_TRY(cudaMemcpyAsync(p, rank, (size_t)n * 4, cudaMemcpyDefault, g->stream));
    a.rank = (const int32_t *)p;
    int32_t *bad = g->err + 9;
    MC_CUDA_TRY(cudaMemsetAsync(bad, 0, 4, g->stream));
    MC_CUDA_TRY(cudaMemsetAsync(a.bestkey, 0, (size_t)n * 8, g->stream));
    rank_check_kernel<<<grid_of(g, n, 256, 8), 256, 0, g->stream>>>(n, a.rank, a.bestkey, bad);
    g_launches++;
    MC_CUDA_TRY(cudaGetLastError());
    MC_CUDA_TRY(cudaMemcpyAsync(g->h_small, bad, 4, cudaMemcpyDeviceToHost, g->stream));
    MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
    if (*(int32_t *)g->h_small) return MC_ERR_ARG;
  }
  MC_TRY(ws_get(g, "co.kd", (size_t)n * 8, &p));
  a.kd = (const unsigned long long *)p;
  key_kernel<<<grid_of(g, n, 256, 8), 256, 0, g->stream>>>(n, a.rp, a.core, (unsigned long long *)p);
  g_launches++;
  MC_CUDA_TRY(cudaMemsetAsync(a.alive, 1, (size_t)n, g->stream));
  MC_CUDA_TRY(cudaMemsetAsync(a.csize, 0, (size_t)n * 4, g->stream));
  a.nbig = (unsigned *)(a.ctl + 6);
  a.take_big = a.nbig + 1;
  a.nstale = (unsigned *)(a.ctl + 7);
  a.take = a.nstale + 1;
  a.nmid = (unsigned *)(a.ctl + 8);
  MC_TRY(ws_get(g, "co.stale", (size_t)n * 4, &p));
  a.stale = (int32_t *)p;
  int32_t *scratch = nullptr;
  const int big_blocks = 2 * g->sm_count;
  const int64_t stride = std::max<int64_t>(g->max_degree, 1);
  const bool any_big = g->max_degree > kMidGrowMin;
  if (any_big) {
    MC_TRY(ws_get(g, "co.big", (size_t)n * 4, &p));
    a.big = (int32_t *)p;
    MC_TRY(ws_get(g, "co.bscratch", (size_t)big_blocks * stride * 4, &p));
    scratch = (int32_t *)p;
  }
  const int gw = grid_of(g, (n + 31) / 32, kOT / 32, 8), gt = grid_of(g, n, 256, 8);
  // A round is queued before the host looks at what the one before it placed, so
  // the GPU is not idle meanwhile, and one round at most is run in vain.  (Four
  // rounds queued per look: a star of 100,000 vertices 0.75 ms; two, two and then
  // four: R-MAT scale 12 4% slower than four.)
  volatile unsigned long long *look = (volatile unsigned long long *)((char *)g->h_small + 2560);
  *look = 0;
  int64_t placed = 0;
  unsigned long long last = 0;
  for (int32_t r = 0; placed < n; r++) {
    a.round = r;
    check_kernel<<<gt, 256, 0, g->stream>>>(a);
    if (!any_big && n - placed > kManyVertices)
      grow_kernel<1, 6><<<6 * g->sm_count, kGT, 0, g->stream>>>(a, scratch, stride, any_big ? big_blocks : 0);
    else
      grow_kernel<4, 4><<<4 * g->sm_count, kGT, 0, g->stream>>>(a, scratch, stride, any_big ? big_blocks : 0);
    scatter_kernel<<<gt, 256, 0, g->stream>>>(a);
    accept_kernel<<<gt, 256, 0, g->stream>>>(a);
    MC_CUDA_TRY(cudaGetLastError());
    MC_TRY(device_scan(g, n, AccF{a.csize}, AccG{a.goff}, a.ctl + 5, "co.scan"));
    place_kernel<<<gw, kOT, 0, g->stream>>>(a);
    advance_kernel<<<1, 1, 0, g->stream>>>(a.ctl, r, look);
    g_launches += 6;
    MC_CUDA_TRY(cudaGetLastError());
    if (r == 0) continue;
    // wait for round r - 1: for its word, or for the end of everything queued
    unsigned long long seen = *look;
    for (unsigned spins = 1; (int64_t)(seen >> 32) < r; spins++) {
      if ((spins & 1023) == 0) {
        const cudaError_t e = cudaStreamQuery(g->stream);
        if (e != cudaSuccess && e != cudaErrorNotReady) MC_CUDA_TRY(e);
        if (e == cudaSuccess && (int64_t)(*look >> 32) < r) return MC_ERR_DEVICE_CHECK;
      }
      seen = *look;
    }
    // every round places at least the clique of the largest key (the word may be a
    // later round's, and then the same at the next look)
    const int64_t now = (int64_t)(seen & 0xffffffffull);
    if (seen != last && (now <= placed || now > n)) {
      MC_TRY(check_device_error(g));
      return MC_ERR_DEVICE_CHECK;
    }
    placed = now;
    last = seen;
  }
  int64_t *h = (int64_t *)((char *)g->h_small + 2624);
  MC_CUDA_TRY(cudaMemcpyAsync(h, a.ctl, 6 * sizeof(int64_t), cudaMemcpyDeviceToHost, g->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
  *groups_out = h[1];
  *rounds_out = (int32_t)h[4];
  if (work_out) {
    work_out[0] = h[2];
    work_out[1] = h[3];
  }
  MC_CUDA_TRY(cudaMemcpyAsync(d_gstart + h[1], &g->n, sizeof(int64_t), cudaMemcpyHostToDevice, g->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
  return MC_OK;
}

// The order on the device and its inverse; refused unless it is a permutation.
static int load_order(mc_graph *g, const int32_t *order, RA &a) {
  const int64_t n = g->n;
  if (!g->cores_valid) MC_TRY(launch_core_numbers(g, kDefaultSpinLimit));  // sets max_degree
  void *p;
  MC_TRY(ws_get(g, "rl.order", (size_t)n * 4, &p));
  int32_t *d_order = (int32_t *)p;
  MC_CUDA_TRY(cudaMemcpyAsync(d_order, order, (size_t)n * 4, cudaMemcpyDefault, g->stream));
  MC_TRY(ws_get(g, "rl.pos", (size_t)n * 4, &p));
  int32_t *pos = (int32_t *)p;
  int32_t *bad = g->err + 10;
  MC_CUDA_TRY(cudaMemsetAsync(bad, 0, 4, g->stream));
  MC_CUDA_TRY(cudaMemsetAsync(pos, 0xff, (size_t)n * 4, g->stream));
  inverse_kernel<<<grid_of(g, n, 256, 8), 256, 0, g->stream>>>(n, d_order, pos, bad);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  MC_CUDA_TRY(cudaMemcpyAsync(g->h_small, bad, 4, cudaMemcpyDeviceToHost, g->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
  if (*(int32_t *)g->h_small) return MC_ERR_ARG;
  a.n = n;
  a.rp = g->row_ptr;
  a.ci = g->col_idx;
  a.order = d_order;
  a.pos = pos;
  return MC_OK;
}

// The rows of a (order, pos and where they go are set).
template <bool GAP>
static int launch_rows(mc_graph *g, RA a) {
  void *p;
  const bool any_mid = g->max_degree > 32, any_long = g->max_degree > kWarpSortMax;
  if (any_mid) {
    MC_TRY(ws_get(g, "rl.mid", 64 + (size_t)std::min<int64_t>(g->n, g->nnz / 33 + 1) * 4, &p));
    a.nbig = (unsigned long long *)p;
    a.nmid = (unsigned *)(a.nbig + 1);
    a.mid = (int32_t *)((char *)p + 64);
    MC_CUDA_TRY(cudaMemsetAsync(p, 0, 16, g->stream));
  }
  if (any_long) {
    MC_TRY(ws_get(g, "rl.big", (size_t)(g->nnz / kWarpSortMax + 1) * 4, &p));
    a.big = (int32_t *)p;
  }
  short_rows_kernel<GAP><<<grid_of(g, a.n * 8, kOT, 6), kOT, 0, g->stream>>>(a);
  g_launches++;
  if (any_mid) {
    mid_rows_kernel<GAP><<<grid_of(g, std::min<int64_t>(g->n, g->nnz / 33 + 1) * 32, kOT, 3), kOT, 0, g->stream>>>(a);
    g_launches++;
  }
  MC_CUDA_TRY(cudaGetLastError());
  if (any_long) {
    int64_t P = 1;
    while (P < g->max_degree) P <<= 1;
    int32_t *scratch = nullptr;
    int64_t stride = 0;
    int blocks = 2 * g->sm_count;
    if (P > kBlockSortMax) {  // the rows that may need a scratch row are megabytes
      stride = P;
      blocks = g->sm_count;
      MC_TRY(ws_get(g, "rl.scratch", (size_t)blocks * P * 4, &p));
      scratch = (int32_t *)p;
    }
    // the window: all new ids if they fit 192 KiB of bits
    const int words = (int)std::min<int64_t>((a.n + 31) / 32, 48 << 10);
    const int smem = std::max(words, kBlockSortMax) * 4;
    MC_CUDA_TRY(cudaFuncSetAttribute(long_rows_kernel<GAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    long_rows_kernel<GAP><<<blocks, kBigT, smem, g->stream>>>(a, words, scratch, stride);
    g_launches++;
    MC_CUDA_TRY(cudaGetLastError());
  }
  return MC_OK;
}

int relabel(mc_graph *g, const int32_t *order, int64_t *d_nrp, int32_t *d_nci) {
  if (g->n == 0) {
    MC_CUDA_TRY(cudaMemsetAsync(d_nrp, 0, sizeof(int64_t), g->stream));
    return MC_OK;
  }
  RA a{};
  MC_TRY(load_order(g, order, a));
  MC_TRY(device_scan(g, g->n, DegF{g->row_ptr, a.order}, RowG{d_nrp}, d_nrp + g->n, "rl.scan"));
  a.nrp = d_nrp;
  a.nci = d_nci;
  return launch_rows<false>(g, a);
}

int gap_bits_of(mc_graph *g, const int32_t *order, unsigned long long *d_total) {
  MC_CUDA_TRY(cudaMemsetAsync(d_total, 0, sizeof(*d_total), g->stream));
  if (g->n == 0) return MC_OK;
  RA a{};
  MC_TRY(load_order(g, order, a));
  if (g->max_degree > kWarpSortMax) {
    void *p;
    MC_TRY(ws_get(g, "rl.nci", (size_t)std::max<int64_t>(g->nnz, 1) * 4, &p));
    a.nci = (int32_t *)p;
  }
  a.total = d_total;
  return launch_rows<true>(g, a);
}

int gap_bits(mc_graph *g, const int64_t *d_nrp, const int32_t *d_nci, double *d_total) {
  MC_CUDA_TRY(cudaMemsetAsync(d_total, 0, sizeof(double), g->stream));
  if (g->n == 0) return MC_OK;
  gap_kernel<<<grid_of(g, g->n * 32, kOT, 8), kOT, 0, g->stream>>>(g->n, d_nrp, d_nci, d_total);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  return MC_OK;
}

}  // namespace mc
