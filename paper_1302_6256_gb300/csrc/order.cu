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
//           blocks those of more than 512 neighbours.
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
// Rounds repeat until every vertex is placed (four are queued before the host
// reads the placed count; a round after the last vertex changes nothing).  Cliques live in one arena laid out like the
// CSR: vertex v's candidates occupy the front of [rp[v], rp[v+1]) while it
// grows, and its members other than v end at the top of that range, so the
// arena is nnz int32 and needs no per-warp buffers or size limits.
//
// The gap cost relabels the graph by an order (new id = position), sorts
// every new row (bitonic networks: a warp in registers up to 32 entries, a
// warp in shared memory up to 1,024, a block in shared memory up to 16,384,
// a block over a global scratch row beyond), and sums log2(1 + gap) over the
// entries, the first gap of row p taken from p itself: 1 + gap rounded once
// to single precision, log2f (within 1 ulp), summed in double.
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
constexpr int64_t kBlockGrowMin = 512;  // neighbours above which a block grows the clique
constexpr int kTake = 4;                // listed vertices a warp takes at a time while there are many
constexpr int kNear = 256;              // candidates, and entries of a row, that a warp holds in shared memory
constexpr int kFly = 4;                 // entries or candidates a lane has in flight
constexpr int kRoundsPerSync = 4;       // rounds queued before the host looks at the placed count

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
                 // [6] the block grower's list length and next entry, [7] the warps' (two unsigned each)
  int64_t *goff;
  int32_t *order;
  int64_t *gstart;
  int32_t *ground;
  int32_t round;
  int32_t *err;
  int32_t *big;     // vertices for the block grower this round
  unsigned *nbig;
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
// kFly candidates side by side: a binary search of the fence posts in shared
// memory, then of the step - 1 entries behind one.  in and out may be the same
// list (a tile is read before anything of it is written).
__device__ __forceinline__ int filter(const OA &a, const Fence &f, int w, const int32_t *in, int i0, int i1,
                                      int32_t *out, CKey &nb) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int kept = 0;
  for (int base = i0; base < i1; base += 32 * kFly) {
    int x[kFly], lo[kFly], left[kFly];
    bool keep[kFly];
#pragma unroll
    for (int q = 0; q < kFly; q++) {
      const int i = base + 32 * q + lane;
      x[q] = i < i1 ? in[i] : -1;
      lo[q] = 0;  // posts <= x
    }
    for (int st = f.top; st > 0; st >>= 1) {
#pragma unroll
      for (int q = 0; q < kFly; q++)
        if (base + 32 * q < i1 && lo[q] + st <= f.posts && f.post[lo[q] + st - 1] <= x[q]) lo[q] += st;
    }
    int any = 0;
#pragma unroll
    for (int q = 0; q < kFly; q++) {
      keep[q] = lo[q] > 0 && f.post[lo[q] - 1] == x[q];
      const int at = (lo[q] - 1) * f.step + 1;
      left[q] = (lo[q] > 0 && !keep[q]) ? min(f.step - 1, f.len - at) : 0;
      lo[q] = at;
      any |= left[q];
    }
    while (any) {
      int y[kFly];
#pragma unroll
      for (int q = 0; q < kFly; q++) y[q] = left[q] ? f.row[lo[q] + (left[q] >> 1)] : 0;
      any = 0;
#pragma unroll
      for (int q = 0; q < kFly; q++) {
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
    for (int q = 0; q < kFly; q++) {
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
__device__ __forceinline__ int alive_of(const OA &a, int64_t s0, int64_t s1, int32_t *out, CKey &bk) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int cnt = 0;
  for (int64_t eb = s0; eb < s1; eb += 32 * kFly) {
    int u[kFly];
    bool ok[kFly];
#pragma unroll
    for (int q = 0; q < kFly; q++) {
      const int64_t e = eb + 32 * q + lane;
      u[q] = e < s1 ? a.ci[e] : -1;
    }
#pragma unroll
    for (int q = 0; q < kFly; q++) ok[q] = u[q] >= 0 && a.alive[u[q]] != 0;
#pragma unroll
    for (int q = 0; q < kFly; q++) {
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
      out = filter(a, f, w, cand, 0, cnt, cand, nb);
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
// ones that need a clique (warp-aggregated appends): vertices of more than
// kBlockGrowMin neighbours for the block grower, the rest for the warps
__global__ void check_kernel(OA a) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < a.n; base += stride) {
    const int64_t vv = base + lane;
    bool need = false, big = false;
    if (vv < a.n && a.alive[vv]) {
      a.bestkey[vv] = 0ull;
      need = needs_grow(a, (int)vv);
      big = need && a.rp[vv + 1] - a.rp[vv] > kBlockGrowMin;
    }
    const unsigned ms = __ballot_sync(FULL, need && !big), mb = __ballot_sync(FULL, big);
    unsigned at_s = 0, at_b = 0;
    if (lane == 0) {
      if (ms) at_s = atomicAdd(a.nstale, (unsigned)__popc(ms));
      if (mb) at_b = atomicAdd(a.nbig, (unsigned)__popc(mb));
    }
    at_s = __shfl_sync(FULL, at_s, 0);
    at_b = __shfl_sync(FULL, at_b, 0);
    if (need && !big) a.stale[at_s + __popc(ms & lt)] = (int32_t)vv;
    if (big) a.big[at_b + __popc(mb & lt)] = (int32_t)vv;
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
__device__ int block_grow(const OA &a, int v, int32_t *B, GrowSmem &S, int *scnt, CKey *sk,
                          unsigned long long &tests) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const CKey none{INT_MIN, INT_MIN, INT_MAX};
  const int64_t e0 = a.rp[v], e1 = a.rp[v + 1], len = e1 - e0;
  int32_t *A = a.arena + e0;
  int64_t s0 = len * wid / kGW, s1 = len * (wid + 1) / kGW;
  CKey nb = none;
  int c = alive_of(a, e0 + s0, e0 + s1, B + s0, nb);
  int cnt, j = 0;
  for (;;) {
    __syncwarp();
    const int at = block_place(c, scnt, &cnt);
    for (int i = lane; i < c; i += 32) A[at + i] = B[s0 + i];
    const CKey bk = block_first(nb, sk);
    if (cnt <= kNear) {
      int size = 0;
      if (wid == 0) size = warp_steps(a, e1, A, cnt, bk, j, S.post[0], S.cand[0], tests);
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
    c = filter(a, f, w, A, (int)s0, (int)s1, B + s0, nb);
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
// merged in L2 and blocks only above 4,096 neighbours; 2.0 ms now (blocks above
// 512; above 1,024 or 2,048: 3.56 or 3.95 ms per order instead of 3.70 at this
// scale, 5.83 or 5.87 instead of 5.51 at scale 17).
__global__ void __launch_bounds__(kGT, 4) grow_kernel(OA a, int32_t *scratch, int64_t scratch_stride, int big_blocks) {
  __shared__ GrowSmem S;
  __shared__ CKey sk[kGW];
  __shared__ int scnt[kGW];
  __shared__ unsigned s_b;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const CKey none{INT_MIN, INT_MIN, INT_MAX};
  unsigned long long grows = 0, tests = 0;
  const unsigned nbig = *a.nbig;
  if ((int)blockIdx.x < big_blocks && nbig) {
    for (;;) {
      if (threadIdx.x == 0) s_b = atomicAdd(a.take_big, 1u);
      __syncthreads();
      const unsigned b = s_b;
      __syncthreads();
      if (b >= nbig) break;
      const int v = a.big[b];
      const int size = block_grow(a, v, scratch + blockIdx.x * scratch_stride, S, scnt, sk, tests);
      if (threadIdx.x == 0) {
        a.csize[v] = size;
        grows++;
      }
    }
  }
  const unsigned total = *a.nstale;
  const unsigned chunk = total > 8u * kGW * gridDim.x ? (unsigned)kTake : 1u;
  for (;;) {
    unsigned idx = 0;
    if (lane == 0) idx = atomicAdd(a.take, chunk);
    idx = __shfl_sync(FULL, idx, 0);
    if (idx >= total) break;
    const unsigned end = min(total, idx + chunk);
    for (unsigned t = idx; t < end; t++) {
      const int v = a.stale[t];
      const int64_t e0 = a.rp[v], e1 = a.rp[v + 1];
      int32_t *cand = e1 - e0 <= kNear ? S.cand[wid] : a.arena + e0;
      CKey bk = none;
      __syncwarp();
      const int cnt = alive_of(a, e0, e1, cand, bk);
      __syncwarp();
      const int size = warp_steps(a, e1, cand, cnt, warp_first(bk), 0, S.post[wid], S.cand[wid], tests);
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

__global__ void advance_kernel(int64_t *ctl) {
  const int64_t t = ctl[5];
  ctl[0] += t & 0xffffffffLL;
  ctl[1] += t >> 32;
  ctl[4] += t != 0;  // (a round that was queued after the last vertex was placed has none)
  ((unsigned *)(ctl + 6))[0] = 0u;  // the growers' lists, empty for the next round
  ((unsigned *)(ctl + 6))[1] = 0u;
  ((unsigned *)(ctl + 7))[0] = 0u;
  ((unsigned *)(ctl + 7))[1] = 0u;
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

// a warp per new row: copy the old row through pos, sort rows of at most
// kWarpSortMax entries at once (bitonic; registers up to 32, shared memory
// above), and list the longer rows for the block sorter
__global__ void __launch_bounds__(kOT) fill_sort_kernel(int64_t n, const int64_t *rp, const int32_t *ci,
                                                        const int32_t *order, const int32_t *pos,
                                                        const int64_t *nrp, int32_t *nci, int32_t *big,
                                                        unsigned long long *nbig) {
  __shared__ int32_t sm[kOT / 32][kWarpSortMax];
  const int lane = threadIdx.x & 31;
  int32_t *buf = sm[threadIdx.x >> 5];
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p = gw; p < n; p += nw) {
    const int v = order[p];
    const int64_t e0 = rp[v], L = rp[v + 1] - e0, o0 = nrp[p];
    if (L > kWarpSortMax) {
      for (int64_t i = lane; i < L; i += 32) nci[o0 + i] = pos[ci[e0 + i]];
      if (lane == 0) big[atomicAdd(nbig, 1ull)] = (int32_t)p;
      continue;
    }
    if (L <= 32) {
      int x = lane < L ? pos[ci[e0 + lane]] : INT_MAX;
      // bitonic network over the 32 lanes
      for (int k = 2; k <= 32; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
          const int y = __shfl_xor_sync(FULL, x, j);
          const bool up = (lane & k) == 0, lower = (lane & j) == 0;
          x = (lower == up) ? min(x, y) : max(x, y);
        }
      if (lane < L) nci[o0 + lane] = x;
      continue;
    }
    int P = 64;
    while (P < L) P <<= 1;
    for (int i = lane; i < P; i += 32) buf[i] = i < L ? pos[ci[e0 + i]] : INT_MAX;
    __syncwarp();
    for (int k = 2; k <= P; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = lane; i < P; i += 32) {
          const int l = i ^ j;
          if (l > i) {
            const int x = buf[i], y = buf[l];
            const bool up = (i & k) == 0;
            if ((x > y) == up) {
              buf[i] = y;
              buf[l] = x;
            }
          }
        }
        __syncwarp();
      }
    for (int i = lane; i < L; i += 32) nci[o0 + i] = buf[i];
    __syncwarp();
  }
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

// a block per long row: shared memory up to kBlockSortMax entries, else a
// scratch row of the next power of two in global memory whose stages with
// j below kBlockSortMax run chunk by chunk in shared memory
__global__ void __launch_bounds__(kBigT) block_sort_kernel(const int64_t *nrp, int32_t *nci, const int32_t *big,
                                                           const unsigned long long *nbig, int32_t *scratch,
                                                           int64_t scratch_stride) {
  extern __shared__ int32_t sbuf[];
  const int64_t cnt = (int64_t)*nbig;
  for (int64_t b = blockIdx.x; b < cnt; b += gridDim.x) {
    const int64_t p = big[b];
    const int64_t o0 = nrp[p], L = nrp[p + 1] - o0;
    int64_t P = 1;
    while (P < L) P <<= 1;
    if (P <= kBlockSortMax) {
      for (int64_t i = threadIdx.x; i < P; i += blockDim.x) sbuf[i] = i < L ? nci[o0 + i] : INT_MAX;
      __syncthreads();
      for (int k = 2; k <= P; k <<= 1) bitonic_stages(sbuf, (int)P, 0, k, k >> 1, 1);
      for (int64_t i = threadIdx.x; i < L; i += blockDim.x) nci[o0 + i] = sbuf[i];
      __syncthreads();
      continue;
    }
    int32_t *row = scratch + blockIdx.x * scratch_stride;
    for (int64_t i = threadIdx.x; i < P; i += blockDim.x) row[i] = i < L ? nci[o0 + i] : INT_MAX;
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
    for (int64_t i = threadIdx.x; i < L; i += blockDim.x) nci[o0 + i] = row[i];
    __syncthreads();
  }
}

// sum over the entries of the relabelled graph of log2(1 + gap): each term
// in single precision (one rounding of 1 + gap, log2f within 1 ulp, so a
// relative error below 2^-22), the sum in double
__global__ void __launch_bounds__(kOT) gap_kernel(int64_t n, const int64_t *nrp, const int32_t *nci, double *total) {
  __shared__ double red[kOT / 32];
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  double s = 0.0;
  for (int64_t p = gw; p < n; p += nw) {
    const int64_t e0 = nrp[p], e1 = nrp[p + 1];
    for (int64_t e = e0 + lane; e < e1; e += 32) {
      const int64_t x = nci[e];
      const int64_t prev = e == e0 ? p : (int64_t)nci[e - 1];
      const int64_t gap = e == e0 ? (x > p ? x - p : p - x) : x - prev;
      s += (double)log2f((float)(gap + 1));
    }
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
  MC_TRY(ws_get(g, "co.ctl", 64, &p));
  a.ctl = (int64_t *)p;
  a.err = g->err;
  a.order = d_order;
  a.gstart = d_gstart;
  a.ground = d_ground;
  MC_CUDA_TRY(cudaMemsetAsync(a.ctl, 0, 64, g->stream));
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
  MC_TRY(ws_get(g, "co.stale", (size_t)n * 4, &p));
  a.stale = (int32_t *)p;
  int32_t *scratch = nullptr;
  const int big_blocks = 2 * g->sm_count, grow_blocks = 4 * g->sm_count;
  const int64_t stride = std::max<int64_t>(g->max_degree, 1);
  const bool any_big = g->max_degree > kBlockGrowMin;
  if (any_big) {
    MC_TRY(ws_get(g, "co.big", (size_t)n * 4, &p));
    a.big = (int32_t *)p;
    MC_TRY(ws_get(g, "co.bscratch", (size_t)big_blocks * stride * 4, &p));
    scratch = (int32_t *)p;
  }
  const int gw = grid_of(g, (n + 31) / 32, kOT / 32, 8), gt = grid_of(g, n, 256, 8);
  int64_t *h = (int64_t *)((char *)g->h_small + 2560);
  int64_t placed = 0;
  for (int32_t r = 0;;) {
    for (int i = 0; i < kRoundsPerSync; i++) {
      a.round = r++;
      check_kernel<<<gt, 256, 0, g->stream>>>(a);
      grow_kernel<<<grow_blocks, kGT, 0, g->stream>>>(a, scratch, stride, any_big ? big_blocks : 0);
      scatter_kernel<<<gt, 256, 0, g->stream>>>(a);
      accept_kernel<<<gt, 256, 0, g->stream>>>(a);
      MC_CUDA_TRY(cudaGetLastError());
      MC_TRY(device_scan(g, n, AccF{a.csize}, AccG{a.goff}, a.ctl + 5, "co.scan"));
      place_kernel<<<gw, kOT, 0, g->stream>>>(a);
      advance_kernel<<<1, 1, 0, g->stream>>>(a.ctl);
      g_launches += 6;
    }
    MC_CUDA_TRY(cudaGetLastError());
    MC_CUDA_TRY(cudaMemcpyAsync(h, a.ctl, 6 * sizeof(int64_t), cudaMemcpyDeviceToHost, g->stream));
    MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
    // every round places at least the clique of the largest key
    if (h[0] <= placed || h[0] > n) {
      MC_TRY(check_device_error(g));
      return MC_ERR_DEVICE_CHECK;
    }
    placed = h[0];
    if (placed == n) break;
  }
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

int relabel(mc_graph *g, const int32_t *order, int64_t *d_nrp, int32_t *d_nci) {
  const int64_t n = g->n;
  if (n == 0) {
    MC_CUDA_TRY(cudaMemsetAsync(d_nrp, 0, sizeof(int64_t), g->stream));
    return MC_OK;
  }
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
  MC_TRY(device_scan(g, n, DegF{g->row_ptr, d_order}, RowG{d_nrp}, d_nrp + n, "rl.scan"));
  MC_TRY(ws_get(g, "rl.big", (size_t)n * 4, &p));
  int32_t *big = (int32_t *)p;
  MC_TRY(ws_get(g, "rl.nbig", 8, &p));
  unsigned long long *nbig = (unsigned long long *)p;
  MC_CUDA_TRY(cudaMemsetAsync(nbig, 0, 8, g->stream));
  fill_sort_kernel<<<grid_of(g, n * 32, kOT, 8), kOT, 0, g->stream>>>(n, g->row_ptr, g->col_idx, d_order, pos,
                                                                        d_nrp, d_nci, big, nbig);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  if (g->max_degree > kWarpSortMax) {
    int64_t P = 1;
    while (P < g->max_degree) P <<= 1;
    const int blocks = g->sm_count;
    int32_t *scratch = nullptr;
    int64_t stride = 0;
    if (P > kBlockSortMax) {
      stride = P;
      MC_TRY(ws_get(g, "rl.scratch", (size_t)blocks * P * 4, &p));
      scratch = (int32_t *)p;
    }
    const int smem = kBlockSortMax * 4;
    MC_CUDA_TRY(cudaFuncSetAttribute(block_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    block_sort_kernel<<<blocks, kBigT, smem, g->stream>>>(d_nrp, d_nci, big, nbig, scratch, stride);
    g_launches++;
    MC_CUDA_TRY(cudaGetLastError());
  }
  return MC_OK;
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
