// Neighbourhood branch and bound: InitialBranch and Branch of Algorithm 2
// (Section 4.3), with the incumbent shared by every worker as soon as it
// changes (Section 4.5).
//
// For a root u of the oriented pruned graph the candidate set is
//   P = { w in N+(u) : K(w) >= omega }           (N_R(u) of Section 4.3)
// and the search looks for a clique larger than omega containing u:
//   1. |P| < omega                    -> return (degree bound, Fact 2 (3))
//   2. bitset adjacency of G[P]       (the small-graph adjacency matrix of
//      Section 4.4): gathered from bit rows of the top ranks, or each member's
//      later-neighbour row probed against a bitmap or hash table of P; that
//      sets the lower triangle (a later neighbour has a smaller index in P),
//      and transposes of 32 x 32 tiles fill the upper triangle
//   3. (omega-1)-core of G[P]: exactly the vertices with neighbourhood core
//      number K_N >= |H| when u is counted (lines 15-18 of InitialBranch;
//      the tight form of the test); fewer than omega left -> return
//   4. greedy colouring, L colours; 1 + L <= omega -> return (Fact 2 (1))
//   5. Branch({u}, P): depth-first, each node colours its candidates
//      greedily in index order (independent-set extraction with ballot and
//      popc over bit rows) and branches on the vertices whose colour can still
//      beat omega; a maximal clique larger than omega raises the incumbent.
// Bit positions are P sorted by decreasing rank, so "index order" colours the
// latest vertices of the degeneracy order first (the degeneracy-order
// colouring of InitialBranch) and every node uses the same natural order.
//
// Workers, split by the out-degree of the root (an upper bound on |P|):
//   warp class   |N+(u)| <= 128: one warp per root, matrix in shared memory;
//   block class  |N+(u)| <= 1024: one block per root, matrix in shared
//                memory; a 512-candidate and an 864-candidate layout at two
//                blocks per SM first (the second for dense rows only), then a
//                1,024-candidate launch for the roots they deferred; the
//                block's 16 warps share the root's search tree through a
//                shared-memory pool (a busy warp hands the shallowest untried
//                branch to an idle one);
//   big class    larger: as the block class with the matrix in global memory.
// Task queue: a root whose colouring leaves branches (in the warp class, one
// that a few nodes do not decide) copies its matrix to an
// arena and becomes one task of a GPU-wide ring; the task kernel searches
// tasks with single warps, which hand the untried branches of their
// shallowest level to the ring while other warps wait for work, so one hard
// neighbourhood spreads over the whole GPU.
// Every spin-wait is bounded; on timeout the device error word is set.
#include <algorithm>
#include <climits>

#include "mc_internal.cuh"

namespace mc {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kBW = 16;  // warps per block-class block
constexpr int kBT = kBW * 32;
constexpr int kSW = 8;   // warps per warp-class block
constexpr int kWarpCap = 128;
constexpr int kPoolCap = 16;

struct SA {
  const int64_t *orow;
  const int32_t *ocol, *ocore, *oold, *ogid;
  const int32_t *roots;
  const int64_t *nroots;    // device: number of roots in this class
  const int64_t *np_count;  // device: vertices of the pruned graph
  const uint32_t *dense;    // bit rows of the top ranks (null: none), see dense_rows_kernel
  int32_t dense_cap, dense_stride;  // ranks covered, words per row
  int32_t use_bitmap;       // look members up in a bitmap of the later ranks when they fit
  int32_t *best, *lock, *wit;
  const int64_t *voff;
  int32_t *err;
  long long spin;
  int32_t *next;            // root grab counter
  uint32_t *stack;          // per-warp DFS stacks
  int64_t stack_stride;     // words per warp stack
  int64_t small_stack;      // task kernel: offset of the compact search's levels in it
  uint32_t *gmat;           // per-block global matrix (big class)
  int64_t gmat_stride;      // words per block matrix
  int32_t neigh_cores;
  unsigned long long *counters;  // colored, branched, nodes, donations, entries
  // published roots: matrix + P list in a global arena, first-level tasks
  uint32_t *arena;
  long long arena_cap;           // words
  unsigned long long *arena_used;
  struct RootRec *recs;
  int32_t rec_cap;
  int32_t *nrec;
  uint32_t *tasks;               // kTaskWords words per task
  int32_t *ready;                // per ring slot: 2*lap free for lap's writer, 2*lap+1 written
  int32_t task_cap;              // ring slots (a power of two)
  int32_t *ntasks;               // positions taken (the queue's tail, monotonic)
  int32_t *task_next;            // tickets taken by the task kernel's warps (runs ahead of ntasks by the waiting ones)
  int32_t *pending;              // tasks published and not yet finished
  int32_t *progress;             // heartbeat: bumped every 256 Branch nodes, and at every one above the compact form
  uint32_t *sort;                // per-block room for a sorted matrix (roots searched in place)
  int64_t sort_stride;
  int32_t *overflow;             // roots too large for this launch's layout (or null)
  int64_t *noverflow;
  int32_t task_warps;            // warps of a task kernel that fills the chip
  int32_t offer_nodes;           // Branch nodes of a task between two looks for waiting warps
};

struct RootRec {
  int u, g, p, W, Ws, pad;
  long long off;  // arena word offset: matrix (p x Ws words), then the P list (p ints)
};
constexpr int kTaskWords = 2 + 64;  // root record, clique size, C bits, P bits (32 words each)
constexpr long long kArenaWords = 64ll << 20;  // 256 MB of published matrices
constexpr int kRecCap = 1 << 16;
constexpr int kTaskCap = 1 << 20;          // ring slots, 277 MB
constexpr size_t kCtrBytes = 96 * 8;       // counters and the queue's control words
// Default SA::offer_nodes.  R-MAT scale 17 (ef 12) / 18 (ef 12) / 20 (ef 16),
// task kernel: 4 nodes 3.2 / 4.2 / 11 ms, 6 nodes 2.8 / 3.3 / 6.5 ms, 16 nodes
// 3.5 / 4.4 / 5.7 ms, 64 nodes 8 / 10 / 12 ms: rare offers leave warps idle,
// frequent ones make tasks too small for their set-up (10-30 us).
constexpr int kOfferNodes = 8;
constexpr int kMidCap = 512;               // candidates of the two-blocks-per-SM block layout ...
// ... and of the one that serves dense rows only, also two blocks per SM: 102
// KB without the lookup structures.  At one block per SM (the 1,024 layout) its
// 7,850 roots at R-MAT scale 22 took 9.0 ms, now 5.5.
constexpr int kWideCap = 864;

template <int WPL>
struct Bits {
  uint32_t w[WPL];
};

template <int WPL>
__device__ __forceinline__ void bzero(Bits<WPL> &b) {
#pragma unroll
  for (int k = 0; k < WPL; k++) b.w[k] = 0;
}
template <int WPL>
__device__ __forceinline__ bool bany(const Bits<WPL> &b) {
  uint32_t x = 0;
#pragma unroll
  for (int k = 0; k < WPL; k++) x |= b.w[k];
  return __any_sync(FULL, x != 0);
}
template <int WPL>
__device__ __forceinline__ int bcount(const Bits<WPL> &b) {
  int c = 0;
#pragma unroll
  for (int k = 0; k < WPL; k++) c += __popc(b.w[k]);
  return dev::warp_sum(c);
}
template <int WPL>
__device__ __forceinline__ int blowest(const Bits<WPL> &b) {
  // one reduction: shorter than ballot, shuffle and two find-first-sets
  int v = INT_MAX;
#pragma unroll
  for (int k = WPL - 1; k >= 0; k--)
    if (b.w[k]) v = ((k * 32 + (int)(threadIdx.x & 31)) << 5) + __ffs(b.w[k]) - 1;
  v = __reduce_min_sync(FULL, v);
  return v == INT_MAX ? -1 : v;
}
template <int WPL>
__device__ __forceinline__ int bhighest(const Bits<WPL> &b) {
  int v = -1;
#pragma unroll
  for (int k = 0; k < WPL; k++)
    if (b.w[k]) v = ((k * 32 + (int)(threadIdx.x & 31)) << 5) + 31 - __clz(b.w[k]);
  return __reduce_max_sync(FULL, v);
}
template <int WPL>
__device__ __forceinline__ void bclear(Bits<WPL> &b, int v) {
  const int lane = threadIdx.x & 31, wi = v >> 5;
  const uint32_t m = ~(1u << (v & 31));
#pragma unroll
  for (int k = 0; k < WPL; k++)
    if ((wi >> 5) == k && (wi & 31) == lane) b.w[k] &= m;
}
template <int WPL>
__device__ __forceinline__ void bset(Bits<WPL> &b, int v) {
  const int lane = threadIdx.x & 31, wi = v >> 5;
  const uint32_t m = 1u << (v & 31);
#pragma unroll
  for (int k = 0; k < WPL; k++)
    if ((wi >> 5) == k && (wi & 31) == lane) b.w[k] |= m;
}
template <bool SM>
__device__ __forceinline__ uint32_t rw(const uint32_t *A, int64_t i) {
  if (SM) return A[i];
  return __ldcg(A + i);
}
// b &= row v  (words >= W are zero)
template <int WPL, bool SM>
__device__ __forceinline__ void band_row(Bits<WPL> &b, const uint32_t *A, int Ws, int W, int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < WPL; k++) {
    int w = k * 32 + lane;
    b.w[k] = (w < W) ? (b.w[k] & rw<SM>(A, (int64_t)v * Ws + w)) : 0u;
  }
}
template <int WPL, bool SM>
__device__ __forceinline__ void bandnot_row(Bits<WPL> &b, const uint32_t *A, int Ws, int W, int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < WPL; k++) {
    int w = k * 32 + lane;
    if (w < W) b.w[k] &= ~rw<SM>(A, (int64_t)v * Ws + w);
  }
}

// Greedy colouring of P in index order by independent-set extraction: colour
// class c takes, in index order, every remaining vertex with no neighbour
// already in class c.  (This is exactly the sequential greedy colouring.)
// B receives the vertices with colour > kmin: what is left after kmin
// classes, so the classes above are never made.
template <int WPL, bool SM>
__device__ void color_ise(const uint32_t *A, int Ws, int W, const Bits<WPL> &P, int kmin, Bits<WPL> &B) {
  B = P;
  for (int col = 1; col <= kmin && bany(B); col++) {
    Bits<WPL> Q = B;
    for (;;) {
      int v = blowest(Q);
      if (v < 0) break;
      bclear(Q, v);
      bclear(B, v);
      bandnot_row<WPL, SM>(Q, A, Ws, W, v);
    }
  }
}

__device__ __forceinline__ int read_best(const int32_t *best, int g) {
  int x = 0;
  if ((threadIdx.x & 31) == 0) x = *(const volatile int32_t *)(best + g);
  return __shfl_sync(FULL, x, 0);
}

__device__ __forceinline__ int hash_slot(int key, int mask) { return (int)(((unsigned)key * 2654435761u) >> 7) & mask; }

__device__ __forceinline__ int hash_find(const int *hk, const short *hv, int mask, int key) {
  int s = hash_slot(key, mask);
  for (;;) {
    int k = hk[s];
    if (k == key) return hv[s];
    if (k < 0) return -1;
    s = (s + 1) & mask;
  }
}

__device__ __forceinline__ void hash_insert(int *hk, short *hv, int mask, int key, int val) {
  int s = hash_slot(key, mask);
  for (;;) {
    int prev = atomicCAS(hk + s, -1, key);
    if (prev == -1 || prev == key) {
      hv[s] = (short)val;
      return;
    }
    s = (s + 1) & mask;
  }
}

// Index in P of a later-neighbour entry y, or -1 if y is not in P.
// Hash form: P's members in an open-addressing table.
struct HashLookup {
  const int *hk;
  const short *hv;
  int mask;
  __device__ __forceinline__ int operator()(int y) const { return hash_find(hk, hv, mask, y); }
};
// Bitmap form, for a root u whose later ranks (u, n') fit the block's
// bitmap: bit y - base marks a member of P, pre[w] counts the members in
// words before w, and P is sorted by decreasing id, so the member y has
// index p - 1 - (members below y).  Every entry a build reads is a later
// neighbour of a member, so y - base is never negative.
struct BitmapLookup {
  const uint32_t *bm;
  const uint16_t *pre;
  int base, p;
  __device__ __forceinline__ int operator()(int y) const {
    const int r = y - base;
    const uint32_t w = bm[r >> 5], bit = 1u << (r & 31);
    if (!(w & bit)) return -1;
    return p - 1 - ((int)pre[r >> 5] + __popc(w & (bit - 1u)));
  }
};
constexpr int kBitmapWords = 6144;  // later-rank window of the bitmap lookup: 196,608 ranks

// bitonic sort (descending) of a[0..npow2) in shared memory by `nthr`
// cooperating threads (thread index t); BLOCK selects the barrier.
template <bool BLOCK>
__device__ void bitonic_desc(int *a, int npow2, int t, int nthr) {
  for (int k = 2; k <= npow2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = t; i < npow2; i += nthr) {
        int ixj = i ^ j;
        if (ixj > i) {
          int x = a[i], y = a[ixj];
          bool desc = (i & k) == 0;
          if (desc ? (x < y) : (x > y)) {
            a[i] = y;
            a[ixj] = x;
          }
        }
      }
      if (BLOCK) __syncthreads(); else __syncwarp();
    }
  }
}

// Write the clique {u} + C (+ v) in original ids.  All lanes.
template <int WPL>
__device__ void write_clique(int32_t *base, const Bits<WPL> &C, int v, const int32_t *Pidx, const int32_t *oold,
                             int u) {
  const int lane = threadIdx.x & 31;
  Bits<WPL> X = C;
  if (v >= 0) bset(X, v);
  int cnt = 0;
#pragma unroll
  for (int k = 0; k < WPL; k++) cnt += __popc(X.w[k]);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += y;
  }
  int pos = 1 + incl - cnt;
#pragma unroll
  for (int k = 0; k < WPL; k++) {
    uint32_t x = X.w[k];
    while (x) {
      int b = __ffs(x) - 1;
      x &= x - 1;
      int idx = ((k * 32 + lane) << 5) + b;
      base[pos++] = oold[Pidx[idx]];
    }
  }
  if (lane == 0) base[0] = oold[u];
}

// A word of a stack level that lane 0 wrote (omega at colouring, the chosen
// vertex), read back by lane 0 and broadcast: the other lanes did not write
// it and must not act on a copy of their own.
__device__ __forceinline__ int level_word(const uint32_t *p) {
  int x = 0;
  if ((threadIdx.x & 31) == 0) x = (int)*p;
  return __shfl_sync(FULL, x, 0);
}

// Shared-memory task pool of a block worker.
template <int WPL>
struct Pool {
  int lock, count, idle, beat;
  int csize[kPoolCap];
  uint32_t C[kPoolCap][32 * WPL];
  uint32_t P[kPoolCap][32 * WPL];
};

template <int WPL>
__device__ bool pool_lock(Pool<WPL> *pl, int32_t *err, long long spin) {
  long long it = 0;
  while (atomicCAS(&pl->lock, 0, 1) != 0) {
    if (++it > spin) {
      atomicExch(err, kDevTimeout);
      return false;
    }
    __nanosleep(32);
  }
  __threadfence_block();
  return true;
}
template <int WPL>
__device__ void pool_unlock(Pool<WPL> *pl) {
  __threadfence_block();
  atomicExch(&pl->lock, 0);
}

struct Root {
  int u, g;
  const int32_t *Pidx;
  int p;  // |P|: rows of the root's matrix
};

// Take k consecutive queue positions, all or none; returns the first or -1.
// The queue is a ring of task_cap slots: positions are taken only while
// fewer than task_cap are taken and not yet handed out.  The positions count
// as pending from here on (the caller still holds a task, so the count cannot
// reach zero in between).  tries bounds the
// compare-and-swap attempts: thousands of warps offer branches at once when
// the queue runs dry, and one that loses goes on searching instead.
__device__ int reserve_tasks(const SA &a, int k, long long tries) {
  int cur = *(volatile int32_t *)a.ntasks;
  for (long long it = 0; it < tries; it++) {
    const int head = *(volatile int32_t *)a.task_next;
    if (cur - head + k > a.task_cap || cur > INT_MAX - k) return -1;
    const int prev = atomicCAS(a.ntasks, cur, cur + k);
    if (prev == cur) {
      atomicAdd(a.pending, k);
      return cur;
    }
    cur = prev;
  }
  return -1;
}

// One queue position for a root, before the task kernel starts; -1: the ring is
// full.  Nothing is handed out yet, so the first task_cap takers have theirs for
// good and a later one only takes back its own count.  (A compare-and-swap lets
// one of thousands of warps through per round trip to L2: 90,000 roots took 115
// ms.)
__device__ int reserve_root_task(const SA &a) {
  const int t = atomicAdd(a.ntasks, 1);
  if (t >= a.task_cap) {
    atomicSub(a.ntasks, 1);
    return -1;
  }
  atomicAdd(a.pending, 1);
  return t;
}

// Reserve arena room and a record for a root's matrix and P list.  Returns
// the record index (and the arena offset) or -1 without room.
__device__ int reserve_record(const SA &a, const Root &r, int Ws, long long *off_out) {
  const long long need = ((long long)r.p * Ws + r.p + 31) & ~31ll;  // records start on 128-byte lines
  // a root that does not fit takes nothing: smaller ones after it still may
  if ((long long)*(volatile unsigned long long *)a.arena_used + need > a.arena_cap) return -1;
  const long long off = (long long)atomicAdd(a.arena_used, (unsigned long long)need);
  if (off + need > a.arena_cap) return -1;
  const int rec = atomicAdd(a.nrec, 1);
  if (rec >= a.rec_cap) return -1;
  *off_out = off;
  return rec;
}

// Write the task at queue position t (clique size cs counting u, 0 =
// empty; clique bits C; candidates P) and mark its slot written.  Position
// t uses slot t mod task_cap in lap t / task_cap: the slot's word counts
// 2*lap when the previous lap's task has been read (its reader already
// holds it, since t was reserved after that position was handed out) and
// 2*lap+1 once this task is written.  Warp-collective.
__device__ void write_task(const SA &a, int t, int rec, int cs, const Bits<1> &C, const Bits<1> &P) {
  const int lane = threadIdx.x & 31;
  const int slot = t & (a.task_cap - 1);
  const int lap2 = 2 * (t / a.task_cap);
  if (lane == 0) {
    long long w = 0;
    while (*(volatile int32_t *)(a.ready + slot) != lap2) {
      if (++w > a.spin) {
        atomicExch(a.err, kDevTimeout);
        break;
      }
      __nanosleep(32);
    }
  }
  __syncwarp();
  __threadfence();
  uint32_t *tk = a.tasks + (int64_t)slot * kTaskWords;
  if (lane == 0) {
    tk[0] = (uint32_t)rec;
    tk[1] = (uint32_t)cs;
  }
  tk[2 + lane] = C.w[0];
  tk[34 + lane] = P.w[0];
  __syncwarp();
  __threadfence();
  if (lane == 0) atomicExch(a.ready + slot, lap2 + 1);
}

// The branch x of a node with clique Cl (csl vertices with u) and candidates
// Pl (x and its earlier siblings already removed) as task slot t; the task
// is empty when x's subproblem is decided at once (raising the incumbent if
// {u} + Cl + x is a larger maximal clique).
__device__ void emit_task(const SA &a, const Root &r, const uint32_t *A, int Ws, int W, int rec, int t,
                          const Bits<1> &Cl, int csl, const Bits<1> &Pl, int x) {
  Bits<1> TP = Pl;
  band_row<1, false>(TP, A, Ws, W, x);
  const int om = read_best(a.best, r.g);
  int cs = csl + 1;
  if (!bany(TP)) {
    if (csl + 1 > om) {
      const Bits<1> Cc = Cl;
      dev::raise_incumbent(a.best, a.lock, a.wit, a.voff, r.g, csl + 1, a.err, a.spin,
                           [&](int, int32_t *base) { write_clique<1>(base, Cc, x, r.Pidx, a.oold, r.u); });
    }
    cs = 0;
  } else if (csl + 1 + bcount(TP) <= om) {
    cs = 0;
  }
  Bits<1> Cx = Cl;
  bset(Cx, x);
  write_task(a, t, rec, cs, Cx, TP);
}

// Depth-first Branch from one level (csize0 = |C| including the root u).
// Stack levels above the start hold (P, B, omega-at-colouring, chosen).
// If `pool` is not null, untried branches are handed to idle warps.  After
// `limit` nodes it stops: true if the search is done, else `rest` holds the
// candidates of the first level without the branches that are.
template <int WPL, bool SM>
__device__ bool dfs(const SA &a, const Root &r, const uint32_t *A, int Ws, int W, uint32_t *stk, int csize0,
                    Bits<WPL> P, Bits<WPL> B, Bits<WPL> C, int wat, Pool<WPL> *pool, unsigned long long &nodes,
                    unsigned long long &donations, long long limit = LLONG_MAX, Bits<WPL> *rest = nullptr) {
  const int lane = threadIdx.x & 31;
  const int stride = 64 * WPL + 2;
  int d = 0, csize = csize0;
  long long spent = 0;
  for (;;) {
    if (__shfl_sync(FULL, lane == 0 ? *(volatile int32_t *)a.err : 0, 0)) return true;
    int om = read_best(a.best, r.g);
    if (om > wat) {
      color_ise<WPL, SM>(A, Ws, W, P, om - csize, B);
      wat = om;
    }
    int v = bhighest(B);
    if (v < 0) {
      if (d == 0) return true;
      d--;
      uint32_t *lv = stk + (int64_t)d * stride;
#pragma unroll
      for (int k = 0; k < WPL; k++) {
        P.w[k] = lv[k * 32 + lane];
        B.w[k] = lv[32 * WPL + k * 32 + lane];
      }
      wat = level_word(lv + 64 * WPL);
      const int ch = level_word(lv + 64 * WPL + 1);
      bclear(C, ch);
      csize--;
      continue;
    }
    if (spent >= limit) {
      *rest = P;
      if (d > 0) {
#pragma unroll
        for (int k = 0; k < WPL; k++) rest->w[k] = stk[k * 32 + lane];
        bset(*rest, level_word(stk + 64 * WPL + 1));
      }
      return false;
    }
    bclear(B, v);
    bclear(P, v);
    Bits<WPL> NP = P;
    band_row<WPL, SM>(NP, A, Ws, W, v);
    nodes++;
    spent++;
    if (lane == 0 && a.progress && (spent & 255) == 0) atomicAdd(a.progress, 1);
    if (!bany(NP)) {
      if (csize + 1 > om) {
        const Bits<WPL> Cc = C;
        dev::raise_incumbent(a.best, a.lock, a.wit, a.voff, r.g, csize + 1, a.err, a.spin,
                             [&](int, int32_t *base) { write_clique<WPL>(base, Cc, v, r.Pidx, a.oold, r.u); });
      }
      continue;
    }
    if (csize + 1 + bcount(NP) <= om) continue;
    Bits<WPL> NB;
    color_ise<WPL, SM>(A, Ws, W, NP, om - csize - 1, NB);
    if (!bany(NB)) continue;  // csize + 1 + L <= omega
    // descend: save this level
    uint32_t *lv = stk + (int64_t)d * stride;
#pragma unroll
    for (int k = 0; k < WPL; k++) {
      lv[k * 32 + lane] = P.w[k];
      lv[32 * WPL + k * 32 + lane] = B.w[k];
    }
    if (lane == 0) {
      lv[64 * WPL] = (uint32_t)wat;
      lv[64 * WPL + 1] = (uint32_t)v;
    }
    d++;
    bset(C, v);
    csize++;
    P = NP;
    B = NB;
    wat = om;

    // hand the shallowest untried branch to an idle warp of the block
    if (pool) {
      if (lane == 0) atomicAdd(&pool->beat, 1);  // progress signal for waiting warps
      int hungry = 0;
      if (lane == 0) {
        int idle = *(volatile int *)&pool->idle, cnt = *(volatile int *)&pool->count;
        hungry = idle > 0 && cnt < idle && cnt < kPoolCap;
      }
      hungry = __shfl_sync(FULL, hungry, 0);
      if (hungry) {
        __syncwarp();
        // shallowest stored level with an untried branch (levels 0..d-1 are in memory)
        int lev = -1;
        Bits<WPL> Bl, Pl;
        for (int l = 0; l < d; l++) {
          uint32_t *q = stk + (int64_t)l * stride;
#pragma unroll
          for (int k = 0; k < WPL; k++) Bl.w[k] = q[32 * WPL + k * 32 + lane];
          if (bany(Bl)) {
            lev = l;
            break;
          }
        }
        if (lev >= 0) {
          uint32_t *q = stk + (int64_t)lev * stride;
#pragma unroll
          for (int k = 0; k < WPL; k++) Pl.w[k] = q[k * 32 + lane];
          int x = bhighest(Bl);
          bclear(Bl, x);
          bclear(Pl, x);
#pragma unroll
          for (int k = 0; k < WPL; k++) {
            q[k * 32 + lane] = Pl.w[k];
            q[32 * WPL + k * 32 + lane] = Bl.w[k];
          }
          // clique at level lev: C minus the vertices chosen at levels >= lev
          Bits<WPL> Cl = C;
          for (int l = lev; l < d; l++) bclear(Cl, level_word(stk + (int64_t)l * stride + 64 * WPL + 1));
          bset(Cl, x);
          Bits<WPL> TP = Pl;
          band_row<WPL, SM>(TP, A, Ws, W, x);
          int tcs = csize0 + lev + 1;
          int om2 = read_best(a.best, r.g);
          if (bany(TP) && tcs + bcount(TP) > om2) {
            int ok = 0;
            if (lane == 0) {
              if (pool_lock(pool, a.err, a.spin)) {
                if (pool->count < kPoolCap) ok = 1 + pool->count++;
                else pool_unlock(pool);
              }
            }
            ok = __shfl_sync(FULL, ok, 0);
            if (ok) {
              int slot = ok - 1;
#pragma unroll
              for (int k = 0; k < WPL; k++) {
                pool->C[slot][k * 32 + lane] = Cl.w[k];
                pool->P[slot][k * 32 + lane] = TP.w[k];
              }
              // a *_sync exchange does not reconverge the warp: every lane's
              // words must be written before lane 0 releases the pool
              __syncwarp();
              if (lane == 0) {
                pool->csize[slot] = tcs;
                pool_unlock(pool);
              }
              donations++;
            } else {
              // pool full: search the branch here, later, by restoring it
              bset(Bl, x);
              bset(Pl, x);
#pragma unroll
              for (int k = 0; k < WPL; k++) {
                q[k * 32 + lane] = Pl.w[k];
                q[32 * WPL + k * 32 + lane] = Bl.w[k];
              }
            }
          } else if (!bany(TP) && tcs > om2) {
            // nothing left to add: {u} + Cl is maximal and beats the incumbent
            const Bits<WPL> Cc = Cl;
            dev::raise_incumbent(a.best, a.lock, a.wit, a.voff, r.g, tcs, a.err, a.spin,
                                 [&](int, int32_t *base) { write_clique<WPL>(base, Cc, -1, r.Pidx, a.oold, r.u); });
          }
        }
        __syncwarp();
      }
    }
  }
}

// Load P = {w in N+(u) : K(w) >= om} into Pidx (unsorted).  Cooperative over
// nthr threads; *cnt is a shared counter (pre-zeroed).  Reads rows as int4.
__device__ __forceinline__ void load_P(const SA &a, int u, int om, int *Pidx, int cap, int *cnt, int t, int nthr) {
  const int64_t e0 = a.orow[u], e1 = a.orow[u + 1];
  const int4 *row = reinterpret_cast<const int4 *>(a.ocol + e0);
  const int64_t nq = (e1 - e0) >> 2;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  // whole warps step together (t - lane is the warp's first index), so the
  // members a warp finds take one shared atomic per ballot
  for (int64_t q0 = t - lane; q0 < nq; q0 += nthr) {
    const int64_t q = q0 + lane;
    int ys[4] = {-1, -1, -1, -1};
    if (q < nq) {
      const int4 y = __ldg(row + q);
      ys[0] = y.x;
      ys[1] = y.y;
      ys[2] = y.z;
      ys[3] = y.w;
    }
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const bool keep = ys[j] >= 0 && __ldg(a.ocore + ys[j]) >= om;
      const unsigned m = __ballot_sync(FULL, keep);
      int base = 0;
      if (lane == 0 && m) base = atomicAdd(cnt, __popc(m));
      base = __shfl_sync(FULL, base, 0);
      if (keep) {
        const int p = base + __popc(m & lt);
        if (p < cap) Pidx[p] = ys[j];
      }
    }
  }
}

// Matrix rows of P: for each member x (index i), every later neighbour y of x
// that is in P (index j) sets bits (i, j) and (j, i).  The lanes of a warp
// form four groups of eight, each walking a different member's row, with two
// int4 loads per lane in flight, so a warp keeps eight rows' loads in the
// memory system instead of one.  scanned: the row entries a lane's group read
// (Fact 3's work) are added by the group's first lane.
template <class Lookup>
__device__ __forceinline__ void build_rows(const SA &a, const int *Pidx, int p, const Lookup &find, uint32_t *A, int Ws,
                                           int wid, int nw, unsigned long long &scanned, int *dyn = nullptr) {
  const int lane = threadIdx.x & 31;
  const int grp = lane >> 3, gl = lane & 7;
  // groups of 4 rows: statically wid, wid + nw, ...; or, with a shared
  // counter (dyn, zero before the call), taken by each warp as it frees up,
  // so rows of uneven length do not leave warps waiting at the next barrier
  int i0 = wid * 4;
  if (dyn) {
    if (lane == 0) i0 = atomicAdd(dyn, 4);
    i0 = __shfl_sync(FULL, i0, 0);
  }
  for (; i0 < p;) {
    const int i = i0 + grp;
    int64_t e0 = 0, e1 = 0;
    if (i < p) {
      const int x = Pidx[i];
      e0 = a.orow[x];
      e1 = a.orow[x + 1];
    }
    const int4 *row = reinterpret_cast<const int4 *>(a.ocol + e0);
    const int nq = (int)((e1 - e0) >> 2);
    const int nqmax = max(max(__shfl_sync(FULL, nq, 0), __shfl_sync(FULL, nq, 8)),
                          max(__shfl_sync(FULL, nq, 16), __shfl_sync(FULL, nq, 24)));
    if (gl == 0) scanned += 4ull * (unsigned long long)nq;
    for (int q0 = gl; q0 < nqmax; q0 += 16) {
      int4 ys[2];
#pragma unroll
      for (int u = 0; u < 2; u++) {
        const int q = q0 + 8 * u;
        ys[u] = (q < nq) ? __ldg(row + q) : make_int4(-1, -1, -1, -1);
      }
#pragma unroll
      for (int u = 0; u < 2; u++) {
        const int yy[4] = {ys[u].x, ys[u].y, ys[u].z, ys[u].w};
#pragma unroll
        for (int j = 0; j < 4; j++) {
          if (yy[j] < 0) continue;
          int b = find(yy[j]);
          if (b >= 0) atomicOr(A + (int64_t)i * Ws + (b >> 5), 1u << (b & 31));
        }
      }
    }
    if (dyn) {
      if (lane == 0) i0 = atomicAdd(dyn, 4);
      i0 = __shfl_sync(FULL, i0, 0);
    } else {
      i0 += nw * 4;
    }
  }
}

// 32 x 32 bit transpose across a warp: lane r holds row r (bit c = column
// c); returns row c of the transpose for lane c (bit r = row r's bit c).
// Five exchange stages swap ever smaller off-diagonal blocks: in the stage
// of width j, the lane with bit j clear trades its upper j-bit halves for its
// partner's lower ones.
__device__ __forceinline__ uint32_t transpose32(uint32_t x) {
  const int lane = threadIdx.x & 31;
  uint32_t m = 0x0000ffffu;
#pragma unroll
  for (int j = 16; j != 0; j >>= 1, m ^= (m << j)) {
    const uint32_t y = __shfl_xor_sync(FULL, x, j);
    x = (lane & j) ? (((y >> j) & m) | (x & ~m)) : ((x & m) | ((y & m) << j));
  }
  return x;
}

// Complete the adjacency matrix from its lower triangle.  build_rows sets
// bit (i, b) for every edge of G[P] with b < i (a later neighbour has a
// higher rank, hence a smaller index in P); the 32 x 32 tiles on and below
// the diagonal are transposed with warp ballots and OR-ed into their mirror
// tiles.  A tile's reads (lower words) and writes (upper words, or the same
// diagonal tile after all its rows were read) never overlap another tile's.
template <bool SM>
__device__ void symmetrize(uint32_t *A, int Ws, int W, int p, int wid, int nw) {
  const int lane = threadIdx.x & 31;
  const int tiles = W * (W + 1) / 2;
  for (int t = wid; t < tiles; t += nw) {
    // tile t = (I, J) with J <= I, row-major over the lower triangle
    int I = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
    while (I * (I + 1) / 2 > t) I--;
    while ((I + 1) * (I + 2) / 2 <= t) I++;
    const int J = t - I * (I + 1) / 2;
    const int r = 32 * I + lane;
    const uint32_t x = (r < p) ? rw<SM>(A, (int64_t)r * Ws + J) : 0u;
    const uint32_t col = transpose32(x);
    const int rt = 32 * J + lane;
    if (rt < p) {
      const int64_t at = (int64_t)rt * Ws + I;
      A[at] = (I == J) ? (x | col) : (rw<SM>(A, at) | col);
    }
  }
}

// Arena room, record and queue position (*t_out, -1: none) of a root of m
// candidates; the record, or -1.  One thread.
__device__ int open_record(const SA &a, const Root &r, int m, int *t_out) {
  const Root rm{r.u, r.g, r.Pidx, m};
  const int Wsm = ((m + 31) >> 5) | 1;
  long long off = 0;
  *t_out = -1;
  const int rec = reserve_record(a, rm, Wsm, &off);
  if (rec < 0) return -1;
  *t_out = reserve_root_task(a);
  RootRec rr;
  rr.u = r.u;
  rr.g = r.g;
  rr.p = m;
  rr.W = (m + 31) >> 5;
  rr.Ws = Wsm;
  rr.pad = 0;
  rr.off = off;
  a.recs[rec] = rr;
  return rec;
}
__device__ __forceinline__ uint32_t first_bits(int m) {  // this lane's word of the set {0 .. m-1}
  const int lane = threadIdx.x & 31;
  return m >= 32 * (lane + 1) ? FULL : (m > 32 * lane ? (1u << (m - 32 * lane)) - 1u : 0u);
}
// Row i of a matrix in another order (word w: a ballot over new positions 32w
// .. 32w+31); keys hold the complement of the old index in their low half.
__device__ __forceinline__ uint32_t permuted_row(const uint32_t *A, int Ws, const uint32_t *keys, int m, int i) {
  const int lane = threadIdx.x & 31;
  const uint32_t *row = A + (int64_t)(0xffff - (int)(keys[i] & 0xffffu)) * Ws;
  uint32_t mine = 0;
  for (int w = 0; w < (m + 31) >> 5; w++) {
    const int j = 32 * w + lane;
    const int at = j < m ? 0xffff - (int)(keys[j] & 0xffffu) : 0;
    const unsigned word = __ballot_sync(FULL, j < m && ((row[at >> 5] >> (at & 31)) & 1u));
    if (lane == w) mine = word;
  }
  return mine;
}

// The candidates of a warp's root (at most kWarpCap) in bits al, in
// minimum-width order (see width_keys); returns how many.  keys: kWarpCap
// words.
__device__ int width_keys_warp(const Root &r, const uint32_t *A, int Ws, int W, const uint32_t *al, uint32_t *keys) {
  const int lane = threadIdx.x & 31;
  int deg[4], m = 0;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int i = 32 * q + lane;
    deg[q] = INT_MAX;
    keys[i] = 0;
    if (q >= W) continue;
    m += __popc(al[q]);
    if (i < r.p && ((al[q] >> lane) & 1u)) {
      deg[q] = 0;
      for (int w = 0; w < W; w++) deg[q] += __popc(A[i * Ws + w] & al[w]);
    }
  }
  int left = m;
  for (uint32_t step = 1; left > 0; step++) {
    const int lo = __reduce_min_sync(FULL, min(min(deg[0], deg[1]), min(deg[2], deg[3])));
    unsigned out[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      out[q] = __ballot_sync(FULL, deg[q] == lo);
      if (deg[q] == lo) {
        keys[32 * q + lane] = (step << 16) | (uint32_t)(0xffff - (32 * q + lane));
        deg[q] = INT_MAX;
      }
      left -= __popc(out[q]);
    }
#pragma unroll
    for (int w = 0; w < 4; w++)
      if (out[w]) {
#pragma unroll
        for (int q = 0; q < 4; q++)
          if (deg[q] != INT_MAX) deg[q] -= __popc(A[(32 * q + lane) * Ws + w] & out[w]);
      }
  }
  __syncwarp();
  bitonic_desc<false>((int *)keys, kWarpCap, lane, 32);
  return m;
}

// The matrix and P list of those m candidates in that order, to dm (m rows of
// Wsm words) and dp, by a warp.
__device__ __forceinline__ void permute_rows_warp(const Root &r, const uint32_t *A, int Ws, const uint32_t *keys,
                                                  int m, uint32_t *dm, int Wsm, int *dp) {
  const int lane = threadIdx.x & 31;
  for (int i = 0; i < m; i++) {
    const uint32_t x = permuted_row(A, Ws, keys, m, i);
    if (lane < Wsm) dm[i * Wsm + lane] = x;
  }
  for (int i = lane; i < m; i += 32) dp[i] = r.Pidx[0xffff - (int)(keys[i] & 0xffffu)];
  __syncwarp();
}

// A warp's root as a task, its matrix copied to the arena once.  False,
// publishing nothing, without room for the record or in the queue.
__device__ bool publish_warp(const SA &a, const Root &r, const uint32_t *A, int Ws, const uint32_t *keys, int m) {
  const int lane = threadIdx.x & 31;
  int rec = -1, t = -1;
  if (lane == 0) rec = open_record(a, r, m, &t);
  rec = __shfl_sync(FULL, rec, 0);
  t = __shfl_sync(FULL, t, 0);
  if (t < 0) return false;
  uint32_t *dm = a.arena + __shfl_sync(FULL, lane == 0 ? a.recs[rec].off : 0ll, 0);
  const int Wsm = ((m + 31) >> 5) | 1;
  permute_rows_warp(r, A, Ws, keys, m, dm, Wsm, (int *)(dm + m * Wsm));
  __threadfence();
  Bits<1> C, P;
  bzero(C);
  P.w[0] = first_bits(m);
  write_task(a, t, rec, 1, C, P);
  return true;
}

// ------------------------------------------------------------- dense rows ---
//
// The adjacency of the top ranks as a bit matrix: row r holds r's later
// neighbours, for the last dense_cap ranks of the pruned graph (all of it at
// R-MAT scale 22: 35,500 vertices, 2.9% of the pairs, 79 MB used of the upper
// triangle, in L2).  A root's matrix is then gathered from it, 32 members per
// load and ballot, where the row lists took a lookup per entry (9.5 G per
// solve) and an atomic per member.  It is bound by L2: nearly every sector of
// a row's later part holds a member, 30-40 GB per solve.  The builder takes
// 0.1 ms, the block kernels 11.7 ms at scale 22 (24.4 before), 5.4 at scale 21
// (8.5), 2.6 at scale 20 (3.5).  Words before a row's own are not written and
// not read.  The cap bounds the room to 210 MB; roots below the covered ranks
// use the row lists.
constexpr int64_t kDenseCap = 40960;
constexpr int kDW = 8;  // warps per block of the builder

__host__ __device__ __forceinline__ int64_t dense_base(int64_t np, int64_t cap) { return np > cap ? np - cap : 0; }

__global__ void __launch_bounds__(kDW * 32) dense_rows_kernel(const int64_t *__restrict__ d_np,
                                                              const int64_t *__restrict__ orow,
                                                              const int32_t *__restrict__ ocol, int32_t cap,
                                                              int32_t stride, uint32_t *__restrict__ dense) {
  extern __shared__ uint32_t drow[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint32_t *row = drow + (size_t)wib * stride;
  const int64_t np = *d_np, base = dense_base(np, cap);
  const int words = (int)((np - base + 31) >> 5);
  for (int64_t r = base + (int64_t)blockIdx.x * kDW + wib; r < np; r += (int64_t)gridDim.x * kDW) {
    const int w0 = (int)((r - base) >> 5);
    for (int w = w0 + lane; w < words; w += 32) row[w] = 0;
    __syncwarp();
    const int64_t e0 = orow[r];
    const int4 *q = reinterpret_cast<const int4 *>(ocol + e0);
    const int nq = (int)((orow[r + 1] - e0) >> 2);
    for (int i = lane; i < nq; i += 32) {
      const int4 y = __ldg(q + i);
      const int ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const int c = (int)(ys[j] - base);
        if (ys[j] >= 0) atomicOr(&row[c >> 5], 1u << (c & 31));
      }
    }
    __syncwarp();
    uint32_t *out = dense + (r - base) * stride;
    for (int w = w0 + lane; w < words; w += 32) out[w] = row[w];
    __syncwarp();
  }
}

// ------------------------------------------------------------ warp class ---

struct WarpSmem {
  int Pidx[kWarpCap];
  int hk[2 * kWarpCap];
  short hv[2 * kWarpCap];
  uint32_t A[kWarpCap * 5];
  uint32_t al[4];
  int cnt;
};

// An upper bound of the edges of G[P] by one warp: the members' later-neighbour
// entries whose hash bit is set in a 2,048-bit filter of P (bits: 64 words).
// Eight lanes per row, four rows at a time, the next rows' offsets on their way.
__device__ __forceinline__ int edges_upto(const SA &a, const int *Pidx, int p, uint32_t *bits,
                                          unsigned long long &scanned) {
  const int lane = threadIdx.x & 31, grp = lane >> 3, gl = lane & 7;
  auto slot = [](int y) { return (unsigned)((unsigned)y * 2654435761u) >> 21; };
  bits[lane] = 0;
  bits[lane + 32] = 0;
  __syncwarp();
  for (int i = lane; i < p; i += 32) {
    const unsigned h = slot(Pidx[i]);
    atomicOr(&bits[h >> 5], 1u << (h & 31));
  }
  __syncwarp();
  int hits = 0;
  int64_t e0 = 0, e1 = 0;
  if (grp < p) {
    const int x = Pidx[grp];
    e0 = a.orow[x];
    e1 = a.orow[x + 1];
  }
  for (int i0 = 0; i0 < p; i0 += 4) {
    const int64_t c0 = e0;
    const int nq = (int)((e1 - e0) >> 2);
    e0 = e1 = 0;
    if (i0 + 4 + grp < p) {
      const int x = Pidx[i0 + 4 + grp];
      e0 = a.orow[x];
      e1 = a.orow[x + 1];
    }
    if (gl == 0) scanned += 4ull * (unsigned long long)nq;
    const int4 *row = reinterpret_cast<const int4 *>(a.ocol + c0);
    for (int q = gl; q < nq; q += 8) {
      const int4 y = __ldg(row + q);
      const int ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const unsigned h = slot(ys[j]);
        hits += (ys[j] >= 0 && ((bits[h >> 5] >> (h & 31)) & 1u)) ? 1 : 0;
      }
    }
  }
  __syncwarp();
  return dev::warp_sum(hits);
}

// Branch nodes that a warp expands on its root before what is left becomes a
// task: few while there are not as many tasks as the chip has warps for, many once
// there are, or while no clique is known (a first clique lies deeper than a few
// nodes, and every root would become a task under omega 0); none where the launch
// has fewer roots than that (a node takes 35 us here on a dense graph: G(150, 0.8)
// 8.9 ms, 9.5 with four).  With every
// branching root published at once, 300 graphs of 150-400 vertices took 130 ms
// (now 2.6), 5,000 of 30-80 vertices 160 (4.5), a 300 x 300 grid without a lower
// bound 118 (2.6, the search 0.2), R-MAT scale 17 (ef 12) without one 166 (5.5).
// 16 nodes always: R-MAT scale 15 loaded and solved 6% slower, the 300 graphs
// 3.2 ms; 32 instead of 64: 2.8 ms; 256: R-MAT 17 without a bound 10.3 ms.
constexpr int kRootNodes = 4, kRootNodesBusy = 64;

// Branching roots leave the kernel's registers to the others: their part is
// kept out of line.  What a root that needs more nodes has left becomes a
// task; without room for one it is searched here, in the order that the task
// would have had.
__device__ __noinline__ void branch_warp_root(const SA &a, Root r, uint32_t *A, int Ws, int W, uint32_t *al,
                                              uint32_t *keys, int *Pidx, uint32_t *stk, int om, bool few_roots,
                                              unsigned long long *nodes) {
  const int lane = threadIdx.x & 31;
  Bits<1> P, B, C, rest;
  P.w[0] = (lane < 4) ? al[lane] : 0u;
  bzero(C);
  unsigned long long n = 0, don = 0;
  color_ise<1, true>(A, Ws, W, P, om - 1, B);
  long long limit = LLONG_MAX;
  if (a.tasks) {
    const int t = lane == 0 ? *(volatile int32_t *)a.ntasks : 0;
    limit = om == 0 || __shfl_sync(FULL, t, 0) >= a.task_warps ? kRootNodesBusy : few_roots ? 0 : kRootNodes;
  }
  if (!dfs<1, true>(a, r, A, Ws, W, stk, 1, P, B, C, om, (Pool<1> *)nullptr, n, don, limit, &rest)) {
    __syncwarp();
    if (lane < 4) al[lane] = rest.w[0];
    __syncwarp();
    const int m = width_keys_warp(r, A, Ws, W, al, keys);
    if (!publish_warp(a, r, A, Ws, keys, m)) {
      const int Wm = (m + 31) >> 5, Wsm = Wm | 1;
      int *dp = (int *)(stk + m * Wsm);  // the stack is free: it has room for more than m rows of 66 words
      permute_rows_warp(r, A, Ws, keys, m, stk, Wsm, dp);
      for (int i = lane; i < m * Wsm; i += 32) A[i] = stk[i];
      for (int i = lane; i < m; i += 32) Pidx[i] = dp[i];
      __syncwarp();
      r.p = m;
      om = read_best(a.best, r.g);
      P.w[0] = first_bits(m);
      color_ise<1, true>(A, Wsm, Wm, P, om - 1, B);
      dfs<1, true>(a, r, A, Wsm, Wm, stk, 1, P, B, C, om, (Pool<1> *)nullptr, n, don);
    }
  }
  *nodes += n;
}

__global__ void __launch_bounds__(kSW * 32, 6) search_warp_kernel(SA a) {
  __shared__ WarpSmem sm[kSW];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  WarpSmem &S = sm[wib];
  const int64_t gw = (int64_t)blockIdx.x * kSW + wib;
  uint32_t *stk = a.stack + gw * a.stack_stride;
  unsigned long long colored = 0, branched = 0, nodes = 0, scanned = 0;
  int probe = 0;
  const int hmask = 2 * kWarpCap - 1;
  const int64_t nroots = *a.nroots;
  int score = nroots > 4 * (int64_t)gridDim.x * kSW ? 0 : -8;  // of the edge test below
  for (;;) {
    __syncwarp();
    int idx = 0;
    if (lane == 0) idx = *(volatile int32_t *)a.err ? INT_MAX : atomicAdd(a.next, 1);
    idx = __shfl_sync(FULL, idx, 0);
    if (idx >= nroots) break;
    const int u = a.roots[idx];
    const int g = a.ogid ? a.ogid[u] : 0;
    int om = read_best(a.best, g);
    if (a.ocore[u] < om) continue;
    if (lane == 0) S.cnt = 0;
    __syncwarp();
    load_P(a, u, om, S.Pidx, kWarpCap, &S.cnt, lane, 32);
    __syncwarp();
    const int p = S.cnt;
    if (p > kWarpCap) {
      if (lane == 0) atomicExch(a.err, kDevCheck);
      break;
    }
    if (p < om || p == 0) continue;
    // a larger clique needs om (om - 1) / 2 edges among the candidates: while
    // that decides most roots (sparse graphs), it is tested before the matrix
    // is built.  2.2 M roots of a 2,000-graph batch: 7.2 to 3.0 ms (3,100
    // instructions per root before); with a few roots per warp only, the test
    // costs more than it can learn (R-MAT scale 15: 0.21 to 0.27 ms)
    if (score >= 0 || (++probe & 31) == 0) {
      const int e = edges_upto(a, S.Pidx, p, S.A, scanned);
      if (2 * e < om * (om - 1)) {
        score = min(score + 1, 8);
        continue;
      }
      score = max(score - 2, -8);
    }
    int np2 = 32;
    while (np2 < p) np2 <<= 1;
    for (int i = lane; i < 2 * kWarpCap; i += 32) S.hk[i] = -1;
    for (int i = p + lane; i < np2; i += 32) S.Pidx[i] = INT_MIN;
    __syncwarp();
    bitonic_desc<false>(S.Pidx, np2, lane, 32);
    for (int i = lane; i < p; i += 32) hash_insert(S.hk, S.hv, hmask, S.Pidx[i], i);
    const int W = (p + 31) >> 5, Ws = W | 1;
    for (int i = lane; i < p * Ws; i += 32) S.A[i] = 0;
    __syncwarp();
    build_rows(a, S.Pidx, p, HashLookup{S.hk, S.hv, hmask}, S.A, Ws, 0, 1, scanned);
    __syncwarp();
    symmetrize<true>(S.A, Ws, W, p, 0, 1);
    __syncwarp();
    // alive set = all p vertices; (omega-1)-core of G[P]
    if (lane < 4) S.al[lane] = (lane < W) ? ((lane == W - 1 && (p & 31)) ? ((1u << (p & 31)) - 1u) : FULL) : 0u;
    __syncwarp();
    om = read_best(a.best, g);
    if (a.neigh_cores) {
      for (;;) {
        // lanes own rows k*32 + lane; row i's live bit is bit (i & 31) of word i >> 5
        uint32_t rm[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int k = 0; k < 4; k++) {
          if (k < W) {
            int i = k * 32 + lane;
            bool live = i < p && ((S.al[k] >> lane) & 1u);
            int deg = 0;
            if (live)
              for (int w = 0; w < W; w++) deg += __popc(S.A[i * Ws + w] & S.al[w]);
            rm[k] = __ballot_sync(FULL, live && deg < om - 1);
          }
        }
        __syncwarp();
        bool ch = (rm[0] | rm[1] | rm[2] | rm[3]) != 0;
        if (lane < 4) {
          uint32_t mine = lane == 0 ? rm[0] : lane == 1 ? rm[1] : lane == 2 ? rm[2] : rm[3];
          S.al[lane] &= ~mine;
        }
        __syncwarp();
        if (!ch) break;
      }
    }
    Bits<1> al;
    al.w[0] = (lane < 4) ? S.al[lane] : 0u;
    if (a.neigh_cores && bcount(al) < om) continue;
    colored++;
    Bits<1> B;
    color_ise<1, true>(S.A, Ws, W, al, om - 1, B);
    if (!bany(B)) continue;
    branched++;
    branch_warp_root(a, Root{u, g, S.Pidx, p}, S.A, Ws, W, S.al, (uint32_t *)S.hk, S.Pidx, stk, om, nroots <= a.task_warps,
                     &nodes);
  }
  if (lane == 0) {
    atomicAdd(a.counters + 0, colored);
    atomicAdd(a.counters + 1, branched);
    atomicAdd(a.counters + 2, nodes);
  }
  if ((lane & 7) == 0 && scanned) atomicAdd(a.counters + 4, scanned);
}

// ----------------------------------------------------------- block class ---

// DENSE: roots of the dense rows only, so neither the hash table (its place
// holds sort keys) nor the bitmap is needed.
template <int WPL, bool SM, int PC = 1024 * WPL, bool DENSE = false>
struct BlockLayout {
  static constexpr int PCAP = PC;
  static constexpr int HCAP = DENSE ? 1024 : 4 * PCAP;  // load factor 1/4: short probes
  static constexpr int WMAX = 32 * WPL;                 // alive / removal words (one per lane)
  static constexpr int WSMAX = ((PCAP + 31) / 32) | 1;  // largest matrix row stride, W | 1
  // bytes: Pidx, hk, hv, alive/rm words, pool, control, matrix
  static constexpr size_t off_P = 0;
  static constexpr size_t off_hk = off_P + PCAP * 4;
  static constexpr size_t off_hv = off_hk + HCAP * 4;
  static constexpr size_t off_al = off_hv + (DENSE ? 0 : HCAP * 2);
  static constexpr size_t off_rm = off_al + WMAX * 4;
  static constexpr size_t off_pool = off_rm + WMAX * 4;
  static constexpr size_t off_ctl = off_pool + ((sizeof(Pool<WPL>) + 15) / 16) * 16;
  static constexpr size_t off_bm = off_ctl + 64;                        // kBitmapWords words
  static constexpr size_t off_pre = off_bm + (DENSE ? 0 : (size_t)kBitmapWords * 4);  // kBitmapWords uint16
  static constexpr size_t off_A = off_pre + (DENSE ? 0 : (size_t)kBitmapWords * 2);
  static constexpr size_t bytes = off_A + (SM ? (size_t)PCAP * WSMAX * 4 : 0);
};

// P = {w in N+(u) : K(w) >= om} from u's dense row, in decreasing rank, into
// Pidx; returns its size, or more than cap (nothing usable written) when u has
// more later neighbours than that.  scan: kBW + 1 words, cnt: one word.  All
// threads.
__device__ int dense_P(const SA &a, int u, int om, int64_t base, int64_t np, int *Pidx, int cap, uint32_t *scan) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const uint32_t *row = a.dense + (u - base) * a.dense_stride;
  const int w0 = (int)((u - base) >> 5), words = (int)((np - base + 31) >> 5);
  const int last = words - 1;
  // words from the last one down, kBT at a time
  int total = 0;
  for (int k0 = 0; k0 <= last - w0; k0 += kBT) {
    const int w = last - (k0 + tid);
    uint32_t x = 0;
    if (w >= w0) {
      x = __ldg(row + w);
      if (w == w0) x &= ~((2u << ((u - (int)base) & 31)) - 1u);  // later ranks only
    }
    const int c = __popc(x);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    __syncthreads();
    if (lane == 31) scan[wid] = (uint32_t)incl;
    __syncthreads();
    int at = total + incl - c, all = 0;
    for (int i = 0; i < kBW; i++) {
      if (i < wid) at += (int)scan[i];
      all += (int)scan[i];
    }
    for (; x; at++) {
      const int b = 31 - __clz(x);
      x ^= 1u << b;
      if (at < cap) Pidx[at] = (int)base + 32 * w + b;
    }
    total += all;
  }
  __syncthreads();
  if (total > cap) return total;
  // drop the members whose core number omega has passed (none, unless omega
  // rose since the pruning)
  bool low = false;
  for (int i = tid; i < total; i += kBT) low |= __ldg(a.ocore + Pidx[i]) < om;
  if (!__syncthreads_or(low)) return total;
  int kept = 0;
  for (int i0 = 0; i0 < total; i0 += kBT) {
    const int i = i0 + tid, y = i < total ? Pidx[i] : 0;
    const bool keep = i < total && __ldg(a.ocore + y) >= om;
    const unsigned m = __ballot_sync(FULL, keep);
    __syncthreads();
    if (lane == 0) scan[wid] = (uint32_t)__popc(m);
    __syncthreads();
    int at = kept + __popc(m & ((1u << lane) - 1u)), all = 0;
    for (int k = 0; k < kBW; k++) {
      if (k < wid) at += (int)scan[k];
      all += (int)scan[k];
    }
    if (keep) Pidx[at] = y;
    kept += all;
  }
  __syncthreads();
  return kept;
}

// Lower triangle of G[P] from the dense rows: word w of row i is a ballot over
// members 32w .. 32w+31 (later ranks than member i for indices below i).  Rows
// go to warps as they free up, the longest first; eight words in flight.
__device__ __forceinline__ void dense_build(const SA &a, const int *Pidx, int p, int64_t base, uint32_t *A, int Ws,
                                            int W, int *dyn, unsigned long long &scanned) {
  const int lane = threadIdx.x & 31;
  for (;;) {
    int i = 0;
    if (lane == 0) i = p - 1 - atomicAdd(dyn, 1);
    i = __shfl_sync(FULL, i, 0);
    if (i < 0) break;
    const uint32_t *row = a.dense + (int64_t)(Pidx[i] - base) * a.dense_stride;
    const int nw = (i + 31) >> 5;  // words with an index below i
    uint32_t mine = 0;
    for (int w0 = 0; w0 < nw; w0 += 8) {
      uint32_t x[8];
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int j = 32 * (w0 + q) + lane;
        const int c = j < i ? Pidx[j] - (int)base : -1;
        x[q] = c >= 0 ? __ldg(row + (c >> 5)) >> (c & 31) : 0u;
      }
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const unsigned m = __ballot_sync(FULL, x[q] & 1u);
        if (lane == w0 + q) mine = m;
      }
    }
    if (lane < W) A[i * Ws + lane] = mine;
    if (lane == 0) scanned += (unsigned long long)i;
  }
}

// The candidates left by the core test (bits al) in minimum-width order: those
// of smallest degree among the remaining ones leave step by step (all of them
// at once), and later ones come first (ties: smaller index).  keys[0..m) =
// step and complement of the index, sorted; returns m.  keys: room for the
// next power of two above p; gone: one word per 32 candidates.  All threads.
__device__ int width_keys(const uint32_t *A, int p, int Ws, int W, const uint32_t *al, uint32_t *keys, uint32_t *gone) {
  __shared__ int s_min;
  const int tid = threadIdx.x, lane = tid & 31;
  int np2 = 32;
  while (np2 < p) np2 <<= 1;
  int m = 0;
  for (int w = 0; w < W; w++) m += __popc(al[w]);
  int deg[2];  // candidates tid and tid + kBT; INT_MAX: not (or no longer) there
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const int i = tid + q * kBT;
    deg[q] = INT_MAX;
    if (i < p && ((al[i >> 5] >> (i & 31)) & 1u)) {
      deg[q] = 0;
      for (int w = 0; w < W; w++) deg[q] += __popc(A[i * Ws + w] & al[w]);
    }
    if (i < np2) keys[i] = 0;
  }
  int left = m;
  for (uint32_t step = 1; left > 0; step++) {
    __syncthreads();
    if (tid == 0) s_min = INT_MAX;
    __syncthreads();
    const int mine = __reduce_min_sync(FULL, min(deg[0], deg[1]));
    if (lane == 0 && mine != INT_MAX) atomicMin(&s_min, mine);
    __syncthreads();
    const int lo = s_min;
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const int i = tid + q * kBT;
      const unsigned out = __ballot_sync(FULL, deg[q] == lo);
      if (deg[q] == lo) {
        keys[i] = (step << 16) | (uint32_t)(0xffff - i);
        deg[q] = INT_MAX;
      }
      if (lane == 0 && (i >> 5) < W) gone[i >> 5] = out;
    }
    __syncthreads();
    for (int w = 0; w < W; w++) {
      const uint32_t x = gone[w];
      if (!x) continue;
      left -= __popc(x);
#pragma unroll
      for (int q = 0; q < 2; q++)
        if (deg[q] != INT_MAX) deg[q] -= __popc(A[(tid + q * kBT) * Ws + w] & x);
    }
  }
  __syncthreads();
  bitonic_desc<true>((int *)keys, np2, tid, kBT);
  return m;
}

// Their matrix and P list in that order, to global memory: dm (m rows of Wsm
// words), dp.  All threads.
__device__ void permute_rows(const uint32_t *A, int Ws, const int *Pidx, const uint32_t *keys, int m, uint32_t *dm,
                             int Wsm, int *dp) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int i = wid; i < m; i += kBW) {
    const uint32_t x = permuted_row(A, Ws, keys, m, i);
    if (lane < Wsm) dm[(int64_t)i * Wsm + lane] = x;
  }
  for (int i = tid; i < m; i += kBT) dp[i] = Pidx[0xffff - (int)(keys[i] & 0xffffu)];
}

// A block's root as a task, sorted as above (the colouring of the task's upper
// levels takes the densest first too).  ctl: two words.  False, publishing
// nothing, without room.  All threads.
__device__ bool publish_sorted(const SA &a, const Root &r, const uint32_t *A, int Ws, const uint32_t *keys, int m,
                               int *ctl) {
  const int Wsm = ((m + 31) >> 5) | 1;
  if (threadIdx.x == 0) ctl[1] = open_record(a, r, m, &ctl[0]);
  __syncthreads();
  if (ctl[0] < 0) return false;
  uint32_t *dm = a.arena + a.recs[ctl[1]].off;
  permute_rows(A, Ws, r.Pidx, keys, m, dm, Wsm, (int *)(dm + (int64_t)m * Wsm));
  __threadfence();
  __syncthreads();
  if (threadIdx.x < 32) {
    Bits<1> C, P;
    bzero(C);
    P.w[0] = first_bits(m);
    write_task(a, ctl[0], ctl[1], 1, C, P);
  }
  return true;
}

// The warps of a block search one root (or one task) together: warps that
// hold work run the depth-first Branch and hand untried branches to idle
// warps through the block's pool; the call returns when the pool is empty
// and every warp is idle.  All warps of the block call it.
template <int WPL, bool SM>
__device__ void block_search(const SA &a, const Root &r, const uint32_t *A, int Ws, int W, uint32_t *stk,
                             Pool<WPL> *pool, bool have, Bits<WPL> P, Bits<WPL> B, Bits<WPL> C, int cs, int wat,
                             unsigned long long &nodes, unsigned long long &don) {
  const int lane = threadIdx.x & 31;
  const int g = r.g;
  long long waited = 0;
  int lastbeat = -1;
  for (;;) {
    if (have) {
      dfs<WPL, SM>(a, r, A, Ws, W, stk, cs, P, B, C, wat, pool, nodes, don);
      have = false;
      if (lane == 0) {
        if (pool_lock(pool, a.err, a.spin)) {
          pool->idle++;
          pool_unlock(pool);
        }
      }
      __syncwarp();
    }
    int got = 0;
    if (lane == 0) {
      if (pool_lock(pool, a.err, a.spin)) {
        if (pool->count > 0) {
          got = pool->count--;
          pool->idle--;
        } else if (pool->idle == kBW) {
          got = -1;
        }
        if (got <= 0) pool_unlock(pool);
      } else {
        got = -1;
      }
    }
    got = __shfl_sync(FULL, got, 0);
    if (got < 0) break;
    if (got == 0) {
      int beat = *(volatile int *)&pool->beat;
      if (beat != lastbeat) {
        lastbeat = beat;
        waited = 0;
      }
      if (__shfl_sync(FULL, (++waited > a.spin || (lane == 0 && *(volatile int32_t *)a.err)) ? 1 : 0, 0)) {
        if (lane == 0) atomicExch(a.err, kDevTimeout);
        break;
      }
      __nanosleep(128);
      continue;
    }
    // copy the task while still holding the lock (lane 0 holds it)
    const int slot = got - 1;
#pragma unroll
    for (int k = 0; k < WPL; k++) {
      C.w[k] = pool->C[slot][k * 32 + lane];
      P.w[k] = pool->P[slot][k * 32 + lane];
    }
    cs = pool->csize[slot];
    __syncwarp();
    if (lane == 0) pool_unlock(pool);
    __syncwarp();
    int om2 = read_best(a.best, g);
    color_ise<WPL, SM>(A, Ws, W, P, om2 - cs, B);
    wat = om2;
    have = bany(B);
    if (!have && lane == 0) {
      if (pool_lock(pool, a.err, a.spin)) {
        pool->idle++;
        pool_unlock(pool);
      }
    }
    __syncwarp();
  }
}

// PC: candidate capacity of the shared-memory layout.  The kMidCap layout
// fits two blocks per SM; its roots with more candidates go to the overflow
// list, which the 1,024-candidate launch then searches.
template <int WPL, bool SM, int PC, bool DENSE = false>
__global__ void __launch_bounds__(kBT, (SM && (PC <= kMidCap || DENSE)) ? 2 : 1) search_block_kernel(SA a) {
  using L = BlockLayout<WPL, SM, PC, DENSE>;
  extern __shared__ __align__(16) unsigned char smem[];
  int *Pidx = (int *)(smem + L::off_P);
  int *hk = (int *)(smem + L::off_hk);
  short *hv = (short *)(smem + L::off_hv);
  uint32_t *al = (uint32_t *)(smem + L::off_al);
  uint32_t *rm = (uint32_t *)(smem + L::off_rm);
  Pool<WPL> *pool = (Pool<WPL> *)(smem + L::off_pool);
  int *ctl = (int *)(smem + L::off_ctl);  // [0] root idx, [1] omega, [2] count, [3] flag, [4] go, [5] error
  uint32_t *A = SM ? (uint32_t *)(smem + L::off_A) : (a.gmat + (int64_t)blockIdx.x * a.gmat_stride);
  uint32_t *bm = (uint32_t *)(smem + L::off_bm);
  uint16_t *pre = (uint16_t *)(smem + L::off_pre);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  uint32_t *stk = a.stack + ((int64_t)blockIdx.x * kBW + wid) * a.stack_stride;
  unsigned long long colored = 0, branched = 0, nodes = 0, don = 0, scanned = 0;
  const int hmask = L::HCAP - 1;
  const int64_t nroots = *a.nroots;
  const int64_t npr = *a.np_count;
  if (!DENSE)
    for (int i = tid; i < kBitmapWords; i += kBT) bm[i] = 0u;  // each root clears the bits it set

  for (;;) {
    __syncthreads();
    if (tid == 0) {
      ctl[0] = atomicAdd(a.next, 1);
      ctl[2] = 0;
      ctl[5] = *(volatile int32_t *)a.err;
      ctl[6] = 0;  // the row builder's group counter
    }
    __syncthreads();
    const int idx = ctl[0];
    if (idx >= nroots || ctl[5]) break;
    const int u = a.roots[idx];
    const int g = a.ogid ? a.ogid[u] : 0;
    if (tid == 0) ctl[1] = *(volatile int32_t *)(a.best + g);
    __syncthreads();
    int om = ctl[1];
    if (a.ocore[u] < om) continue;
    // u among the dense rows: its candidates and their matrix from those;
    // else by member lookups, in a bitmap when the later ranks (u, n') fit it,
    // otherwise in a hash table
    const int64_t dbase = dense_base(npr, a.dense_cap);
    const bool dense = SM && a.dense && u >= dbase;
    if (DENSE && !dense) {  // to the launch with the lookup structures
      if (tid == 0) a.overflow[atomicAdd((unsigned long long *)a.noverflow, 1ull)] = u;
      continue;
    }
    const int base = u + 1;
    const bool use_bm = !dense && a.use_bitmap && ((npr - base + 31) >> 5) <= kBitmapWords;
    int p;
    if (dense) {
      p = dense_P(a, u, om, dbase, npr, Pidx, L::PCAP, rm);
    } else {
      if (!use_bm)
        for (int i = tid; i < L::HCAP; i += kBT) hk[i] = -1;
      for (int i = tid; i < L::PCAP; i += kBT) Pidx[i] = INT_MIN;
      __syncthreads();
      load_P(a, u, om, Pidx, L::PCAP, &ctl[2], tid, kBT);
      __syncthreads();
      p = ctl[2];
    }
    if (p > L::PCAP) {
      if (a.overflow) {
        if (tid == 0) a.overflow[atomicAdd((unsigned long long *)a.noverflow, 1ull)] = u;
        continue;
      }
      if (tid == 0) atomicExch(a.err, kDevUnsupported);
      break;
    }
    if (p < om || p == 0) continue;
    const int wwin = (int)((npr - base + 31) >> 5);
    if (dense) {
    } else if (use_bm) {
      // P in any order: its bits, the prefix counts, and then every member
      // moves to its index in decreasing-rank order, which the counts give
      // (the hash table's space, unused on this path, holds the list)
      int *tmp = hk;
      for (int i = tid; i < p; i += kBT) {
        const int y = Pidx[i];
        atomicOr(&bm[(y - base) >> 5], 1u << ((y - base) & 31));
        tmp[i] = y;
      }
      __syncthreads();
      // pre[w] = members in words [0, w): each thread counts a contiguous
      // chunk of words, the warps' totals are scanned in rm[], then each
      // thread writes its chunk's prefixes
      const int per = (wwin + kBT - 1) / kBT;
      const int w0 = min(wwin, tid * per), w1 = min(wwin, w0 + per);
      int mine = 0;
      for (int w = w0; w < w1; w++) mine += __popc(bm[w]);
      int incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) rm[wid] = (uint32_t)incl;
      __syncthreads();
      int before = 0;
      for (int w = 0; w < wid; w++) before += (int)rm[w];
      int run = before + incl - mine;
      for (int w = w0; w < w1; w++) {
        pre[w] = (uint16_t)run;
        run += __popc(bm[w]);
      }
      __syncthreads();
      const BitmapLookup at{bm, pre, base, p};
      for (int i = tid; i < p; i += kBT) Pidx[at(tmp[i])] = tmp[i];
    } else {
      int np2 = 32;
      while (np2 < p) np2 <<= 1;
      bitonic_desc<true>(Pidx, np2, tid, kBT);
      for (int i = tid; i < p; i += kBT) hash_insert(hk, hv, hmask, Pidx[i], i);
    }
    const int W = (p + 31) >> 5, Ws = W | 1;
    if (!dense)
      for (int64_t i = tid; i < (int64_t)p * Ws; i += kBT) A[i] = 0;
    if (!SM) __threadfence();
    __syncthreads();
    if (dense)
      dense_build(a, Pidx, p, dbase, A, Ws, W, &ctl[6], scanned);
    else if (use_bm)
      build_rows(a, Pidx, p, BitmapLookup{bm, pre, base, p}, A, Ws, wid, kBW, scanned, &ctl[6]);
    else
      build_rows(a, Pidx, p, HashLookup{hk, hv, hmask}, A, Ws, wid, kBW, scanned, &ctl[6]);
    if (!SM) __threadfence();
    __syncthreads();
    if (use_bm)
      for (int i = tid; i < p; i += kBT) {
        const int r = Pidx[i] - base;
        atomicAnd(&bm[r >> 5], ~(1u << (r & 31)));
      }
    symmetrize<SM>(A, Ws, W, p, wid, kBW);
    if (!SM) __threadfence();
    __syncthreads();
    for (int w = tid; w < L::WMAX; w += kBT)
      al[w] = (w < W) ? ((w == W - 1 && (p & 31)) ? ((1u << (p & 31)) - 1u) : FULL) : 0u;
    if (tid == 0) ctl[1] = *(volatile int32_t *)(a.best + g);
    __syncthreads();
    om = ctl[1];
    if (a.neigh_cores) {
      // (omega-1)-core of G[P]: drop rows with fewer than omega-1 live neighbours
      for (;;) {
        for (int k = wid; k < W; k += kBW) {
          int i = k * 32 + lane;
          int deg = 0;
          bool live = i < p && ((al[k] >> lane) & 1u);
          if (live)
            for (int w = 0; w < W; w++) deg += __popc(rw<SM>(A, (int64_t)i * Ws + w) & al[w]);
          unsigned m = __ballot_sync(FULL, live && deg < om - 1);
          if (lane == 0) rm[k] = m;
        }
        if (tid == 0) ctl[3] = 0;
        __syncthreads();
        for (int k = tid; k < W; k += kBT)
          if (rm[k]) {
            al[k] &= ~rm[k];
            ctl[3] = 1;
          }
        __syncthreads();
        if (!ctl[3]) break;
        __syncthreads();
      }
    }
    // colouring test and the search, started by warp 0
    Root r{u, g, Pidx, p};
    Bits<WPL> P, B, C;
    bzero(C);
    int cs = 1, wat = om;
    bool have = false;
    if (wid == 0) {
#pragma unroll
      for (int k = 0; k < WPL; k++) P.w[k] = al[k * 32 + lane];
      int go = 0;
      if (!a.neigh_cores || bcount(P) >= om) {
        colored++;
        color_ise<WPL, SM>(A, Ws, W, P, om - 1, B);
        go = bany(B) ? 1 : 0;
        if (go) branched++;
      }
      have = go != 0;
      if (lane == 0) {
        ctl[4] = go;
        pool->lock = 0;
        pool->count = 0;
        pool->idle = kBW - 1;
        pool->beat = 0;
      }
    }
    __syncthreads();
    if (!ctl[4]) continue;
    int Wr = W, Wsr = Ws;  // row words and stride of the searched matrix
    if constexpr (WPL == 1 && SM) {
      // in minimum-width order (in the hash table's space: the matrix is
      // built); a task, or searched here: the matrix goes through global
      // memory, and the colouring test is taken again in the new order.  In
      // rank order the search in place took 1 to 10 s on 2 of 3 R-MAT scale-20
      // graphs (5.7 and 9.4 ms sorted), 10-14 ms at scale 21 (9).  Where most
      // roots of a dense graph find the arena full: G(1200, 0.4) 187 ms in
      // rank order, 175 sorted; G(1500, 0.3), smaller trees, 90 and 100
      const int m = width_keys(A, p, Ws, W, al, (uint32_t *)hk, rm);
      if (a.tasks && publish_sorted(a, r, A, Ws, (uint32_t *)hk, m, ctl + 8)) continue;
      uint32_t *dm = a.sort + (int64_t)blockIdx.x * a.sort_stride;
      Wr = (m + 31) >> 5;
      Wsr = Wr | 1;
      int *dp = (int *)(dm + (int64_t)m * Wsr);
      permute_rows(A, Ws, Pidx, (uint32_t *)hk, m, dm, Wsr, dp);
      __syncthreads();
      for (int i = tid; i < m * Wsr; i += kBT) A[i] = dm[i];
      for (int i = tid; i < m; i += kBT) Pidx[i] = dp[i];
      __syncthreads();
      r.p = m;
      if (wid == 0) {
        P.w[0] = first_bits(m);
        color_ise<WPL, SM>(A, Wsr, Wr, P, om - 1, B);
        have = bany(B);
        if (lane == 0) ctl[4] = have ? 1 : 0;
      }
      __syncthreads();
      if (!ctl[4]) continue;
    }
    block_search<WPL, SM>(a, r, A, Wsr, Wr, stk, pool, have, P, B, C, cs, wat, nodes, don);
    __syncthreads();
  }
  if (lane == 0) {
    atomicAdd(a.counters + 0, colored);
    atomicAdd(a.counters + 1, branched);
    atomicAdd(a.counters + 2, nodes);
    atomicAdd(a.counters + 3, don);
  }
  if ((lane & 7) == 0 && scanned) atomicAdd(a.counters + 5, scanned);
}


// ------------------------------------------------------------ task queue ---
//
// Tasks are searched by single warps on a compact copy of their subproblem.
// A task's candidates are a few hundred at most (a neighbourhood of a
// neighbourhood), so their adjacency matrix takes 2 or 8 KB of shared memory
// per warp (16 warps per SM), and every lane holds whole vertex sets in
// registers.  The search is bound by the latency of the greedy colouring, a
// chain from vertex to vertex.  Against whole blocks per task with a bit
// matrix of up to 1,024 candidates, the candidates in rank order and one set
// word per lane: 13 us per Branch node before, 7 us now, and 5 to 30 times
// fewer nodes, since a root's candidates are in the minimum-width order of its
// neighbourhood.  R-MAT scale 18, edge factor 12: search 83-330 ms before (it
// depends on when the larger cliques are found), 3.5-4.9 ms now, of which the tasks
// 2.5-3.9; scale 15, edge factor 16: 60-104 ms before, 0.9-1.2 ms now.  (While a
// branch that was handed over stayed among its level's candidates, and came back
// when omega rose, scale 17 took 260,000 nodes and 3.8 ms; now 165,000 and 2.6.)
// Subproblems above 256 candidates are searched depth first by the warp on the
// root's matrix until a child fits; publishing every branch of such a node
// instead (breadth first) let the queue fill with them before omega rose: two
// of 40 R-MAT scale-20 graphs then took 36 and 85 s, now none of 129 takes
// more than 65 ms.  Block roots are published with their candidates in
// minimum-width order (width_keys), so that these levels are coloured densest
// first as well.
constexpr int kTM = 256;    // candidates of a compact subproblem
constexpr int kTW = 4;      // warps per block of the task kernel
constexpr int kTStk = 20;   // stack words per level (two sets of at most 8 words, omega, chosen vertex)

struct TaskSmem {
  uint32_t A[kTM * (kTM / 32)];
  int mem[kTM];       // position in the root's P list of compact vertex i
  uint32_t bits[32];  // sets over the root's positions
  uint32_t drop[32];
  uint8_t lst[kTM + 16];  // vertices of the set being coloured
};

template <int NW>
struct Set {
  uint32_t w[NW];
};
template <int NW>
__device__ __forceinline__ bool sany(const Set<NW> &s) {
  uint32_t x = 0;
#pragma unroll
  for (int i = 0; i < NW; i++) x |= s.w[i];
  return x != 0;
}
template <int NW>
__device__ __forceinline__ int scount(const Set<NW> &s) {
  int c = 0;
#pragma unroll
  for (int i = 0; i < NW; i++) c += __popc(s.w[i]);
  return c;
}
template <int NW>
__device__ __forceinline__ int shighest(const Set<NW> &s) {
  int v = -1;
#pragma unroll
  for (int i = 0; i < NW; i++)
    if (s.w[i]) v = 32 * i + 31 - __clz(s.w[i]);
  return v;
}
template <int NW>
__device__ __forceinline__ void sclear(Set<NW> &s, int v) {
  const uint32_t m = ~(1u << (v & 31));
#pragma unroll
  for (int i = 0; i < NW; i++)
    if (i == (v >> 5)) s.w[i] &= m;
}
template <int NW>
__device__ __forceinline__ Set<NW> sload(const uint32_t *p) {
  Set<NW> s;
#pragma unroll
  for (int i = 0; i < NW / 4; i++) {
    const uint4 x = reinterpret_cast<const uint4 *>(p)[i];
    s.w[4 * i] = x.x;
    s.w[4 * i + 1] = x.y;
    s.w[4 * i + 2] = x.z;
    s.w[4 * i + 3] = x.w;
  }
  return s;
}
// one lane stores
template <int NW>
__device__ __forceinline__ void sstore(uint32_t *p, const Set<NW> &s) {
#pragma unroll
  for (int i = 0; i < NW / 4; i++)
    reinterpret_cast<uint4 *>(p)[i] = make_uint4(s.w[4 * i], s.w[4 * i + 1], s.w[4 * i + 2], s.w[4 * i + 3]);
}

// Greedy colouring of P in index order with at most q classes: a vertex takes
// the first class that holds none of its neighbours; R receives the vertices
// no class takes.  Class 32 s + lane is in this lane's registers, so placing a
// vertex is a few ANDs and a ballot per 32 classes, 64 classes at a time
// without a branch.  The vertices are listed first: a row is on its way from
// shared memory while the one before is placed, and no find-first-set is on
// the chain from one vertex to the next.  Every lane holds the same P and R.
template <int NW>
__device__ __forceinline__ void colour_set(const uint32_t *A, uint8_t *lst, const Set<NW> &P, int q, Set<NW> &R) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int end[NW];
  __syncwarp();
#pragma unroll
  for (int w = 0; w < NW; w++) {
    const int at = w ? end[w - 1] : 0;
    if ((P.w[w] >> lane) & 1u) lst[at + __popc(P.w[w] & lt)] = (uint8_t)(32 * w + lane);
    end[w] = at + __popc(P.w[w]);
  }
  __syncwarp();
  Set<NW> cls[NW];
#pragma unroll
  for (int s = 0; s < NW; s++)
#pragma unroll
    for (int i = 0; i < NW; i++) cls[s].w[i] = 0;
  int v = lst[0], vn = lst[1];  // past the end: some row of the matrix's space, not used
  Set<NW> row = sload<NW>(A + v * NW);
  int i = 0;
#pragma unroll
  for (int w = 0; w < NW; w++) {
    R.w[w] = 0;
    for (; i < end[w]; i++) {
      const Set<NW> next = sload<NW>(A + vn * NW);
      const int vnn = lst[i + 2];
      const uint32_t bit = 1u << (v & 31);
      bool placed = false;
#pragma unroll
      for (int p = 0; p < NW / 2; p++) {
        if (p == 0 || (!placed && 64 * p < q)) {
          // vertices come in index order: no class holds one of a later word
          uint32_t y0 = 0, y1 = 0;
#pragma unroll
          for (int k = 0; k <= w; k++) {
            y0 |= cls[2 * p].w[k] & row.w[k];
            y1 |= cls[2 * p + 1].w[k] & row.w[k];
          }
          const bool free0 = y0 == 0 && 64 * p + lane < q, free1 = y1 == 0 && 64 * p + 32 + lane < q;
          const unsigned f0 = __ballot_sync(FULL, free0), f1 = __ballot_sync(FULL, free1);
          if (free0 && !(f0 & lt)) cls[2 * p].w[w] |= bit;
          if (free1 && !(f0 | (f1 & lt))) cls[2 * p + 1].w[w] |= bit;
          placed = (f0 | f1) != 0;
        }
      }
      if (!placed) R.w[w] |= bit;
      row = next;
      v = vn;
      vn = vnn;
    }
  }
}

// What a warp knows of its task.
struct TaskCtx {
  int rec, cs;          // record, clique size (counting u) at the task's start
  uint32_t C;           // the task's clique over the root's positions, one word per lane
  int u, g, p, W, Ws;
  const uint32_t *A;    // the root's matrix (arena)
  const int *Pidx;      // the root's P list (arena)
  uint32_t *lev;        // levels of more than kTM candidates (kBigLev words each) ...
  int nlev;             // ... and how many there are
};
constexpr int kBigLev = 66;  // two sets of 32 words, omega at the colouring, chosen vertex

// The clique {u} + C + the compact vertices path[0..d) (+ v) in original
// ids.  All lanes.
__device__ void write_task_clique(int32_t *base, const SA &a, const TaskCtx &T, const int *mem, const uint32_t *stk,
                                  int d, int v) {
  const int lane = threadIdx.x & 31;
  const int cnt = __popc(T.C);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += y;
  }
  const int tot = __shfl_sync(FULL, incl, 31);
  int pos = 1 + incl - cnt;
  uint32_t x = T.C;
  while (x) {
    const int b = __ffs(x) - 1;
    x &= x - 1;
    base[pos++] = a.oold[__ldcg(T.Pidx + 32 * lane + b)];
  }
  if (lane == 0) base[0] = a.oold[T.u];
  const int n = d + (v >= 0 ? 1 : 0);
  for (int i = lane; i < n; i += 32) {
    const int y = i < d ? (int)stk[i * kTStk + 17] : v;
    base[1 + tot + i] = a.oold[__ldcg(T.Pidx + mem[y])];
  }
}

// Hand the untried branches of the shallowest level that has some to the
// queue, one task each; that level keeps none, also among its candidates, so
// that a colouring under a higher omega does not bring them back.  All or
// nothing: without room in the queue nothing changes.  Returns the tasks
// written.
template <int NW>
__device__ int offer_level(const SA &a, const TaskCtx &T, TaskSmem &S, uint32_t *stk, int d, Set<NW> &P, Set<NW> &B) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  int l = 0;
  Set<NW> Pl = P, Bl = B;
  for (; l < d; l++) {
    Bl = sload<NW>(stk + l * kTStk + 8);
    if (sany(Bl)) break;
  }
  if (l < d) Pl = sload<NW>(stk + l * kTStk);
  else Bl = B;
  const int k = scount(Bl);
  if (k == 0) return 0;
  int t = -1;
  if (lane == 0) t = reserve_tasks(a, k, 1);
  t = __shfl_sync(FULL, t, 0);
  if (t < 0) return 0;
  // the clique at this level, over the root's positions
  S.bits[lane] = T.C;
  __syncwarp();
  for (int i = lane; i < l; i += 32) {
    const int pos = S.mem[stk[i * kTStk + 17]];
    atomicOr(&S.bits[pos >> 5], 1u << (pos & 31));
  }
  __syncwarp();
  const uint32_t Cl = S.bits[lane];
  const int csl = T.cs + l;
  for (int i = 0; i < k; i++) {
    const int x = shighest(Bl);
    sclear(Bl, x);
    sclear(Pl, x);
    const Set<NW> row = sload<NW>(S.A + x * NW);
    Set<NW> TP;
#pragma unroll
    for (int q = 0; q < NW; q++) TP.w[q] = Pl.w[q] & row.w[q];
    const int om = read_best(a.best, T.g);
    const int n = scount(TP);
    int cs = csl + 1;
    if (cs + n <= om) cs = 0;  // decided: an empty task
    // the child's candidates over the root's positions
    __syncwarp();
    S.bits[lane] = 0;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < NW; q++)
      if ((TP.w[q] >> lane) & 1u) {
        const int pos = S.mem[32 * q + lane];
        atomicOr(&S.bits[pos >> 5], 1u << (pos & 31));
      }
    __syncwarp();
    const int px = S.mem[x];
    Bits<1> Cx, Px;
    Cx.w[0] = Cl | (lane == (px >> 5) ? 1u << (px & 31) : 0u);
    Px.w[0] = S.bits[lane];
    write_task(a, t + i, T.rec, cs, Cx, Px);
  }
  if (l < d) {
    if (lane == 0) {
      Set<NW> none;
#pragma unroll
      for (int q = 0; q < NW; q++) none.w[q] = 0;
      sstore<NW>(stk + l * kTStk, Pl);
      sstore<NW>(stk + l * kTStk + 8, none);
    }
    __syncwarp();
  } else {
    P = Pl;
#pragma unroll
    for (int q = 0; q < NW; q++) B.w[q] = 0;
  }
  return k;
}

// The same for the levels above the compact form, of which the first `chosen`
// have a chosen vertex in T's clique; returns the tasks written.
__device__ __noinline__ int offer_big(const SA &a, const TaskCtx &T, int chosen) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  for (int l = 0; l < T.nlev; l++) {
    uint32_t *q = T.lev + (int64_t)l * kBigLev;
    Bits<1> Pl, Bl, Cl;
    Bl.w[0] = q[32 + lane];
    const int k = bcount(Bl);
    if (k == 0) continue;
    int t = -1;
    if (lane == 0) t = reserve_tasks(a, k, 1);
    t = __shfl_sync(FULL, t, 0);
    if (t < 0) return 0;
    Pl.w[0] = q[lane];
    Cl.w[0] = T.C;
    for (int i = l; i < chosen; i++) bclear(Cl, level_word(T.lev + (int64_t)i * kBigLev + 65));
    const Root r{T.u, T.g, T.Pidx, T.p};
    for (int i = 0; i < k; i++) {
      const int x = bhighest(Bl);
      bclear(Bl, x);
      bclear(Pl, x);
      emit_task(a, r, T.A, T.Ws, T.W, T.rec, t + i, Cl, T.cs - (chosen - l), Pl, x);
    }
    q[lane] = Pl.w[0];
    q[32 + lane] = 0;
    __syncwarp();
    return k;
  }
  return 0;
}

// Depth-first Branch on the compact subproblem S.A over m vertices.
template <int NW>
__device__ void task_dfs(const SA &a, const TaskCtx &T, TaskSmem &S, uint32_t *stk, int m, unsigned long long &nodes,
                         unsigned long long &don) {
  const int lane = threadIdx.x & 31;
  Set<NW> P, B;
#pragma unroll
  for (int i = 0; i < NW; i++)
    P.w[i] = m >= 32 * (i + 1) ? FULL : (m > 32 * i ? (1u << (m - 32 * i)) - 1u : 0u);
  int d = 0, wat = -1, csize = T.cs;
  int since = 0;
  long long spent = 0;
  // omega, read one step ahead (an old value only prunes less)
  int ahead = *(const volatile int32_t *)(a.best + T.g);
  for (;;) {
    const int om = __shfl_sync(FULL, ahead, 0);
    ahead = *(const volatile int32_t *)(a.best + T.g);
    if (om > wat) {  // a new node, or omega has risen since it was coloured
      colour_set<NW>(S.A, S.lst, P, om - csize, B);
      wat = om;
    }
    const int v = shighest(B);
    if (v < 0) {
      if (d == 0) return;
      d--;
      csize--;
      P = sload<NW>(stk + d * kTStk);
      B = sload<NW>(stk + d * kTStk + 8);
      wat = (int)stk[d * kTStk + 16];
      continue;
    }
    if (++since >= a.offer_nodes) {
      // waiting warps hold tickets beyond the last published task
      since = 0;
      int hungry = 0;
      if (lane == 0) {
        hungry = *(volatile int32_t *)a.task_next > *(volatile int32_t *)a.ntasks;
        if (*(volatile int32_t *)a.err) hungry = -1;
      }
      hungry = __shfl_sync(FULL, hungry, 0);
      if (hungry < 0) return;
      if (hungry) {
        int k = offer_big(a, T, T.nlev);
        if (k == 0) k = offer_level<NW>(a, T, S, stk, d, P, B);
        don += (unsigned long long)k;
        if (k) continue;
      }
    }
    sclear(B, v);
    sclear(P, v);
    const Set<NW> row = sload<NW>(S.A + v * NW);
    Set<NW> NP;
#pragma unroll
    for (int i = 0; i < NW; i++) NP.w[i] = P.w[i] & row.w[i];
    nodes++;
    if ((++spent & 255) == 0 && lane == 0) atomicAdd(a.progress, 1);
    const int cnt = scount(NP);
    if (cnt == 0) {
      if (csize + 1 > om) {
        __syncwarp();
        const int dd = d;
        dev::raise_incumbent(a.best, a.lock, a.wit, a.voff, T.g, csize + 1, a.err, a.spin,
                             [&](int, int32_t *base) { write_task_clique(base, a, T, S.mem, stk, dd, v); });
      }
      continue;
    }
    if (csize + 1 + cnt <= om) continue;
    if (lane == 0) {
      sstore<NW>(stk + d * kTStk, P);
      sstore<NW>(stk + d * kTStk + 8, B);
      stk[d * kTStk + 16] = (uint32_t)wat;
      stk[d * kTStk + 17] = (uint32_t)v;
    }
    __syncwarp();
    d++;
    csize++;
    P = NP;
    wat = -1;
  }
}

// Compact matrix of the m listed members (S.mem): row i, word w holds the
// adjacency of member i to members 32w .. 32w+31.  A row of the root's matrix
// is at most 32 words: one coalesced load, then a shuffle, a shift and a
// ballot per compact word.
template <int NW>
__device__ void compact_matrix(const TaskCtx &T, TaskSmem &S, int m) {
  const int lane = threadIdx.x & 31;
  int at[NW];
#pragma unroll
  for (int w = 0; w < NW; w++) at[w] = 32 * w + lane < m ? S.mem[32 * w + lane] : -1;
  for (int i0 = 0; i0 < m; i0 += 4) {
    uint32_t x[4];
#pragma unroll
    for (int k = 0; k < 4; k++)
      x[k] = (i0 + k < m && lane < T.W) ? __ldcg(T.A + (int64_t)S.mem[i0 + k] * T.Ws + lane) : 0u;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      uint32_t mine = 0;
#pragma unroll
      for (int w = 0; w < NW; w++) {
        const uint32_t y = __shfl_sync(FULL, x[k], (at[w] < 0 ? 0 : at[w]) >> 5);
        const unsigned word = __ballot_sync(FULL, at[w] >= 0 && ((y >> (at[w] & 31)) & 1u));
        if (lane == w) mine = word;
      }
      if (i0 + k < m && lane < NW) S.A[(i0 + k) * NW + lane] = mine;
    }
  }
  __syncwarp();
}

// Candidates that can be in a clique larger than omega with T's clique: omega
// + 1 - cs of them are needed, each with at least omega - cs neighbours among
// them; the others are dropped until none is.  Returns how many are left (0:
// decided; a maximal clique {u} + C larger than omega was raised).  Their
// positions are left in S.A.
__device__ int prune_candidates(const SA &a, const TaskCtx &T, Bits<1> &P, TaskSmem &S) {
  const int lane = threadIdx.x & 31;
  const int om = read_best(a.best, T.g);
  // the candidates' list uses the matrix's space, which is not built yet; lane
  // i takes every 32nd candidate
  int *lst = (int *)S.A;
  for (;;) {
    const int cnt = __popc(P.w[0]);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    const int m = __shfl_sync(FULL, incl, 31);
    if (T.cs + m <= om) return 0;
    if (m == 0) {
      dev::raise_incumbent(a.best, a.lock, a.wit, a.voff, T.g, T.cs, a.err, a.spin,
                           [&](int, int32_t *base) { write_task_clique(base, a, T, S.mem, nullptr, 0, -1); });
      return 0;
    }
    __syncwarp();
    S.bits[lane] = P.w[0];
    S.drop[lane] = 0;
    int slot = incl - cnt;
    for (uint32_t x = P.w[0]; x; x &= x - 1) lst[slot++] = 32 * lane + __ffs(x) - 1;
    __syncwarp();
    for (int i = lane; i < m; i += 32) {
      const int pos = lst[i];
      const uint32_t *row = T.A + (int64_t)pos * T.Ws;
      int deg = 0;
#pragma unroll 4
      for (int w = 0; w < T.W; w++) deg += __popc(__ldcg(row + w) & S.bits[w]);
      if (deg < om - T.cs) atomicOr(&S.drop[pos >> 5], 1u << (pos & 31));
    }
    __syncwarp();
    const uint32_t dr = S.drop[lane];
    if (!__any_sync(FULL, dr != 0)) return m;
    P.w[0] &= ~dr;
  }
}

// Search T's clique with its m pruned candidates (at most kTM) on a compact
// matrix, in the order of the record's positions (the root's minimum-width
// order): the colouring takes the densest first, the branching the sparsest.
__device__ __forceinline__ void search_compact(const SA &a, const TaskCtx &T, int m, TaskSmem &S, uint32_t *stk,
                                               unsigned long long &nodes, unsigned long long &don) {
  const int lane = threadIdx.x & 31;
  const int *lst = (const int *)S.A;
  for (int i = lane; i < m; i += 32) S.mem[i] = lst[i];
  __syncwarp();  // the list is read before the matrix takes its place
  if (m <= 128) {
    compact_matrix<4>(T, S, m);
    task_dfs<4>(a, T, S, stk, m, nodes, don);
  } else {
    compact_matrix<8>(T, S, m);
    task_dfs<8>(a, T, S, stk, m, nodes, don);
  }
}

// One task (all lanes): clique T.C, candidates P (a word per lane).  Nodes of
// more than kTM candidates are searched depth first on the arena's matrix (a
// set word per lane, rows of one 128-byte line), until a child fits the
// compact form.
__device__ void run_task(const SA &a, TaskCtx &T, Bits<1> P, TaskSmem &S, uint32_t *stk, unsigned long long &nodes,
                         unsigned long long &don) {
  const int lane = threadIdx.x & 31;
  T.nlev = 0;
  for (;;) {
    // a new node: P with T's clique
    const int m = prune_candidates(a, T, P, S);
    if (m > kTM) {
      uint32_t *q = T.lev + (int64_t)T.nlev * kBigLev;
      q[lane] = P.w[0];
      if (lane == 0) q[64] = (uint32_t)-1;  // not coloured yet
      T.nlev++;
    } else {
      if (m > 0) search_compact(a, T, m, S, stk, nodes, don);
      if (T.nlev == 0) return;
      Bits<1> C;
      C.w[0] = T.C;
      bclear(C, level_word(T.lev + (int64_t)(T.nlev - 1) * kBigLev + 65));
      T.C = C.w[0];
      T.cs--;
    }
    // the next branch of the deepest level that has one
    for (;;) {
      __syncwarp();
      if (__shfl_sync(FULL, lane == 0 ? *(volatile int32_t *)a.err : 0, 0)) return;
      uint32_t *q = T.lev + (int64_t)(T.nlev - 1) * kBigLev;
      Bits<1> LP, LB;
      LP.w[0] = q[lane];
      LB.w[0] = q[32 + lane];
      const int om = read_best(a.best, T.g);
      if (om > level_word(q + 64)) {
        color_ise<1, false>(T.A, T.Ws, T.W, LP, om - T.cs, LB);
        __syncwarp();
        q[32 + lane] = LB.w[0];
        if (lane == 0) q[64] = (uint32_t)om;
        __syncwarp();
      }
      int hungry = 0;
      if (lane == 0) hungry = *(volatile int32_t *)a.task_next > *(volatile int32_t *)a.ntasks;
      if (__shfl_sync(FULL, hungry, 0)) {
        const int k = offer_big(a, T, T.nlev - 1);  // the deepest level has chosen none yet
        don += (unsigned long long)k;
        LB.w[0] = q[32 + lane];
      }
      const int v = bhighest(LB);
      if (v >= 0) {
        bclear(LB, v);
        bclear(LP, v);
        q[lane] = LP.w[0];
        q[32 + lane] = LB.w[0];
        if (lane == 0) q[65] = (uint32_t)v;
        __syncwarp();
        P = LP;
        band_row<1, false>(P, T.A, T.Ws, T.W, v);
        nodes++;
        if (lane == 0) atomicAdd(a.progress, 1);  // (a node of this size takes 10 us and more)
        Bits<1> C;
        C.w[0] = T.C;
        bset(C, v);
        T.C = C.w[0];
        T.cs++;
        break;
      }
      if (--T.nlev == 0) return;
      Bits<1> C;
      C.w[0] = T.C;
      bclear(C, level_word(T.lev + (int64_t)(T.nlev - 1) * kBigLev + 65));
      T.C = C.w[0];
      T.cs--;
    }
  }
}

// The task kernel: every warp takes a ticket (a queue position) and waits for
// the task at that position; tickets beyond the last published task are the
// waiting warps, which the searching warps see and hand branches to.  The
// wait is on the position's own word, so waiting warps do not contend.  It
// ends when no published task is unfinished (pending is 0): nothing can be
// published then.
__global__ void __launch_bounds__(kTW * 32, 4) branch_task_kernel(SA a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  TaskSmem &S = ((TaskSmem *)smem)[wib];
  uint32_t *lev = a.stack + ((int64_t)blockIdx.x * kTW + wib) * a.stack_stride;
  uint32_t *stk = lev + a.small_stack;
  unsigned long long nodes = 0, don = 0;
  for (;;) {
    __syncwarp();
    int got = -1;
    if (lane == 0 && *(volatile int32_t *)a.pending > 0) {
      const int t = atomicAdd(a.task_next, 1);
      const int slot = t & (a.task_cap - 1), lap2 = 2 * (t / a.task_cap);
      long long waited = 0;
      unsigned ns = 64, polls = 0;
      int last = -1;
      for (;;) {
        if (*(volatile int32_t *)(a.ready + slot) == lap2 + 1) {
          got = t;
          break;
        }
        if (*(volatile int32_t *)a.pending == 0) break;
        if ((polls++ & 15) == 0) {
          if (*(volatile int32_t *)a.err) break;
          const int prog = *(volatile int32_t *)a.progress + *(volatile int32_t *)a.ntasks;
          if (prog != last) {
            last = prog;
            waited = 0;
          }
        }
        waited += ns >> 6;
        if (waited > a.spin) {
          atomicExch(a.err, kDevTimeout);
          break;
        }
        __nanosleep(ns);
        if (ns < 4096) ns <<= 1;
      }
      __threadfence();
    }
    got = __shfl_sync(FULL, got, 0);
    if (got < 0) break;
    const int slot = got & (a.task_cap - 1);
    const uint32_t *tk = a.tasks + (int64_t)slot * kTaskWords;
    TaskCtx T;
    T.lev = lev;
    Bits<1> P;
    T.rec = (int)__ldcg(tk + 0);
    T.cs = (int)__ldcg(tk + 1);
    T.C = __ldcg(tk + 2 + lane);
    P.w[0] = __ldcg(tk + 34 + lane);
    __syncwarp();
    if (lane == 0) {
      __threadfence();
      atomicExch(a.ready + slot, 2 * (got / a.task_cap) + 2);  // free for the next lap's writer
    }
    if (T.cs > 0) {
      const int *rp = (const int *)(a.recs + T.rec);
      T.u = __ldcg(rp + 0);
      T.g = __ldcg(rp + 1);
      T.p = __ldcg(rp + 2);
      T.W = __ldcg(rp + 3);
      T.Ws = __ldcg(rp + 4);
      T.A = a.arena + __ldcg((const long long *)(rp + 6));
      T.Pidx = (const int *)(T.A + (int64_t)T.p * T.Ws);
      run_task(a, T, P, S, stk, nodes, don);
    }
    __syncwarp();
    if (lane == 0) {
      __threadfence();
      atomicSub(a.pending, 1);
    }
  }
  if (lane == 0) {
    atomicAdd(a.counters + 2, nodes);
    atomicAdd(a.counters + 3, don);
  }
}

}  // namespace

int launch_search(mc_graph *g, const Pruned &pg, int no_neigh_cores, int no_split, int split_nodes,
                  long long spin_limit, SearchCounters *cnt, int layout, int no_bitmap, bool same_graph) {
  // Persistent kernels with fixed grids; the root counts are read on the
  // device (pg.d_counts), and sizes are bounded by K(G) >= |N+(u)|, so the
  // launches need no host synchronisation.
  void *p;
  MC_TRY(ws_get(g, "se.ctr", kCtrBytes, &p));
  // [0..5] colored, branched, nodes, donations, row entries read by warp
  // workers, by block workers; [8..9] four root queue heads, [12] a fifth;
  // [10] arena words used; [11] records; [14], [15] roots left to the wider
  // launches;
  // the queue's hot words on 128-byte lines of their own: [32] tasks, [48]
  // tickets, [64] unfinished tasks, [80] heartbeat
  unsigned long long *ctr = (unsigned long long *)p;
  int32_t *next = (int32_t *)(ctr + 8);
  MC_CUDA_TRY(cudaMemsetAsync(ctr, 0, kCtrBytes, g->stream));
  SA a{};
  a.np_count = pg.d_counts;
  a.use_bitmap = no_bitmap ? 0 : 1;
  a.orow = pg.orow;
  a.ocol = pg.ocol;
  a.ocore = pg.ocore;
  a.oold = pg.oold;
  a.ogid = pg.ogid;
  a.best = g->best;
  a.lock = g->lock;
  a.wit = g->wit;
  a.voff = g->gid ? g->voff : nullptr;
  a.err = g->err;
  a.spin = spin_limit;
  a.neigh_cores = no_neigh_cores ? 0 : 1;
  a.counters = ctr;
  // |P| <= |N+(u)| <= K(u) <= K(G); roots above kBigCap are not in any of
  // the lists launched here (single graphs solve them as induced subgraphs;
  // a batch with such a graph is refused before anything is launched)
  if (g->count > 1 && g->max_core > kBigCap) return MC_ERR_UNSUPPORTED;
  const int kbound = std::min(std::max(g->max_core, 1), kBigCap);
  const int wmax = g->warp_max_used;
  if (!no_split) {
    // queue sizes grow with the graph (a small graph gets a small queue; a
    // full queue only keeps work where it is)
    const long long arena_words = std::min<long long>(kArenaWords, std::max<long long>(1ll << 18, 4 * g->nnz));
    const int rec_cap = (int)std::min<int64_t>(kRecCap, std::max<int64_t>(1024, g->n));
    int task_cap = 1 << 12;
    while (task_cap < kTaskCap && (int64_t)task_cap < 4 * g->n) task_cap <<= 1;
    MC_TRY(ws_get(g, "se.arena", (size_t)arena_words * 4, &p));
    a.arena = (uint32_t *)p;
    a.arena_cap = arena_words;
    a.arena_used = ctr + 10;
    MC_TRY(ws_get(g, "se.recs", (size_t)rec_cap * sizeof(RootRec), &p));
    a.recs = (RootRec *)p;
    a.rec_cap = rec_cap;
    a.nrec = (int32_t *)(ctr + 11);
    MC_TRY(ws_get(g, "se.tasks", (size_t)task_cap * kTaskWords * 4, &p));
    a.tasks = (uint32_t *)p;
    MC_TRY(ws_get(g, "se.ready", (size_t)task_cap * 4, &p));
    a.ready = (int32_t *)p;
    MC_CUDA_TRY(cudaMemsetAsync(a.ready, 0, (size_t)task_cap * 4, g->stream));
    a.task_cap = task_cap;
    a.ntasks = (int32_t *)(ctr + 32);
    a.task_next = (int32_t *)(ctr + 48);
    a.pending = (int32_t *)(ctr + 64);
    a.progress = (int32_t *)(ctr + 80);
    a.offer_nodes = split_nodes > 0 ? split_nodes : kOfferNodes;
  }
  // Block workers (shared-memory matrices): a 512-candidate launch first,
  // then a 1,024-candidate launch over the roots it could not hold.
  using LB = BlockLayout<1, true>;
  using LM = BlockLayout<1, true, kMidCap>;
  const size_t smem_b = LB::bytes, smem_m = LM::bytes;
  MC_CUDA_TRY(cudaFuncSetAttribute(search_block_kernel<1, true, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)smem_b));
  MC_CUDA_TRY(cudaFuncSetAttribute(search_block_kernel<1, true, kMidCap>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)smem_m));
  const size_t smem_t = kTW * sizeof(TaskSmem);
  MC_CUDA_TRY(cudaFuncSetAttribute(branch_task_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_t));
  int per_sm_b = 0, per_sm_t = 0, per_sm_m = 0;
  MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_b, search_block_kernel<1, true, 1024>, kBT, smem_b));
  MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_t, branch_task_kernel, kTW * 32, smem_t));
  MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_m, search_block_kernel<1, true, kMidCap>, kBT,
                                                            smem_m));
  if (per_sm_b < 1 || per_sm_m < 1 || per_sm_t < 1) return MC_ERR_CUDA;
  // grids (and the stacks sized by them) shrink for small graphs: a block
  // per 64 vertices at most, a warp per four vertices in the warp class
  const int64_t small_cap = std::max<int64_t>(1, (g->n + 63) / 64);
  const int blocks_b = (int)std::min<int64_t>((int64_t)g->sm_count * per_sm_b, small_cap);
  const int blocks_m = (int)std::min<int64_t>((int64_t)g->sm_count * per_sm_m, small_cap);
  const int blocks_t = (int)std::min<int64_t>((int64_t)g->sm_count * per_sm_t, std::max<int64_t>(1, (g->n + 15) / 16));
  a.task_warps = g->sm_count * per_sm_t * kTW;
  const int64_t stride_b = (int64_t)(std::min(kbound, 1024) + 2) * (64 + 2);
  const int64_t stride_m = (int64_t)(std::min(kbound, kMidCap) + 2) * (64 + 2);
  // levels above the compact form, then those of the compact form (uint4)
  const int64_t stride_t = ((stride_b + 3) & ~(int64_t)3) + (int64_t)kTStk * (std::min(kbound, kTM) + 2);
  uint32_t *stk_b = nullptr, *stk_t = nullptr;
  if (kbound > wmax) {
    MC_TRY(ws_get(g, "se.stk_b", (size_t)blocks_b * kBW * stride_b * 4, &p));
    stk_b = (uint32_t *)p;
  }
  if (!no_split) {
    MC_TRY(ws_get(g, "se.stk_t", (size_t)blocks_t * kTW * stride_t * 4, &p));
    stk_t = (uint32_t *)p;
  }

  if (kbound > wmax) {  // also for roots that find the queue or the arena full
    const int cap = std::min(kbound, 1024);
    a.sort_stride = (int64_t)cap * (((cap + 31) / 32) | 1) + cap;
    const int blocks = std::max({blocks_b, blocks_m, g->sm_count * 2});
    MC_TRY(ws_get(g, "se.sort", (size_t)blocks * a.sort_stride * 4, &p));
    a.sort = (uint32_t *)p;
  }
  // one graph's block workers gather their matrices from dense rows; the
  // builder's time counts with theirs
  const bool dense = g->count == 1 && !no_bitmap && kbound > wmax;
  if (dense) {
    // a block root has more than wmax later neighbours, so K > wmax from its rank on:
    // at most one vertex per wmax + 1 entries
    const int64_t useful = std::min(g->n, g->nnz / (wmax + 1) + 1);
    a.dense_cap = (int32_t)std::min(kDenseCap, (useful + 31) & ~(int64_t)31);
    a.dense_stride = a.dense_cap / 32;
    MC_TRY(ws_get(g, "se.dense", (size_t)a.dense_cap * a.dense_stride * 4, &p));
    a.dense = (const uint32_t *)p;
  }

  // block class first (largest trees), then big, then warp class, then the
  // tasks the first and last of these published; events 8-12 time each
  MC_TRY(record_event(g, 8));
  if (dense && !same_graph) {
    const size_t smem = (size_t)kDW * a.dense_stride * 4;
    MC_CUDA_TRY(cudaFuncSetAttribute(dense_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    dense_rows_kernel<<<(int)std::min<int64_t>((int64_t)g->sm_count * 4, (g->n + kDW - 1) / kDW), kDW * 32, smem,
                        g->stream>>>(pg.d_counts, pg.orow, pg.ocol, a.dense_cap, a.dense_stride, (uint32_t *)a.dense);
    g_launches++;
    MC_CUDA_TRY(cudaGetLastError());
  }
  if (kbound > wmax) {
    a.gmat = nullptr;
    a.roots = pg.roots_block;
    a.nroots = pg.d_counts + 4;
    a.next = next + 0;
    const bool wide_only = layout == 1 && kbound > kMidCap;
    if (wide_only) {
      // every block-class root in the 1,024-candidate layout
      a.stack = stk_b;
      a.stack_stride = stride_b;
      search_block_kernel<1, true, 1024><<<blocks_b, kBT, smem_b, g->stream>>>(a);
      g_launches++;
      MC_CUDA_TRY(cudaGetLastError());
    } else {
      if (kbound > kMidCap) {
        MC_TRY(ws_get(g, "se.ovf", (size_t)std::max<int64_t>(g->n, 1) * 4, &p));
        a.overflow = (int32_t *)p;
        a.noverflow = (int64_t *)(ctr + 14);
      }
      MC_TRY(ws_get(g, "se.stk_m", (size_t)blocks_m * kBW * stride_m * 4, &p));
      a.stack = (uint32_t *)p;
      a.stack_stride = stride_m;
      search_block_kernel<1, true, kMidCap><<<blocks_m, kBT, smem_m, g->stream>>>(a);
      g_launches++;
      MC_CUDA_TRY(cudaGetLastError());
      if (kbound > kMidCap) {
        a.roots = a.overflow;
        a.nroots = a.noverflow;
        if (dense) {
          // roots of up to kWideCap candidates on the dense rows: without the
          // lookup structures two blocks fit an SM
          using LW = BlockLayout<1, true, kWideCap, true>;
          int per_sm_w = 0;
          MC_CUDA_TRY(cudaFuncSetAttribute(search_block_kernel<1, true, kWideCap, true>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LW::bytes));
          MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
              &per_sm_w, search_block_kernel<1, true, kWideCap, true>, kBT, LW::bytes));
          const int blocks_w = (int)std::min<int64_t>((int64_t)g->sm_count * std::max(per_sm_w, 1), small_cap);
          MC_TRY(ws_get(g, "se.ovf2", (size_t)std::max<int64_t>(g->n, 1) * 4, &p));
          a.overflow = (int32_t *)p;
          a.noverflow = (int64_t *)(ctr + 15);
          a.next = (int32_t *)(ctr + 12);
          MC_TRY(ws_get(g, "se.stk_x", (size_t)blocks_w * kBW * stride_b * 4, &p));
          a.stack = (uint32_t *)p;
          a.stack_stride = stride_b;
          search_block_kernel<1, true, kWideCap, true><<<blocks_w, kBT, LW::bytes, g->stream>>>(a);
          g_launches++;
          MC_CUDA_TRY(cudaGetLastError());
          a.roots = a.overflow;
          a.nroots = a.noverflow;
        }
        a.next = next + 3;
        a.overflow = nullptr;
        a.noverflow = nullptr;
        a.stack = stk_b;
        a.stack_stride = stride_b;
        search_block_kernel<1, true, 1024><<<blocks_b, kBT, smem_b, g->stream>>>(a);
        g_launches++;
        MC_CUDA_TRY(cudaGetLastError());
      }
    }
  }
  MC_TRY(record_event(g, 9));
  if (kbound > 1024) {
    using L = BlockLayout<4, false>;
    const size_t smem = L::bytes;
    MC_CUDA_TRY(cudaFuncSetAttribute(search_block_kernel<4, false, 4096>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
    const int blocks = g->sm_count;
    const int pmax = kbound;
    a.stack_stride = (int64_t)(pmax + 2) * (64 * 4 + 2);
    MC_TRY(ws_get(g, "se.stk_g", (size_t)blocks * kBW * a.stack_stride * 4, &p));
    a.stack = (uint32_t *)p;
    const int Wm = (pmax + 31) / 32;
    a.gmat_stride = (int64_t)pmax * (Wm | 1) + 64;
    MC_TRY(ws_get(g, "se.gmat", (size_t)blocks * a.gmat_stride * 4, &p));
    a.gmat = (uint32_t *)p;
    a.roots = pg.roots_big;
    a.nroots = pg.d_counts + 5;
    a.next = next + 1;
    search_block_kernel<4, false, 4096><<<blocks, kBT, smem, g->stream>>>(a);
    g_launches++;
    MC_CUDA_TRY(cudaGetLastError());
  }
  MC_TRY(record_event(g, 10));
  {
    int per_sm = 0;
    MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, search_warp_kernel, kSW * 32, 0));
    if (per_sm < 1) return MC_ERR_CUDA;
    const int blocks = (int)std::min<int64_t>((int64_t)g->sm_count * per_sm,
                                              std::max<int64_t>(1, (g->n + 4 * kSW - 1) / (4 * kSW)));
    const int pmax = std::min(kbound, kWarpCap);
    a.stack_stride = (int64_t)(pmax + 2) * (64 + 2);
    MC_TRY(ws_get(g, "se.stk_w", (size_t)blocks * kSW * a.stack_stride * 4, &p));
    a.stack = (uint32_t *)p;
    a.roots = pg.roots_small;
    a.nroots = pg.d_counts + 3;
    a.next = next + 2;
    search_warp_kernel<<<blocks, kSW * 32, 0, g->stream>>>(a);
    g_launches++;
    MC_CUDA_TRY(cudaGetLastError());
  }
  MC_TRY(record_event(g, 11));
  if (!no_split) {
    a.stack_stride = stride_t;
    a.small_stack = (stride_b + 3) & ~(int64_t)3;
    a.stack = stk_t;
    branch_task_kernel<<<blocks_t, kTW * 32, smem_t, g->stream>>>(a);
    g_launches++;
    MC_CUDA_TRY(cudaGetLastError());
  }
  MC_TRY(record_event(g, 12));
  cnt->d_counters = ctr;
  return MC_OK;
}

int read_search_counters(mc_graph *g, SearchCounters *cnt) {
  unsigned long long *h = (unsigned long long *)g->h_small;
  MC_CUDA_TRY(cudaMemcpyAsync(h, cnt->d_counters, 33 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, g->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
  cnt->roots_colored = h[0];
  cnt->roots_branched = h[1];
  cnt->nodes = h[2];
  cnt->donations = h[3];
  cnt->entries = h[4] + h[5];
  cnt->entries_block = h[5];
  cnt->tasks = (unsigned long long)*(const int32_t *)(h + 32);
  return MC_OK;
}

}  // namespace mc
