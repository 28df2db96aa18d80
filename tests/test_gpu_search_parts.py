"""Single device functions of the search and the heuristic, called by themselves: a
small library that includes search.cu and heuristic.cu is compiled here and linked
against libmc.so."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SRC = r"""
#include "%s"
using namespace mc;

// Requests of one record each (words[i] candidates, 1 word per row): their
// results, taken in turn by one thread.
__global__ void records_kernel(SA a, int n, const int *cand, int *out) {
  for (int i = 0; i < n; i++) {
    long long off = -1;
    out[2 * i] = reserve_record(a, Root{0, 0, nullptr, cand[i]}, 1, &off);
    out[2 * i + 1] = (int)off;
  }
}
extern "C" int t_records(int n, const int *cand, int *out, uint32_t *arena, long long cap, unsigned long long *used,
                         void *recs, int rec_cap, int *nrec) {
  SA a{};
  a.arena = arena;
  a.arena_cap = cap;
  a.arena_used = used;
  a.recs = (RootRec *)recs;
  a.rec_cap = rec_cap;
  a.nrec = nrec;
  records_kernel<<<1, 1>>>(a, n, cand, out);
  return (int)cudaDeviceSynchronize();
}

// One warp's task on a compact matrix A (m rows of 4 words), d levels in stk,
// the sets P, B of the current one in pb: what offer_level leaves of them, and
// what it returns.
__global__ void offer_kernel(SA a, const uint32_t *A, int m, uint32_t *stk, int d, uint32_t *pb, int *k) {
  __shared__ __align__(16) TaskSmem S;
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < 4 * m; i += 32) S.A[i] = A[i];
  for (int i = lane; i < m; i += 32) S.mem[i] = i;
  __syncwarp();
  TaskCtx T{};
  T.cs = 1;
  Set<4> P = sload<4>(pb), B = sload<4>(pb + 4);
  __syncwarp();
  const int r = offer_level<4>(a, T, S, stk, d, P, B);
  if (lane == 0) {
    sstore<4>(pb, P);
    sstore<4>(pb + 4, B);
    *k = r;
  }
}
// The same for offer_big: levels of 66 words in lev, matrix of ws words a row.
__global__ void offer_big_kernel(SA a, const uint32_t *A, int m, int ws, uint32_t *lev, int nlev, int *k) {
  TaskCtx T{};
  T.cs = 1 + nlev;
  T.p = m;
  T.W = (m + 31) / 32;
  T.Ws = ws;
  T.A = A;
  T.lev = lev;
  T.nlev = nlev;
  const int r = offer_big(a, T, nlev);
  if ((threadIdx.x & 31) == 0) *k = r;
}
// ctr: best, tasks, tickets, pending, error; the queue has 256 places
extern "C" int t_offer(int big, const uint32_t *A, int m, int ws, uint32_t *stk, int d, uint32_t *pb, int *k, int *ctr,
                       uint32_t *tasks, int *ready) {
  SA a{};
  a.best = ctr;
  a.ntasks = ctr + 1;
  a.task_next = ctr + 2;
  a.pending = ctr + 3;
  a.err = ctr + 4;
  a.tasks = tasks;
  a.ready = ready;
  a.task_cap = 256;
  a.spin = 1000;
  if (big) offer_big_kernel<<<1, 32>>>(a, A, m, ws, stk, d, k);
  else offer_kernel<<<1, 32>>>(a, A, m, stk, d, pb, k);
  return (int)cudaDeviceSynchronize();
}
// One task of m candidates on the matrix A (ws words a row): run_task by one warp.
__global__ void run_kernel(SA a, const uint32_t *A, int m, int ws, uint32_t *lev, uint32_t *stk,
                           unsigned long long *out) {
  __shared__ __align__(16) TaskSmem S;
  TaskCtx T{};
  T.cs = 1;
  T.p = m;
  T.W = (m + 31) / 32;
  T.Ws = ws;
  T.A = A;
  T.lev = lev;
  Bits<1> P;
  P.w[0] = first_bits(m);
  unsigned long long nodes = 0, don = 0;
  run_task(a, T, P, S, stk, nodes, don);
  if ((threadIdx.x & 31) == 0) out[0] = nodes;
}
// ctr: best, tasks, tickets, error, progress
extern "C" int t_run(const uint32_t *A, int m, int ws, uint32_t *lev, uint32_t *stk, int *ctr,
                     unsigned long long *out) {
  SA a{};
  a.best = ctr;
  a.ntasks = ctr + 1;
  a.task_next = ctr + 2;
  a.err = ctr + 3;
  a.progress = ctr + 4;
  a.spin = 1000;
  a.offer_nodes = 8;
  run_kernel<<<1, 32>>>(a, A, m, ws, lev, stk, out);
  return (int)cudaDeviceSynchronize();
}
extern "C" long long t_ws_bytes(mc_graph *g, const char *name) {
  auto it = g->ws.find(name);
  return it == g->ws.end() ? -1 : (long long)it->second.bytes;
}
"""


@pytest.fixture(scope="module")
def mc():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_1302_6256_gb300 as m
    m.load_library()
    return m


@pytest.fixture(scope="module")
def lib(mc, tmp_path_factory):
    from paper_1302_6256_gb300 import _build
    d = tmp_path_factory.mktemp("parts")
    src, out = str(d / "parts.cu"), str(d / "libparts.so")
    with open(src, "w") as f:
        f.write(SRC % os.path.join(_build.CSRC, "search.cu"))
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", src, "-o", out, _build.LIB, "-lcudart",
                    "-Xlinker", "-rpath=" + _build.BUILD], check=True)
    return ctypes.CDLL(out)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def test_record_that_does_not_fit_takes_nothing(lib):
    """Room of 512 words (a record of c candidates takes 2 c, rounded up to 32):
    320 words, then one of 256 that does not fit, then two of 64 that do, then
    none of 128, then the last 64."""
    cand = torch.tensor([160, 128, 32, 32, 64, 32, 16], dtype=torch.int32, device="cuda")
    out = torch.zeros(14, dtype=torch.int32, device="cuda")
    arena = torch.zeros(512, dtype=torch.int32, device="cuda")
    used, nrec = (torch.zeros(2, dtype=torch.int64, device="cuda") for _ in range(2))
    recs = torch.zeros(64 * 8, dtype=torch.int32, device="cuda")
    lib.t_records.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong,
                              ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    assert lib.t_records(7, _p(cand), _p(out), _p(arena), 512, _p(used), _p(recs), 64, _p(nrec)) == 0
    assert out.view(7, 2).tolist() == [[0, 0], [-1, -1], [1, 320], [2, 384], [-1, -1], [3, 448], [-1, -1]]


def test_full_arena_keeps_the_search_order(mc, lib):
    """Block roots of a dense graph overflow the arena (4 words per CSR entry;
    a root of 400 candidates takes 5,600).  Those searched in place have the
    room to be put in minimum-width order first, and omega is kept."""
    g = gg.relabel(gg.erdos_renyi(1000, 0.4, planted=28, seed=1), 3)
    h = mc.mc_load_csr(torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col_idx).cuda(), mc.MC_VALIDATE)
    for opts in (dict(), dict(heuristic=2), dict(no_bitmap=True), dict(layout=1)):
        om, wit, st = mc.mc_max_clique(h, **opts)
        assert om == 28 and oracle.is_clique(g, wit)
        assert st["max_core"] > 256 and st["roots_branched"] > 100
    lib.t_ws_bytes.argtypes, lib.t_ws_bytes.restype = [ctypes.c_void_p, ctypes.c_char_p], ctypes.c_longlong
    cap = st["max_core"]
    assert lib.t_ws_bytes(h.handle, b"se.sort") >= 4 * (cap * (((cap + 31) // 32) | 1) + cap)
    h.close()


def _words(members, n):
    w = np.zeros(n, np.uint32)
    for x in members:
        w[x >> 5] |= np.uint32(1) << np.uint32(x & 31)
    return w


def _members(words):
    return {32 * i + b for i, w in enumerate(words) for b in range(32) if (int(w) >> b) & 1}


@pytest.mark.parametrize("big", [False, True])
@pytest.mark.parametrize("level", [0, 2, 3])
def test_handed_over_branches_leave_their_level(lib, big, level):
    """Four levels (three stored and the current one; in the large form all
    stored), of which those from `level` on have untried branches.  The first
    of these hands over every branch x with its candidates (x's neighbours
    among the candidates that no branch before x took), and keeps neither the
    branches nor, as candidates, the vertices: a later colouring of the level
    cannot bring them back.  The other levels stay as they are."""
    rng = np.random.default_rng(10 * level + big)
    m, ws, sw = (300, 11, 32) if big else (100, 4, 4)
    adj = np.triu(rng.random((m, m)) < 0.5, 1)
    adj |= adj.T
    A = np.stack([_words(np.nonzero(r)[0], ws) for r in adj])
    P = [set(rng.choice(m, m // 2, replace=False).tolist()) for _ in range(4)]
    B = [set(rng.choice(sorted(p), 9 + l, replace=False).tolist()) if l >= level else set() for l, p in enumerate(P)]
    chosen = [int(v) for v in rng.choice(m, 4, replace=False)]
    if big:
        stk = np.zeros((4, 66), np.uint32)
        for l in range(4):
            stk[l, :32], stk[l, 32:64], stk[l, 65] = _words(P[l], 32), _words(B[l], 32), chosen[l]
        pb = np.zeros(8, np.uint32)
    else:
        stk = np.zeros((3, 20), np.uint32)
        for l in range(3):
            stk[l, :4], stk[l, 8:12], stk[l, 17] = _words(P[l], 4), _words(B[l], 4), chosen[l]
        pb = np.concatenate([_words(P[3], 4), _words(B[3], 4)])
    dev = [torch.from_numpy(x.view(np.int32)).cuda() for x in (A.reshape(-1), stk.reshape(-1), pb)]
    k, ctr = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(5, dtype=torch.int32, device="cuda")
    ctr[0] = 1000  # no clique found here is larger
    tasks, ready = torch.zeros(256 * 66, dtype=torch.int32, device="cuda"), torch.zeros(256, dtype=torch.int32, device="cuda")
    i, p = ctypes.c_int, ctypes.c_void_p
    lib.t_offer.argtypes = [i, p, i, i, p, i, p, p, p, p, p]
    assert lib.t_offer(int(big), _p(dev[0]), m, ws, _p(dev[1]), 4 if big else 3, _p(dev[2]), _p(k), _p(ctr), _p(tasks),
                       _p(ready)) == 0
    assert int(k) == len(B[level]) and ctr.tolist() == [1000, len(B[level]), 0, len(B[level]), 0]
    got, q = dev[1].cpu().numpy().view(np.uint32).reshape(stk.shape), dev[2].cpu().numpy().view(np.uint32)
    for l in range(4):
        if big:
            g = _members(got[l, :32]), _members(got[l, 32:64])
        else:
            g = (_members(got[l, :4]), _members(got[l, 8:12])) if l < 3 else (_members(q[:4]), _members(q[4:]))
        assert g == ((P[l] - B[l], set()) if l == level else (P[l], B[l])), l
    t = tasks.cpu().numpy().view(np.uint32).reshape(256, 66)
    left = set(P[level])
    for n, x in enumerate(sorted(B[level], reverse=True)):
        left.discard(x)
        assert _members(t[n, 34:]) == left & set(np.nonzero(adj[x])[0].tolist())
        assert x in _members(t[n, 2:34])


def test_bit_rows_take_room_for_ranks_that_can_use_them(mc, lib):
    """A root of more than warp_max candidates has K > warp_max, and so have all
    later ranks; those are at most one vertex per warp_max + 1 entries.  60,000
    vertices of 8 neighbours and a dense part take rows for 4,036 ranks (2 MB), not
    for 40,960 (210 MB); the search is the same as over lookups."""
    r = np.random.default_rng(3)
    s, t = r.integers(0, 60000, (2, 220000))
    d = gg.erdos_renyi(400, 0.5, planted=30, seed=2)
    ds = np.repeat(np.arange(400), d.degrees())
    g = gg.from_edges(60000, np.r_[s[s != t], ds], np.r_[t[s != t], d.col_idx])
    h = mc.mc_load_csr(torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col_idx).cuda(), mc.MC_VALIDATE)
    for wm in (128, 16):
        om, wit, st = mc.mc_max_clique(h, warp_max=wm, heuristic=2)
        assert om == 30 == mc.mc_max_clique(h, warp_max=wm, no_bitmap=True)[0] and oracle.is_clique(g, wit)
        if wm == 128:
            assert st["max_core"] > 128
            ranks = g.nnz // 129 + 1 + 31
            assert lib.t_ws_bytes(h.handle, b"se.dense") <= 2 * (ranks * ranks // 8)
    h.close()


def test_every_large_node_is_a_sign_of_life(lib):
    """A task of 60 disjoint five-cycles (300 candidates) with omega 3: two colours
    leave one vertex of each cycle to branch on, and its two neighbours, which are
    not adjacent, are dropped at once.  60 nodes above the compact form, and as many
    heartbeats for the warps that wait."""
    m, ws = 300, 11
    A = np.zeros((m, ws), np.uint32)
    for v in range(m):
        c = v - v % 5
        A[v] = _words([c + (v + 1) % 5, c + (v + 4) % 5], ws)
    dev = [torch.from_numpy(A.reshape(-1).view(np.int32)).cuda()]
    dev += [torch.zeros(k, dtype=torch.int32, device="cuda") for k in (66 * 304, 20 * 304)]
    ctr = torch.tensor([3, 0, 0, 0, 0], dtype=torch.int32, device="cuda")
    out = torch.zeros(1, dtype=torch.int64, device="cuda")
    i, p = ctypes.c_int, ctypes.c_void_p
    lib.t_run.argtypes = [p, i, i, p, p, p, p]
    assert lib.t_run(_p(dev[0]), m, ws, _p(dev[1]), _p(dev[2]), _p(ctr), _p(out)) == 0
    assert int(out) == 60 and ctr.tolist() == [3, 0, 0, 0, 60]


TOP = r"""
#include "%s"
using namespace mc;
extern "C" int t_top(long long n, int ntop, const int *order, const int *core, const int64_t *rp, int *top) {
  top_kernel<<<kTop / kTopKeys, kTopT>>>(n, ntop, order, core, rp, top);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("n,ntop,degrees", [(4096, 4096, 5), (9000, 4096, 3000), (9000, 4095, 1 << 30), (50, 50, 4), (1, 1, 1)])
def test_front_of_the_visiting_order(mc, tmp_path, n, ntop, degrees):
    """The last ntop positions of the order by core number, then degree, then the
    later position: as numpy sorts them, ties and the largest degrees included."""
    from paper_1302_6256_gb300 import _build
    src, out = str(tmp_path / "top.cu"), str(tmp_path / "libtop.so")
    with open(src, "w") as f:
        f.write(TOP % os.path.join(_build.CSRC, "heuristic.cu"))
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", src, "-o", out, _build.LIB, "-lcudart",
                    "-Xlinker", "-rpath=" + _build.BUILD], check=True)
    lib = ctypes.CDLL(out)
    r = np.random.default_rng(n + ntop)
    order, core = r.permutation(n).astype(np.int32), r.integers(0, 7, n).astype(np.int32)
    core[r.integers(0, n, 5)] = 270000
    deg = r.integers(0, degrees, n)
    rp = np.r_[0, np.cumsum(deg)].astype(np.int64)
    last = order[::-1][:ntop]
    want = last[np.lexsort((np.arange(ntop), -deg[last], -core[last]))]
    dev = [torch.from_numpy(x).cuda() for x in (order, core, rp)]
    top = torch.zeros(ntop, dtype=torch.int32, device="cuda")
    lib.t_top.argtypes = [ctypes.c_longlong, ctypes.c_int] + [ctypes.c_void_p] * 4
    assert lib.t_top(n, ntop, *(_p(x) for x in dev), _p(top)) == 0
    assert np.array_equal(top.cpu().numpy(), want)
