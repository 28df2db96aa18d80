"""Single device functions of the search, called by themselves: a small library
that includes search.cu is compiled here and linked against libmc.so."""
import ctypes
import os
import subprocess

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
