// Learned vertex ordering: per-vertex features and a 6 -> 64 -> 64 -> 1 MLP
// (ReLU, BF16 weights, FP32 accumulation, FP32 master weights and Adam).
// The score only orders the search's roots and seeds the heuristic; omega
// stays exact whatever the network predicts.
//
// Features of vertex v (d = degree, K = core number, Kmax = K(G), Dmax =
// maximum degree, c = number of neighbours with K >= K(v), Q = the first
// min(8, c) of those neighbours in increasing id):
//   f0 = log1p(d) / log1p(Dmax)        f3 = (chi + 1) / 9, chi = colours of
//   f1 = K(v) / Kmax                        the greedy colouring of G[Q] in
//   f2 = t / 28, t = edges among Q          increasing id (a bound on a
//                                           clique through v inside Q + v)
//   f4 = c / max(d, 1)                 f5 = log1p(c) / log1p(Dmax)
// A pass over the row gives c and Q (eight lanes, a warp or a block by its
// length), then eight lanes per vertex find the 28 pairs of Q by binary search
// in the shorter of the two rows and colour, one colour class per lane; fused
// with the network, it has eight hidden units per lane.
//
// Parameters, flat fp32 (4673): W1[64][6], b1[64], W2[64][64], b2[64],
// w3[64], b3.  Loss: binary cross-entropy on the logit s with weight
// pos_weight on positive labels, averaged over the rows.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <vector>

#include "mc_internal.cuh"

namespace mc {

constexpr int kF = 6, kH = 64;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kF, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH, kParams = kOffB3 + 1;

}  // namespace mc

struct mc_mlp {
  cudaStream_t stream = nullptr;
  int device = 0, sm_count = 0;
  float *master = nullptr;   // fp32 master parameters
  uint16_t *wbf = nullptr;   // bf16 copies of the weights (all parameters, same layout)
  float *grad = nullptr, *m = nullptr, *v = nullptr;
  float *loss = nullptr;     // device scalar
  float *part = nullptr;     // the gradient's sums per block; grad and loss follow them
  int part_blocks = 0;
  float *buf = nullptr;      // staging for host inputs
  size_t buf_bytes = 0;
  int64_t step = 0;
  void *h_small = nullptr;
};

namespace mc {
namespace {

__device__ __forceinline__ float bf16_to_f32(uint16_t h) { return __uint_as_float(((uint32_t)h) << 16); }

// round to nearest even
__host__ __device__ __forceinline__ uint16_t f32_to_bf16(float f) {
#ifdef __CUDA_ARCH__
  uint32_t x = __float_as_uint(f);
#else
  uint32_t x;
  memcpy(&x, &f, 4);
#endif
  if ((x & 0x7f800000u) == 0x7f800000u) return (uint16_t)(x >> 16);  // inf / nan
  uint32_t r = x + 0x7fffu + ((x >> 16) & 1u);
  return (uint16_t)(r >> 16);
}

constexpr int kQ = 8;  // neighbours of the triangle and colouring features

// Sub-warp primitive over the 8 lanes of a group (mask gm covers them).
__device__ __forceinline__ unsigned group_ballot(unsigned gm, bool x, int grp) {
  return (__ballot_sync(gm, x) >> (grp * 8)) & 0xFFu;
}

// Row lengths up to which a group of 8 lanes, a whole warp or (above) a block
// counts a vertex's row; entries that a lane has in flight.  With 8 lanes for
// every row the hubs' rows were the tail (R-MAT scale 18: 1.44 ms with 35% of
// the warps, 9 of 32 lanes active; 0.21 ms now).
constexpr int64_t kGroupRow = 256, kWarpRow = 4096;
constexpr int kRowFly = 4;

// Number of u in ci[e0, e1) with core[u] >= kv, counted by LANES lanes (gl =
// the lane's place among them, shift = their first lane, gm = their mask); the
// first kQ of them go to qs.
template <int LANES, int FLY>
__device__ int count_row(const int32_t *__restrict__ ci, const int32_t *__restrict__ core, int kv, int64_t e0,
                         int64_t e1, unsigned gm, int shift, int gl, int *qs) {
  constexpr unsigned all = LANES == 32 ? 0xffffffffu : (1u << (LANES & 31)) - 1u;
  const unsigned below = (1u << gl) - 1u;
  int c = 0;
  for (int64_t eb = e0; eb < e1; eb += LANES * FLY) {
    int u[FLY];
    bool ok[FLY];
#pragma unroll
    for (int i = 0; i < FLY; i++) {
      const int64_t e = eb + i * LANES + gl;
      u[i] = e < e1 ? ci[e] : -1;
    }
#pragma unroll
    for (int i = 0; i < FLY; i++) ok[i] = u[i] >= 0 && core[u[i]] >= kv;
#pragma unroll
    for (int i = 0; i < FLY; i++) {
      const unsigned m = (__ballot_sync(gm, ok[i]) >> shift) & all;
      const int pos = c + __popc(m & below);
      if (ok[i] && pos < kQ) qs[pos] = u[i];
      c += __popc(m);
    }
  }
  return c;
}

// The features from the row's length and count c, the edges t of G[Q] and its
// colours chi.
__device__ __forceinline__ void write_features(float kmax, float ldmax, int64_t deg, int kv, int c, int t, int chi,
                                               float f[kF]) {
  const float d = (float)deg;
  f[0] = log1pf(d) / ldmax;
  f[1] = (float)kv / kmax;
  f[2] = (float)t / (float)(kQ * (kQ - 1) / 2);
  f[3] = (float)(chi + 1) / (float)(kQ + 1);
  f[4] = (float)c / fmaxf(d, 1.f);
  f[5] = log1pf((float)c) / ldmax;
}

// The six features of vertex v (row [e0, e1), core number kv) from its count c
// and Q, by the 8 lanes of one group (every lane returns them).  The 28 pairs
// of Q are four per lane -- member gl with the members gl + 1 .. gl + 4, around
// -- and a lane's four binary searches run side by side.
__device__ void vertex_features(const int64_t *__restrict__ rp, const int32_t *__restrict__ ci, float kmax,
                                float ldmax, int64_t deg, int kv, int c, const int *qs, float f[kF]) {
  const int lane = threadIdx.x & 31, grp = lane >> 3, gl = lane & 7;
  const unsigned gm = 0xFFu << (grp * 8);
  const int q = min(c, kQ);
  const int me = gl < q ? qs[gl] : 0;
  const int64_t my0 = gl < q ? rp[me] : 0;
  const int myl = gl < q ? (int)(rp[me + 1] - my0) : 0;
  const int32_t *row[4];
  int key[4], left[4];
  uint32_t adj = 0u;  // bit i: member gl is adjacent to member gl + 1 + i
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int o = (gl + 1 + i) & 7;
    const int id = __shfl_sync(gm, me, o, 8), len = __shfl_sync(gm, myl, o, 8);
    const int64_t s0 = __shfl_sync(gm, my0, o, 8);
    // the shorter of the two rows
    const bool mine = myl < len || (myl == len && gl < o);
    row[i] = ci + (mine ? my0 : s0);
    key[i] = mine ? id : me;
    left[i] = (gl < q && o < q && (i < 3 || gl < 4)) ? (mine ? myl : len) : 0;
  }
  while ((left[0] | left[1] | left[2] | left[3]) != 0) {
    int x[4];
#pragma unroll
    for (int i = 0; i < 4; i++) x[i] = left[i] ? row[i][left[i] >> 1] : 0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      if (left[i] == 0) continue;
      const int h = left[i] >> 1;
      if (x[i] == key[i]) {
        adj |= 1u << i;
        left[i] = 0;
      } else if (x[i] < key[i]) {
        row[i] += h + 1;
        left[i] -= h + 1;
      } else {
        left[i] = h;
      }
    }
  }
  __syncwarp(gm);
  const int t = __reduce_add_sync(gm, __popc(adj));
  // row gl of G[Q]
  uint32_t nb = 0u;
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int p = (gl - 1 - i) & 7;
    const uint32_t theirs = __shfl_sync(gm, adj, p, 8);
    nb |= ((adj >> i) & 1u) << ((gl + 1 + i) & 7);
    nb |= ((theirs >> i) & 1u) << p;
  }
  // greedy colouring in index order: lane gl holds colour class gl; member
  // i joins the first class with none of its neighbours
  uint32_t cls = 0u;
  for (int i = 0; i < q; i++) {
    const uint32_t ai = __shfl_sync(gm, nb, i, 8);
    const unsigned clash = group_ballot(gm, (cls & ai) != 0u, grp);
    const int k = __ffs(~clash) - 1;
    if (gl == k) cls |= 1u << i;
  }
  write_features(kmax, ldmax, deg, kv, c, t, __popc(group_ballot(gm, cls != 0u, grp)), f);
}

// The same for Q of at most kFewQ members: a pair per lane, and every lane colours
// from the six bits.  For four vertices per warp that all have so few, which is
// most of a sparse graph, the form above lost to the one-search-per-pair form
// before it: 1,000 x 1,000 grid 0.22 ms then, 0.30 with it alone, 0.17 now; 200,000
// cliques of five 0.21, 0.30, 0.16; 10^6 vertices of degree one 0.13, 0.21, 0.13.
constexpr int kFewQ = 4;
__device__ __forceinline__ void few_features(const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                             float kmax, float ldmax, int64_t deg, int kv, int c, const int *qs,
                                             float f[kF]) {
  const int lane = threadIdx.x & 31, grp = lane >> 3, gl = lane & 7;
  const unsigned gm = 0xFFu << (grp * 8);
  const int q = c;
  // pairs (0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)
  const int i = gl < 3 ? 0 : (gl < 5 ? 1 : 2), j = gl < 3 ? gl + 1 : (gl < 5 ? gl - 1 : 3);
  bool adj = false;
  if (gl < 6 && j < q) {
    int x = qs[i], y = qs[j];
    int64_t lo = rp[x], r0 = rp[y];
    int left = (int)(rp[x + 1] - lo);
    const int other = (int)(rp[y + 1] - r0);
    if (other < left) {  // the shorter of the two rows
      left = other;
      lo = r0;
      y = x;
    }
    while (left) {
      const int h = left >> 1, z = ci[lo + h];
      if (z == y) {
        adj = true;
        left = 0;
      } else if (z < y) {
        lo += h + 1;
        left -= h + 1;
      } else {
        left = h;
      }
    }
  }
  __syncwarp(gm);
  const unsigned p = group_ballot(gm, adj, grp);
  // greedy colouring in index order; rows[v]: the earlier neighbours of member v
  const unsigned rows[4] = {0u, p & 1u, ((p >> 1) & 1u) | ((p >> 2) & 2u), ((p >> 2) & 1u) | ((p >> 3) & 6u)};
  unsigned cls[4] = {0u, 0u, 0u, 0u};
  int chi = 0;
#pragma unroll
  for (int v = 0; v < 4; v++) {
    bool placed = v >= q;
#pragma unroll
    for (int k = 0; k <= v; k++)
      if (!placed && !(cls[k] & rows[v])) {
        cls[k] |= 1u << v;
        chi = max(chi, k + 1);
        placed = true;
      }
  }
  write_features(kmax, ldmax, deg, kv, c, __popc(p), chi, f);
}

struct FA {
  int64_t n;
  const int32_t *list;   // the vertices, nullptr: all of [0, n)
  const int64_t *count;  // with a list: its length
  const int64_t *rp;
  const int32_t *ci, *core;
  float kmax, ldmax;
  int32_t *hubs;  // vertices of more than kWarpRow neighbours, left to hub_kernel
  unsigned *nhubs;
  float *out;  // features (6 per vertex) or scores (one)
  const uint16_t *wbf;
  const float *master;
};

__device__ __forceinline__ void put_features(float *f, const float x[kF], int gl) {
  float y = x[0];
#pragma unroll
  for (int i = 1; i < kF; i++) y = gl == i ? x[i] : y;
  if (gl < kF) f[gl] = y;
}

// The network in shared memory, laid out for a group of eight lanes per
// row: lane gl owns hidden units gl, gl + 8, ..., gl + 56; the first two
// layers are stored input-major so a group's reads of one input's weights
// are consecutive words.
struct MlpSmem {
  float w1t[kF][kH];  // w1t[i][j] = W1[j][i]
  float b1[kH];
  float w2t[kH][kH];  // w2t[k][j] = W2[j][k]
  float b2[kH];
  float w3[kH];
  float b3;
};

__device__ void load_mlp(const uint16_t *__restrict__ wbf, const float *__restrict__ master, MlpSmem &S) {
  for (int e = threadIdx.x; e < kH * kF; e += blockDim.x) {
    const int j = e / kF, i = e % kF;
    S.w1t[i][j] = bf16_to_f32(wbf[kOffW1 + e]);
  }
  for (int e = threadIdx.x; e < kH * kH; e += blockDim.x) {
    const int j = e / kH, k = e % kH;
    S.w2t[k][j] = bf16_to_f32(wbf[kOffW2 + e]);
  }
  for (int j = threadIdx.x; j < kH; j += blockDim.x) {
    S.b1[j] = master[kOffB1 + j];  // biases stay fp32
    S.b2[j] = master[kOffB2 + j];
    S.w3[j] = bf16_to_f32(wbf[kOffW3 + j]);
  }
  if (threadIdx.x == 0) S.b3 = master[kOffB3];
  __syncthreads();
}

// The logit of one row x (every lane of the group holds x), by the 8 lanes
// of a group.
__device__ __forceinline__ float mlp_logit_group(const MlpSmem &S, const float x[kF]) {
  const int lane = threadIdx.x & 31, grp = lane >> 3, gl = lane & 7;
  const unsigned gm = 0xFFu << (grp * 8);
  float h[8];
#pragma unroll
  for (int t = 0; t < 8; t++) {
    const int j = gl + 8 * t;
    float z = S.b1[j];
#pragma unroll
    for (int i = 0; i < kF; i++) z = fmaf(S.w1t[i][j], x[i], z);
    h[t] = fmaxf(z, 0.f);
  }
  float z[8];
#pragma unroll
  for (int t = 0; t < 8; t++) z[t] = S.b2[gl + 8 * t];
#pragma unroll
  for (int tk = 0; tk < 8; tk++) {
#pragma unroll
    for (int src = 0; src < 8; src++) {
      const float hk = __shfl_sync(gm, h[tk], src, 8);
      const int k = src + 8 * tk;
#pragma unroll
      for (int t = 0; t < 8; t++) z[t] = fmaf(S.w2t[k][gl + 8 * t], hk, z[t]);
    }
  }
  float sum = 0.f;
#pragma unroll
  for (int t = 0; t < 8; t++) sum = fmaf(S.w3[gl + 8 * t], fmaxf(z[t], 0.f), sum);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(gm, sum, o, 8);
  return sum + S.b3;
}

// Features of the listed vertices, or their scores (features and logit fused:
// the feature rows never reach memory).  Eight lanes per vertex, four vertices
// per warp; rows of more than kGroupRow entries are counted by the whole warp,
// one after the other.
template <bool SCORE>
__global__ void __launch_bounds__(256) features_kernel(FA a) {
  __shared__ MlpSmem S[1];
  __shared__ int qs[8][4][kQ];
  if (SCORE) load_mlp(a.wbf, a.master, S[0]);
  const int lane = threadIdx.x & 31, grp = lane >> 3, gl = lane & 7;
  const unsigned gm = 0xFFu << (grp * 8);
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t total = a.list ? *a.count : a.n;
  auto &Q = qs[threadIdx.x >> 5];
  for (int64_t b = w0 * 4; b < total; b += nw * 4) {
    const int64_t r = b + grp;
    int64_t v = 0, e0 = 0, e1 = 0;
    int kv = 0, c = 0;
    if (r < total) {
      v = a.list ? a.list[r] : r;
      e0 = a.rp[v];
      e1 = a.rp[v + 1];
      kv = a.core[v];
    }
    const int64_t len = e1 - e0;
    const bool hub = a.hubs && len > kWarpRow;
    if (hub && gl == 0) a.hubs[atomicAdd(a.nhubs, 1u)] = (int32_t)v;
    unsigned wide = __ballot_sync(0xffffffffu, !hub && len > kGroupRow) & 0x01010101u;
    while (wide) {
      const int src = __ffs(wide) - 1;
      wide &= wide - 1;
      const int64_t f0 = __shfl_sync(0xffffffffu, e0, src), f1 = __shfl_sync(0xffffffffu, e1, src);
      const int fk = __shfl_sync(0xffffffffu, kv, src);
      const int fc = count_row<32, kRowFly>(a.ci, a.core, fk, f0, f1, 0xffffffffu, 0, lane, Q[src >> 3]);
      if (grp == (src >> 3)) c = fc;
    }
    if (__all_sync(0xffffffffu, len <= 8)) c = count_row<8, 1>(a.ci, a.core, kv, e0, e1, gm, grp * 8, gl, Q[grp]);
    else if (len <= kGroupRow) c = count_row<8, kRowFly>(a.ci, a.core, kv, e0, e1, gm, grp * 8, gl, Q[grp]);
    const bool few = __all_sync(0xffffffffu, hub || c <= kFewQ);
    if (r < total && !hub) {
      float x[kF];
      if (few) few_features(a.rp, a.ci, a.kmax, a.ldmax, len, kv, c, Q[grp], x);
      else vertex_features(a.rp, a.ci, a.kmax, a.ldmax, len, kv, c, Q[grp], x);
      if (SCORE) {
        const float s = mlp_logit_group(S[0], x);
        if (gl == 0) a.out[v] = s;
      } else {
        put_features(a.out + v * kF, x, gl);
      }
    }
    __syncwarp();  // Q is free for the next vertices
  }
}

// The same for the vertices of the longest rows, a block each: every warp
// counts a slice of the row, the first group of lanes does the rest.
constexpr int kUT = 512;
template <bool SCORE>
__global__ void __launch_bounds__(kUT) hub_kernel(FA a) {
  __shared__ MlpSmem S[1];
  __shared__ int qs[kUT / 32][kQ], cs[kUT / 32], Q[kQ];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned nhubs = *a.nhubs;
  if (SCORE && blockIdx.x < nhubs) load_mlp(a.wbf, a.master, S[0]);
  for (unsigned h = blockIdx.x; h < nhubs; h += gridDim.x) {
    const int64_t v = a.hubs[h], e0 = a.rp[v], e1 = a.rp[v + 1], len = e1 - e0;
    const int kv = a.core[v];
    const int64_t s0 = e0 + len * wid / (kUT / 32), s1 = e0 + len * (wid + 1) / (kUT / 32);
    const int c = count_row<32, kRowFly>(a.ci, a.core, kv, s0, s1, 0xffffffffu, 0, lane, qs[wid]);
    if (lane == 0) cs[wid] = c;
    __syncthreads();
    if (threadIdx.x < 8) {
      int all = 0, q = 0;
      for (int w = 0; w < kUT / 32; w++) {
        all += cs[w];
        for (int i = 0; i < min(cs[w], kQ) && q < kQ; i++, q++)
          if (threadIdx.x == 0) Q[q] = qs[w][i];
      }
      __syncwarp(0xFFu);
      float x[kF];
      vertex_features(a.rp, a.ci, a.kmax, a.ldmax, len, kv, all, Q, x);
      if (SCORE) {
        const float s = mlp_logit_group(S[0], x);
        if (threadIdx.x == 0) a.out[v] = s;
      } else {
        put_features(a.out + v * kF, x, threadIdx.x);
      }
    }
    __syncthreads();
  }
}

// hubs and *nhubs for the vertices of g (rows of more than kWarpRow entries
// are at most nnz / kWarpRow), then both kernels.
template <bool SCORE>
int launch_features(mc_graph *g, FA a, int blocks) {
  a.rp = g->row_ptr;
  a.ci = g->col_idx;
  a.core = g->core;
  a.kmax = (float)std::max(g->max_core, 1);
  a.ldmax = log1pf((float)std::max(g->max_degree, 1));
  const bool hubs = g->max_degree > kWarpRow;
  if (hubs) {
    void *p;
    MC_TRY(ws_get(g, "ln.hubs", 64 + (size_t)(g->nnz / kWarpRow + 1) * 4, &p));
    a.nhubs = (unsigned *)p;
    a.hubs = (int32_t *)((char *)p + 64);
    MC_CUDA_TRY(cudaMemsetAsync(p, 0, 4, g->stream));
  }
  features_kernel<SCORE><<<blocks, 256, 0, g->stream>>>(a);
  g_launches++;
  if (hubs) {
    hub_kernel<SCORE><<<2 * g->sm_count, kUT, 0, g->stream>>>(a);
    g_launches++;
  }
  MC_CUDA_TRY(cudaGetLastError());
  return MC_OK;
}

constexpr int kGS = 68;  // row stride of the 64-wide tiles (float4 aligned, off the banks)
__device__ __forceinline__ void fma4x4(float (&c)[4][4], const float4 &a, const float4 &b) {
  const float x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) c[i][j] = fmaf(x[i], y[j], c[i][j]);
}
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// Logits of few feature rows, eight lanes per row, so that they still spread over
// the SMs: a call takes 30.5 us for 4,096 rows (33.2 by tiles), 35.1 for 8,192
// (32.9).
constexpr int64_t kFewRows = 4096;
__global__ void __launch_bounds__(256) forward_few_kernel(int64_t n, const float *__restrict__ feat,
                                                          const uint16_t *__restrict__ wbf,
                                                          const float *__restrict__ master, float *__restrict__ out) {
  __shared__ MlpSmem S;
  load_mlp(wbf, master, S);
  const int lane = threadIdx.x & 31, grp = lane >> 3, gl = lane & 7;
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = w0 * 4; b < n; b += nw * 4) {
    const int64_t r = b + grp;
    if (r >= n) continue;
    float x[kF];
#pragma unroll
    for (int i = 0; i < kF; i++) x[i] = feat[r * kF + i];
    const float s = mlp_logit_group(S, x);
    if (gl == 0) out[r] = s;
  }
}

// Logits of n feature rows: a block takes 128 rows, the second layer as a
// 128 x 64 x 64 product in register tiles of 8 rows x 4 units over operands
// in shared memory (three float4 for 32 FMAs, so the FP32 pipe is the bound,
// not the shared-memory pipe as with eight lanes per row, a weight read per
// FMA).  262,144 rows: 184 us before, 64 us now.
constexpr int kVR = 128, kVT = 256, kVS = kVR + 4;
struct FwdSmem {
  float w2t[kH][kGS], h1t[kH][kVS];
  float w1t[kF][kH], x[kF][kVR];
  float b1[kH], b2[kH], w3[kH], b3;
};
static_assert(offsetof(FwdSmem, h1t) % 16 == 0 && offsetof(FwdSmem, w1t) % 16 == 0 && offsetof(FwdSmem, x) % 16 == 0 &&
                  offsetof(FwdSmem, w2t) % 16 == 0 && kVS % 4 == 0 && kVT == (kVR / 8) * (kH / 4),
              "float4 operands of forward_kernel");
// Column of second-layer unit j: thread pair p of a row (columns 8 p .. 8 p + 7)
// holds the units p, p + 8, ..., p + 56, whose terms of the logit are then added
// in the order of mlp_logit_group (pair sums by distance 4, 2, 1): both give the
// same bits.
__device__ __forceinline__ int column_of(int j) { return 8 * (j & 7) + (j >> 3); }
__global__ void __launch_bounds__(kVT) forward_kernel(int64_t n, const float *__restrict__ feat,
                                                      const uint16_t *__restrict__ wbf,
                                                      const float *__restrict__ master, float *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char fsm_raw[];
  FwdSmem &S = *reinterpret_cast<FwdSmem *>(fsm_raw);
  const int t = threadIdx.x, c0 = 4 * (t & 15), r0 = 8 * (t >> 4);
  for (int e = t; e < kH * kH; e += kVT) S.w2t[e % kH][column_of(e / kH)] = bf16_to_f32(wbf[kOffW2 + e]);
  for (int e = t; e < kH * kF; e += kVT) S.w1t[e % kF][e / kF] = bf16_to_f32(wbf[kOffW1 + e]);
  for (int j = t; j < kH; j += kVT) {
    S.b1[j] = master[kOffB1 + j];  // biases stay fp32
    S.b2[column_of(j)] = master[kOffB2 + j];
    S.w3[column_of(j)] = bf16_to_f32(wbf[kOffW3 + j]);
  }
  if (t == 0) S.b3 = master[kOffB3];
  for (int64_t base = (int64_t)blockIdx.x * kVR; base < n; base += (int64_t)gridDim.x * kVR) {
    const int rows = (int)min((int64_t)kVR, n - base);
    __syncthreads();  // the weights are there; the last tile is done with the buffers
    for (int e = t; e < kVR * kF; e += kVT) S.x[e % kF][e / kF] = e / kF < rows ? feat[base * kF + e] : 0.f;
    __syncthreads();
    float c[2][4][4];
#pragma unroll
    for (int h = 0; h < 2; h++) {
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) c[h][i][j] = S.b1[c0 + j];
#pragma unroll
      for (int i = 0; i < kF; i++) fma4x4(c[h], ld4(&S.x[i][r0 + 4 * h]), ld4(&S.w1t[i][c0]));
#pragma unroll
      for (int j = 0; j < 4; j++)
        *reinterpret_cast<float4 *>(&S.h1t[c0 + j][r0 + 4 * h]) =
            make_float4(fmaxf(c[h][0][j], 0.f), fmaxf(c[h][1][j], 0.f), fmaxf(c[h][2][j], 0.f),
                        fmaxf(c[h][3][j], 0.f));
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; h++)
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) c[h][i][j] = S.b2[c0 + j];
#pragma unroll 4
    for (int k = 0; k < kH; k++) {
      const float4 w = ld4(&S.w2t[k][c0]);
      fma4x4(c[0], ld4(&S.h1t[k][r0]), w);
      fma4x4(c[1], ld4(&S.h1t[k][r0 + 4]), w);
    }
    // the 16 threads of a row share its logit: an odd thread goes on from the
    // even one's partial sum, the eight pairs' sums are added as a tree
#pragma unroll
    for (int h = 0; h < 2; h++)
#pragma unroll
      for (int i = 0; i < 4; i++) {
        float v = 0.f;
#pragma unroll
        for (int j = 0; j < 4; j++) v = fmaf(S.w3[c0 + j], fmaxf(c[h][i][j], 0.f), v);
        float w = __shfl_xor_sync(0xffffffffu, v, 1);
#pragma unroll
        for (int j = 0; j < 4; j++) w = fmaf(S.w3[c0 + j], fmaxf(c[h][i][j], 0.f), w);
        v = w;  // the pair's sum in odd threads
#pragma unroll
        for (int o = 8; o >= 2; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        const int r = r0 + 4 * h + i;
        if ((t & 15) == 1 && r < rows) out[base + r] = v + S.b3;
      }
  }
}

// Gradient of the mean weighted BCE over rows, accumulated into grad (fp32).
// A block takes tiles of kGR rows.  Its three 64 x 64 x 64 products (the second
// layer forward, back to the first layer, and the second layer's weights) and
// the first layer are register tiles of 4 x 4 outputs per thread over operands
// in shared memory, each operand in the layout that the product reads as
// float4; sums over rows stay in registers over all tiles of a block and reach
// memory once per block.  FP32 throughout: the activations are not BF16, so the
// tensor pipe's types would round them.  Every sum has a fixed order.
// 16,384 rows: 190 us with a thread per row (128 rows per block, serial
// 64-long chains per thread, 6% of the warps, sums by atomics), 26 us now with
// 9 us for the sum over the blocks; its error against 64 bits is a quarter of
// what it was (pairwise in a block, in double over the blocks).  Two blocks
// fit an SM (106 KB each), so 16,384 rows are one tile for each of 256 blocks: a
// call takes 67 us, 75 with one block of 124 KB per SM and two tiles in turn.
constexpr int kGR = 64;    // rows per tile
constexpr int kGT = 256;   // threads: 16 x 16, 4 x 4 outputs each
constexpr int kPart = (kParams + 1 + 31) / 32 * 32;  // floats of a block's sums: parameters, loss
struct GradSmem {
  float w2[kH][kGS], w2t[kH][kGS];  // W2[j][k] and its transpose
  float h1[kGR][kGS], h1t[kH][kGS];
  float d2[kGR][kGS], d2t[kH][kGS];
  float w1t[kF][kH], x[kF][kGR];
  float b1[kH], b2[kH], w3[kH], y[kGR], b3;
};
// what is read as float4 starts on 16 bytes, in every row (columns and rows are
// taken at multiples of four)
static_assert(offsetof(GradSmem, w2) % 16 == 0 && offsetof(GradSmem, w2t) % 16 == 0 &&
                  offsetof(GradSmem, h1) % 16 == 0 && offsetof(GradSmem, h1t) % 16 == 0 &&
                  offsetof(GradSmem, d2) % 16 == 0 && offsetof(GradSmem, d2t) % 16 == 0 &&
                  offsetof(GradSmem, w1t) % 16 == 0 && offsetof(GradSmem, x) % 16 == 0 && kGS % 4 == 0 &&
                  kH % 4 == 0 && kGR % 4 == 0,
              "float4 operands of grad_kernel");
static_assert(kGT == (kH / 4) * (kGR / 4) && kGR == kH, "one 4 x 4 tile per thread in each product");

// a tile and its transpose, rows kGS floats apart
__device__ __forceinline__ void st4x4(float *p, float *pt, const float (&c)[4][4]) {
#pragma unroll
  for (int i = 0; i < 4; i++) {
    *reinterpret_cast<float4 *>(p + i * kGS) = make_float4(c[i][0], c[i][1], c[i][2], c[i][3]);
    *reinterpret_cast<float4 *>(pt + i * kGS) = make_float4(c[0][i], c[1][i], c[2][i], c[3][i]);
  }
}

__global__ void __launch_bounds__(kGT, 2) grad_kernel(int64_t n, const float *__restrict__ feat,
                                                      const float *__restrict__ label, float pos_weight,
                                                      const uint16_t *__restrict__ wbf,
                                                      const float *__restrict__ master, float *__restrict__ part) {
  extern __shared__ __align__(16) unsigned char gsm_raw[];
  GradSmem &S = *reinterpret_cast<GradSmem *>(gsm_raw);
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;  // outputs 4 tx .. (columns), 4 ty .. (rows)
  const int c0 = 4 * tx, r0 = 4 * ty;
  bool bad = false;
  for (int e = t; e < kH * kH; e += kGT) {
    const float w = bf16_to_f32(wbf[kOffW2 + e]);
    S.w2[e / kH][e % kH] = w;
    S.w2t[e % kH][e / kH] = w;
    bad |= !isfinite(w);
  }
  for (int e = t; e < kH * kF; e += kGT) S.w1t[e % kF][e / kF] = bf16_to_f32(wbf[kOffW1 + e]);
  for (int j = t; j < kH; j += kGT) {
    S.b1[j] = master[kOffB1 + j];  // biases stay fp32
    S.b2[j] = master[kOffB2 + j];
    S.w3[j] = bf16_to_f32(wbf[kOffW3 + j]);
  }
  if (t == 0) S.b3 = master[kOffB3];
  // a unit that is off passes nothing back, also where a weight is infinite
  const bool odd = __syncthreads_or(bad);
  const float inv_n = 1.f / (float)n;
  float gw2[4][4] = {}, gw1[4][kF] = {}, gb1[4] = {}, gb2[4] = {}, gw3[4] = {}, gb3 = 0.f, lsum = 0.f;
  for (int64_t base = (int64_t)blockIdx.x * kGR; base < n; base += (int64_t)gridDim.x * kGR) {
    const int rows = (int)min((int64_t)kGR, n - base);
    __syncthreads();  // the last tile is done with the buffers
    for (int e = t; e < kGR * kF; e += kGT) {
      const int r = e / kF;
      S.x[e % kF][r] = r < rows ? feat[base * kF + e] : 0.f;
    }
    for (int r = t; r < kGR; r += kGT) S.y[r] = r < rows ? label[base + r] : 0.f;
    __syncthreads();
    // first layer: rows r0.., units c0..
    float c[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) c[i][j] = S.b1[c0 + j];
#pragma unroll
    for (int i = 0; i < kF; i++) fma4x4(c, ld4(&S.x[i][r0]), ld4(&S.w1t[i][c0]));
    bool on[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) {
        on[i][j] = c[i][j] > 0.f;
        c[i][j] = fmaxf(c[i][j], 0.f);
      }
    st4x4(&S.h1[r0][c0], &S.h1t[c0][r0], c);
    __syncthreads();
    // second layer: rows r0.., units c0..
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) c[i][j] = S.b2[c0 + j];
#pragma unroll 4
    for (int k = 0; k < kH; k++) fma4x4(c, ld4(&S.h1t[k][r0]), ld4(&S.w2t[k][c0]));
    // logit of each row: the 16 threads of a row share it
    float gs[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < 4; j++) s = fmaf(S.w3[c0 + j], fmaxf(c[i][j], 0.f), s);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      s += S.b3;
      // d loss / d s for weighted BCE with logits, mean over rows
      gs[i] = 0.f;
      if (r0 + i < rows) {
        const float y = S.y[r0 + i];
        const float w = y > 0.5f ? pos_weight : 1.f;
        const float sig = 1.f / (1.f + expf(-s));
        gs[i] = w * (sig - y) * inv_n;
        // loss = w * (log(1 + e^s) - y s), computed stably
        if (tx == 0) {
          lsum += w * (fmaxf(s, 0.f) + log1pf(expf(-fabsf(s))) - y * s) * inv_n;
          gb3 += gs[i];
        }
      }
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const float d = c[i][j] > 0.f ? gs[i] * S.w3[c0 + j] : 0.f;
        gb2[j] += d;
        gw3[j] += fmaxf(c[i][j], 0.f) * gs[i];
        c[i][j] = d;
      }
    }
    st4x4(&S.d2[r0][c0], &S.d2t[c0][r0], c);
    __syncthreads();
    // back through W2: d loss / d h1, rows r0.., units c0..; and W2's own
    // gradient, its row r0.. (second-layer unit), column c0..
    float d1[4][4] = {};
    if (!odd) {
#pragma unroll 4
      for (int k = 0; k < kH; k++) fma4x4(d1, ld4(&S.d2t[k][r0]), ld4(&S.w2[k][c0]));
    } else {
      for (int k = 0; k < kH; k++)
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const float d = S.d2t[k][r0 + i];
          if (d != 0.f)
#pragma unroll
            for (int j = 0; j < 4; j++) d1[i][j] = fmaf(d, S.w2[k][c0 + j], d1[i][j]);
        }
    }
#pragma unroll 4
    for (int r = 0; r < kGR; r++) fma4x4(gw2, ld4(&S.d2[r][r0]), ld4(&S.h1[r][c0]));
    // first layer: rows of this thread only, summed over the block at the end
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const float d = on[i][j] ? d1[i][j] : 0.f;
        gb1[j] += d;
#pragma unroll
        for (int f = 0; f < kF; f++) gw1[j][f] = fmaf(d, S.x[f][r0 + i], gw1[j][f]);
      }
  }
  // The block's sums, to its place.  W2's gradient is whole in each thread; the
  // others are spread over the 16 threads of a column: the two halves of a warp
  // are added here, the eight warps pairwise, through the tiles' space.
  float *out = part + (int64_t)blockIdx.x * kPart;
#pragma unroll
  for (int i = 0; i < 4; i++)
    *reinterpret_cast<float4 *>(out + kOffW2 + (r0 + i) * kH + c0) =
        make_float4(gw2[i][0], gw2[i][1], gw2[i][2], gw2[i][3]);
  __syncthreads();  // the tiles are free
  constexpr int kWarps = kGT / 32, kUnit = kF + 3;  // warps; sums per unit
  float *red = &S.w2[0][0], *ends = &S.h1[0][0];
  static_assert(kWarps * kUnit * kH <= 2 * kH * kGS && kGT / 16 == 16, "room for the sums");
#pragma unroll
  for (int j = 0; j < 4; j++) {
    float v[kUnit];
#pragma unroll
    for (int f = 0; f < kF; f++) v[f] = gw1[j][f];
    v[kF] = gb1[j];
    v[kF + 1] = gb2[j];
    v[kF + 2] = gw3[j];
#pragma unroll
    for (int f = 0; f < kUnit; f++) {
      v[f] += __shfl_xor_sync(0xffffffffu, v[f], 16);
      if ((t & 16) == 0) red[((t >> 5) * kUnit + f) * kH + c0 + j] = v[f];
    }
  }
  if (tx == 0) {
    ends[ty] = gb3;
    ends[kGT / 16 + ty] = lsum;
  }
  __syncthreads();
  for (int e = t; e < kUnit * kH; e += kGT) {
    float v[kWarps];
#pragma unroll
    for (int w = 0; w < kWarps; w++) v[w] = red[w * kUnit * kH + e];
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1)
#pragma unroll
      for (int w = 0; w < o; w++) v[w] += v[w + o];
    const int f = e / kH, c = e % kH;
    out[f < kF ? kOffW1 + c * kF + f : (f == kF ? kOffB1 : (f == kF + 1 ? kOffB2 : kOffW3)) + c] = v[0];
  }
  if (t < 32) {  // b3 in the first half of the warp, the loss in the second
    float v = ends[t];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((t & 15) == 0) out[t == 0 ? kOffB3 : kParams] = v;
  }
}

// The blocks' sums, added in a fixed order too (the gradient is the same bits on
// every call) and in double, so that each parameter is rounded once here: a
// warp's lanes are 32 parameters, its eight warps an eighth of the blocks each.
constexpr int kRT = 256;
__global__ void __launch_bounds__(kRT) grad_sum_kernel(int blocks, const float *__restrict__ part,
                                                       float *__restrict__ grad, float *__restrict__ loss) {
  __shared__ double sm[kRT / 32][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  double v = 0.0;
  if (e <= kParams) {
#pragma unroll 8
    for (int b = wid; b < blocks; b += kRT / 32) v += (double)part[(int64_t)b * kPart + e];
  }
  sm[wid][lane] = v;
  __syncthreads();
  if (wid == 0 && e <= kParams) {
#pragma unroll
    for (int i = 1; i < kRT / 32; i++) v += sm[i][lane];
    if (e < kParams) grad[e] = (float)v;
    else *loss = (float)v;
  }
}

__global__ void adam_kernel(float *__restrict__ master, uint16_t *__restrict__ wbf, const float *__restrict__ grad,
                            float *__restrict__ m, float *__restrict__ v, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kParams; i += gridDim.x * blockDim.x) {
    const float g = grad[i];
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const float p = master[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    master[i] = p;
    wbf[i] = f32_to_bf16(p);
  }
}

__global__ void round_kernel(const float *__restrict__ master, uint16_t *__restrict__ wbf) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kParams; i += gridDim.x * blockDim.x)
    wbf[i] = f32_to_bf16(master[i]);
}

uint64_t splitmix(uint64_t z) {
  z += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

int stage(mc_mlp *m, const void *src, size_t bytes, const void **dev) {
  if (is_device_ptr(src)) {
    *dev = src;
    return MC_OK;
  }
  if (m->buf_bytes < bytes) {
    if (m->buf) {
      MC_CUDA_TRY(cudaStreamSynchronize(m->stream));
      cudaFree(m->buf);
    }
    m->buf = nullptr;
    m->buf_bytes = 0;
    MC_CUDA_TRY(cudaMalloc(&m->buf, bytes));
    m->buf_bytes = bytes;
  }
  MC_CUDA_TRY(cudaMemcpyAsync(m->buf, src, bytes, cudaMemcpyHostToDevice, m->stream));
  *dev = m->buf;
  return MC_OK;
}

// ------------------------------------------- the learned form of a solve ---

// Vertices that can still be in a clique larger than their graph's current
// bound (K(v) >= best), appended to list (warp-aggregated); *count holds the
// number (zeroed by the caller).
__global__ void subset_kernel(int64_t n, const int32_t *__restrict__ core, const int32_t *__restrict__ gid,
                              const int32_t *__restrict__ best, const int32_t *__restrict__ kfloor,
                              int32_t *__restrict__ list, unsigned long long *__restrict__ count) {
  const int kf = kfloor ? *kfloor : 0;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) & ~(int64_t)31; b < n; b += stride) {
    const int64_t v = b + lane;
    bool in = false;
    if (v < n) in = core[v] >= max(best[gid ? gid[v] : 0], kf);
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (!m) continue;
    unsigned long long at = 0;
    if (lane == 0) at = atomicAdd(count, (unsigned long long)__popc(m));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (in) list[at + __popc(m & lt)] = (int32_t)v;
  }
}

__global__ void fill_kernel(int64_t n, float x, float *__restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = x;
}

// Histogram of the core numbers (bins 0..kmax).
__global__ void core_hist_kernel(int64_t n, const int32_t *__restrict__ core, int kmax, unsigned int *__restrict__ hist) {
  extern __shared__ unsigned int sh[];
  const bool local = kmax < 8192;
  if (local) {
    for (int i = threadIdx.x; i <= kmax; i += blockDim.x) sh[i] = 0;
    __syncthreads();
  }
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int k = min(core[v], kmax);
    atomicAdd(local ? &sh[k] : &hist[k], 1u);
  }
  if (local) {
    __syncthreads();
    for (int i = threadIdx.x; i <= kmax; i += blockDim.x)
      if (sh[i]) atomicAdd(&hist[i], sh[i]);
  }
}

// The core floor of the scored subset: the smallest k such that at most
// `budget` vertices have K(v) >= k (at least the top shell, K(G)).
__global__ void core_floor_kernel(const unsigned int *__restrict__ hist, int kmax, long long budget,
                                  int32_t *__restrict__ kfloor) {
  if (threadIdx.x != 0) return;
  long long above = 0;
  int k = kmax;
  above = hist[kmax];
  while (k > 0 && above + (long long)hist[k - 1] <= budget) {
    k--;
    above += hist[k];
  }
  *kfloor = k;
}

// Selection key of a scored vertex: the score's order as an unsigned
// integer (larger score, larger key; raised to at least 1) in the high
// word, and the complement of the vertex id in the low word, so keys are
// unique and ties go to the smaller id.
__device__ __forceinline__ unsigned long long seed_key(float s, int v) {
  const uint32_t b = __float_as_uint(s);
  const uint32_t k = max((b & 0x80000000u) ? ~b : (b | 0x80000000u), 1u);
  return ((unsigned long long)k << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)v);
}

struct SelectCtl {
  unsigned long long prefix, mask;  // key bits fixed so far
  long long need;                   // keys still to take at or below the prefix
  long long taken;                  // keys collected
  int all;                          // fewer keys than k: take every key
  int pad;
  unsigned int hist[256];
};

__global__ void select_init_kernel(SelectCtl *ctl, int k) {
  if (threadIdx.x == 0) ctl->need = k;
}

// one 8-bit digit of the k-th largest key: histogram of the keys that match
// the prefix so far
__global__ void select_hist_kernel(const int32_t *__restrict__ list, const unsigned long long *__restrict__ count,
                                   const float *__restrict__ score, SelectCtl *ctl, int shift) {
  __shared__ unsigned int h[256];
  for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0;
  __syncthreads();
  const unsigned long long prefix = ctl->prefix, mask = ctl->mask;
  const int64_t total = (int64_t)*count;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < total; r += (int64_t)gridDim.x * blockDim.x) {
    const int v = list[r];
    const unsigned long long key = seed_key(score[v], v);
    if ((key & mask) == prefix) atomicAdd(&h[(key >> shift) & 255ull], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 256; i += blockDim.x)
    if (h[i]) atomicAdd(&ctl->hist[i], h[i]);
}

__global__ void select_pick_kernel(SelectCtl *ctl, int shift) {
  if (threadIdx.x != 0 || ctl->all) return;
  long long acc = 0;
  int b = 255;
  for (; b >= 0; b--) {
    if (acc + (long long)ctl->hist[b] >= ctl->need) break;
    acc += ctl->hist[b];
  }
  if (b < 0) {  // fewer matching keys than needed: only on the first digit
    ctl->all = 1;
  } else {
    ctl->need -= acc;
    ctl->prefix |= (unsigned long long)b << shift;
    ctl->mask |= 255ull << shift;
  }
  for (int i = 0; i < 256; i++) ctl->hist[i] = 0;
}

__global__ void select_collect_kernel(const int32_t *__restrict__ list, const unsigned long long *__restrict__ count,
                                      const float *__restrict__ score, SelectCtl *ctl, int k,
                                      unsigned long long *__restrict__ keys) {
  const unsigned long long thr = ctl->all ? 0ull : ctl->prefix;
  const int64_t total = (int64_t)*count;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < total; r += (int64_t)gridDim.x * blockDim.x) {
    const int v = list[r];
    const unsigned long long key = seed_key(score[v], v);
    if (key >= thr) {
      const long long at = atomicAdd((unsigned long long *)&ctl->taken, 1ull);
      if (at < k) keys[at] = key;
    }
  }
}

// the collected keys in decreasing order -> seed vertices; -1 pads the
// slots past the number collected
constexpr int kMaxSeeds = 1024;
__global__ void __launch_bounds__(1024) select_sort_kernel(const SelectCtl *ctl, int k,
                                                           const unsigned long long *__restrict__ keys,
                                                           int32_t *__restrict__ seeds) {
  __shared__ unsigned long long a[kMaxSeeds];
  const int got = (int)(ctl->taken < (long long)k ? ctl->taken : (long long)k);
  for (int i = threadIdx.x; i < kMaxSeeds; i += blockDim.x) a[i] = i < got ? keys[i] : 0ull;
  __syncthreads();
  for (int len = 2; len <= kMaxSeeds; len <<= 1) {
    for (int j = len >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < kMaxSeeds; i += blockDim.x) {
        const int x = i ^ j;
        if (x > i) {
          const unsigned long long p = a[i], q = a[x];
          const bool desc = (i & len) == 0;
          if (desc ? (p < q) : (p > q)) {
            a[i] = q;
            a[x] = p;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < k; i += blockDim.x)
    seeds[i] = i < got ? (int32_t)(0xFFFFFFFFu - (uint32_t)(a[i] & 0xFFFFFFFFull)) : -1;
}

// Batches: the j best-scored vertices of every graph among those that can
// beat its bound, one warp per graph (j rounds of a warp maximum, each
// below the last key taken).  seeds[g * j + r], -1 where a graph has fewer.
__global__ void graph_seeds_kernel(int32_t count, const int64_t *__restrict__ voff, const int32_t *__restrict__ core,
                                   const int32_t *__restrict__ best, const float *__restrict__ score, int j,
                                   int32_t *__restrict__ seeds) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t g = w0; g < count; g += nw) {
    const int64_t v0 = voff[g], v1 = voff[g + 1];
    const int bg = best[g];
    unsigned long long last = ~0ull;
    for (int r = 0; r < j; r++) {
      unsigned long long mx = 0ull;
      for (int64_t v = v0 + lane; v < v1; v += 32) {
        if (core[v] < bg) continue;
        const unsigned long long key = seed_key(score[v], (int)v);
        if (key < last && key > mx) mx = key;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, mx, o);
        if (y > mx) mx = y;
      }
      if (lane == 0) seeds[g * j + r] = mx ? (int32_t)(0xFFFFFFFFu - (uint32_t)(mx & 0xFFFFFFFFull)) : -1;
      last = mx;
      if (!mx) last = 0ull;
    }
  }
}

}  // namespace

// Scores of the vertices that can still be in a clique larger than their
// graph's current bound -- for one graph, of at most kLearnedBudget of them,
// those of highest core number.  The other vertices get the lowest score
// (they are read only as candidates of a seeded growth, which then takes
// them last).
constexpr long long kLearnedBudget = 1ll << 22;
int learned_scores(mc_graph *g, const mc_mlp *m, float *score) {
  if (g->n == 0) return MC_OK;
  void *p;
  MC_TRY(ws_get(g, "ln.list", (size_t)g->n * 4, &p));
  int32_t *list = (int32_t *)p;
  MC_TRY(ws_get(g, "ln.ctl", 64 + sizeof(SelectCtl), &p));
  unsigned long long *count = (unsigned long long *)p;
  int32_t *kfloor = (int32_t *)((char *)p + 8);
  MC_CUDA_TRY(cudaMemsetAsync(count, 0, 16, g->stream));
  const int blocks = (int)std::min<int64_t>((g->n + 255) / 256, (int64_t)g->sm_count * 8);
  if (g->count == 1 && g->n > kLearnedBudget) {
    // one graph: score at most kLearnedBudget vertices, those of highest
    // core number (a vertex of core number K is in no clique above K + 1)
    const int kmax = std::max(g->max_core, 0);
    MC_TRY(ws_get(g, "ln.hist", (size_t)(kmax + 2) * 4, &p));
    unsigned int *hist = (unsigned int *)p;
    MC_CUDA_TRY(cudaMemsetAsync(hist, 0, (size_t)(kmax + 2) * 4, g->stream));
    const size_t shm = kmax < 8192 ? (size_t)(kmax + 1) * 4 : 0;
    core_hist_kernel<<<blocks, 256, shm, g->stream>>>(g->n, g->core, kmax, hist);
    core_floor_kernel<<<1, 32, 0, g->stream>>>(hist, kmax, kLearnedBudget, kfloor);
    g_launches += 2;
  }
  subset_kernel<<<blocks, 256, 0, g->stream>>>(g->n, g->core, g->gid, g->best, kfloor, list, count);
  fill_kernel<<<blocks, 256, 0, g->stream>>>(g->n, -INFINITY, score);
  g_launches += 2;
  FA a{};
  a.n = g->n;
  a.list = list;
  a.count = (const int64_t *)count;
  a.out = score;
  a.wbf = m->wbf;
  a.master = m->master;
  return launch_features<true>(g, a, g->sm_count * 8);
}

// Seeds of the learned heuristic: for one graph the k best-scored vertices
// of the subset that learned_scores scored (exact selection by 8-bit digits
// of a unique 64-bit key, best first); for a batch the k best of every
// graph.  Writes seeds (k or count * k slots, -1 for missing ones).
int learned_seeds(mc_graph *g, const float *score, int32_t k, int32_t *seeds) {
  if (g->n == 0 || k <= 0) return MC_OK;
  void *p;
  if (g->count > 1) {
    const int blocks = (int)std::min<int64_t>(((int64_t)g->count * 32 + 255) / 256, (int64_t)g->sm_count * 16);
    graph_seeds_kernel<<<blocks, 256, 0, g->stream>>>(g->count, g->voff, g->core, g->best, score, k, seeds);
    g_launches++;
    MC_CUDA_TRY(cudaGetLastError());
    return MC_OK;
  }
  if (k > kMaxSeeds) return MC_ERR_ARG;
  MC_TRY(ws_get(g, "ln.list", (size_t)g->n * 4, &p));
  const int32_t *list = (const int32_t *)p;
  MC_TRY(ws_get(g, "ln.ctl", 64 + sizeof(SelectCtl), &p));
  const unsigned long long *count = (const unsigned long long *)p;
  SelectCtl *ctl = (SelectCtl *)((char *)p + 64);
  MC_TRY(ws_get(g, "ln.keys", (size_t)kMaxSeeds * 8, &p));
  unsigned long long *keys = (unsigned long long *)p;
  MC_CUDA_TRY(cudaMemsetAsync(ctl, 0, sizeof(SelectCtl), g->stream));
  select_init_kernel<<<1, 32, 0, g->stream>>>(ctl, k);
  g_launches++;
  const int blocks = g->sm_count * 4;
  for (int shift = 56; shift >= 0; shift -= 8) {
    select_hist_kernel<<<blocks, 256, 0, g->stream>>>(list, count, score, ctl, shift);
    select_pick_kernel<<<1, 32, 0, g->stream>>>(ctl, shift);
    g_launches += 2;
  }
  select_collect_kernel<<<blocks, 256, 0, g->stream>>>(list, count, score, ctl, k, keys);
  select_sort_kernel<<<1, 1024, 0, g->stream>>>(ctl, k, keys, seeds);
  g_launches += 2;
  MC_CUDA_TRY(cudaGetLastError());
  return MC_OK;
}

}  // namespace mc

using namespace mc;

extern "C" {

int mc_mlp_create(uint64_t seed, void *cuda_stream, mc_mlp **out) {
  if (!out) return MC_ERR_ARG;
  *out = nullptr;
  mc_mlp *m = new mc_mlp();
  m->stream = (cudaStream_t)cuda_stream;
  auto fail = [&](int rc) {
    cudaFree(m->master); cudaFree(m->wbf); cudaFree(m->m); cudaFree(m->v);
    if (m->h_small) cudaFreeHost(m->h_small);
    delete m;
    return rc;
  };
  if (cudaGetDevice(&m->device) != cudaSuccess) return fail(MC_ERR_CUDA);
  cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, m->device);
  if (cudaMalloc(&m->master, kParams * 4) != cudaSuccess || cudaMalloc(&m->wbf, kParams * 2) != cudaSuccess ||
      cudaMalloc(&m->m, kParams * 4) != cudaSuccess || cudaMalloc(&m->v, kParams * 4) != cudaSuccess ||
      cudaMallocHost(&m->h_small, 4096) != cudaSuccess)
    return fail(MC_ERR_OOM);
  // He-uniform initial weights from a counter-based generator, zero biases
  std::vector<float> p(kParams, 0.f);
  uint64_t ctr = seed * 0x9E3779B97F4A7C15ULL + 1;
  auto uni = [&]() { return (double)(splitmix(ctr++) >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0; };
  for (int i = 0; i < kH * kF; i++) p[kOffW1 + i] = (float)(uni() * std::sqrt(6.0 / kF));
  for (int i = 0; i < kH * kH; i++) p[kOffW2 + i] = (float)(uni() * std::sqrt(6.0 / kH));
  for (int i = 0; i < kH; i++) p[kOffW3 + i] = (float)(uni() * std::sqrt(6.0 / kH));
  if (cudaMemcpyAsync(m->master, p.data(), kParams * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess)
    return fail(MC_ERR_CUDA);
  cudaMemsetAsync(m->m, 0, kParams * 4, m->stream);
  cudaMemsetAsync(m->v, 0, kParams * 4, m->stream);
  round_kernel<<<(kParams + 255) / 256, 256, 0, m->stream>>>(m->master, m->wbf);
  g_launches++;
  if (cudaStreamSynchronize(m->stream) != cudaSuccess) return fail(MC_ERR_CUDA);
  *out = m;
  return MC_OK;
}

void mc_mlp_free(mc_mlp *m) {
  if (!m) return;
  cudaStreamSynchronize(m->stream);
  cudaFree(m->master); cudaFree(m->wbf); cudaFree(m->part); cudaFree(m->m); cudaFree(m->v);
  cudaFree(m->buf);
  if (m->h_small) cudaFreeHost(m->h_small);
  delete m;
}

int mc_mlp_num_params(void) { return kParams; }

int mc_mlp_get_params(mc_mlp *m, float *out) {
  if (!m || !out) return MC_ERR_ARG;
  MC_CUDA_TRY(cudaMemcpyAsync(out, m->master, kParams * 4, cudaMemcpyDefault, m->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(m->stream));
  return MC_OK;
}

int mc_mlp_set_params(mc_mlp *m, const float *in) {
  if (!m || !in) return MC_ERR_ARG;
  MC_CUDA_TRY(cudaMemcpyAsync(m->master, in, kParams * 4, cudaMemcpyDefault, m->stream));
  MC_CUDA_TRY(cudaMemsetAsync(m->m, 0, kParams * 4, m->stream));
  MC_CUDA_TRY(cudaMemsetAsync(m->v, 0, kParams * 4, m->stream));
  round_kernel<<<(kParams + 255) / 256, 256, 0, m->stream>>>(m->master, m->wbf);
  g_launches++;
  m->step = 0;
  MC_CUDA_TRY(cudaStreamSynchronize(m->stream));
  return MC_OK;
}

int mc_features(mc_graph *g, float *feat_out) {
  if (!g || (g->n > 0 && !feat_out)) return MC_ERR_ARG;
  if (g->n == 0) return MC_OK;
  if (!g->cores_valid) MC_TRY(launch_core_numbers(g, kDefaultSpinLimit));
  float *dst = feat_out;
  void *p = nullptr;
  const bool dev_out = is_device_ptr(feat_out);
  if (!dev_out) {
    MC_TRY(ws_get(g, "ln.feat", (size_t)g->n * kF * 4, &p));
    dst = (float *)p;
  }
  FA a{};
  a.n = g->n;
  a.out = dst;
  MC_TRY(launch_features<false>(g, a, (int)std::min<int64_t>((g->n + 31) / 32, (int64_t)g->sm_count * 8)));
  if (!dev_out) MC_CUDA_TRY(cudaMemcpyAsync(feat_out, dst, (size_t)g->n * kF * 4, cudaMemcpyDeviceToHost, g->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(g->stream));
  return MC_OK;
}

int mc_mlp_forward(mc_mlp *m, const float *feat, int64_t n, float *score_out) {
  if (!m || n < 0 || (n > 0 && (!feat || !score_out))) return MC_ERR_ARG;
  if (n == 0) return MC_OK;
  const void *df;
  MC_TRY(stage(m, feat, (size_t)n * kF * 4, &df));
  float *out = score_out;
  const bool dev_out = is_device_ptr(score_out);
  float *tmp = nullptr;
  if (!dev_out) {
    MC_CUDA_TRY(cudaMallocAsync((void **)&tmp, (size_t)n * 4, m->stream));
    out = tmp;
  }
  if (n <= kFewRows) {
    forward_few_kernel<<<(int)((n * 8 + 255) / 256), 256, 0, m->stream>>>(n, (const float *)df, m->wbf, m->master, out);
  } else {
    // up to three blocks of shared memory per SM
    const int blocks = (int)std::min<int64_t>((n + kVR - 1) / kVR, (int64_t)m->sm_count * 3);
    MC_CUDA_TRY(cudaFuncSetAttribute(forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FwdSmem)));
    forward_kernel<<<blocks, kVT, sizeof(FwdSmem), m->stream>>>(n, (const float *)df, m->wbf, m->master, out);
  }
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  if (!dev_out) {
    MC_CUDA_TRY(cudaMemcpyAsync(score_out, tmp, (size_t)n * 4, cudaMemcpyDeviceToHost, m->stream));
    MC_CUDA_TRY(cudaFreeAsync(tmp, m->stream));
  }
  MC_CUDA_TRY(cudaStreamSynchronize(m->stream));
  return MC_OK;
}

static int run_grad(mc_mlp *m, const float *feat, const float *label, int64_t n, float pos_weight) {
  const void *df, *dl;
  // features and labels are staged separately (labels after the features)
  if (is_device_ptr(feat) && is_device_ptr(label)) {
    df = feat;
    dl = label;
  } else {
    const size_t fb = (size_t)n * kF * 4, lb = (size_t)n * 4;
    if (m->buf_bytes < fb + lb) {
      if (m->buf) {
        MC_CUDA_TRY(cudaStreamSynchronize(m->stream));
        cudaFree(m->buf);
      }
      m->buf = nullptr;
      m->buf_bytes = 0;
      MC_CUDA_TRY(cudaMalloc(&m->buf, fb + lb));
      m->buf_bytes = fb + lb;
    }
    MC_CUDA_TRY(cudaMemcpyAsync(m->buf, feat, fb, cudaMemcpyDefault, m->stream));
    MC_CUDA_TRY(cudaMemcpyAsync((char *)m->buf + fb, label, lb, cudaMemcpyDefault, m->stream));
    df = m->buf;
    dl = (char *)m->buf + fb;
  }
  MC_CUDA_TRY(cudaFuncSetAttribute(grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem)));
  if (!m->part) {  // made by the first gradient: a network that only scores needs none
    int per_sm = 0;
    MC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, grad_kernel, kGT, sizeof(GradSmem)));
    const int most = std::max(per_sm, 1) * std::max(m->sm_count, 1);  // the blocks that run at once
    MC_CUDA_TRY(cudaMalloc(&m->part, (size_t)(most + 2) * kPart * 4));
    m->part_blocks = most;
    m->grad = m->part + (size_t)most * kPart;
    m->loss = m->grad + kPart;
  }
  const int64_t tiles = (n + kGR - 1) / kGR;
  const int blocks = (int)std::min<int64_t>(tiles, m->part_blocks);
  grad_kernel<<<blocks, kGT, sizeof(GradSmem), m->stream>>>(n, (const float *)df, (const float *)dl, pos_weight, m->wbf,
                                                            m->master, m->part);
  grad_sum_kernel<<<kPart / 32, kRT, 0, m->stream>>>(blocks, m->part, m->grad, m->loss);
  g_launches += 2;
  MC_CUDA_TRY(cudaGetLastError());
  return MC_OK;
}

int mc_mlp_gradient(mc_mlp *m, const float *feat, const float *label, int64_t n, float pos_weight, float *grad_out,
                    float *loss_out) {
  if (!m || n <= 0 || !feat || !label || !grad_out) return MC_ERR_ARG;
  MC_TRY(run_grad(m, feat, label, n, pos_weight));
  MC_CUDA_TRY(cudaMemcpyAsync(grad_out, m->grad, kParams * 4, cudaMemcpyDefault, m->stream));
  float *hl = (float *)m->h_small;
  MC_CUDA_TRY(cudaMemcpyAsync(hl, m->loss, 4, cudaMemcpyDeviceToHost, m->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(m->stream));
  if (loss_out) *loss_out = *hl;
  return MC_OK;
}

int mc_mlp_train_step(mc_mlp *m, const float *feat, const float *label, int64_t n, float pos_weight, float lr,
                      float *loss_out) {
  if (!m || n <= 0 || !feat || !label || !(lr > 0.f)) return MC_ERR_ARG;
  MC_TRY(run_grad(m, feat, label, n, pos_weight));
  m->step++;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)m->step), c2 = 1.f - powf(b2, (float)m->step);
  adam_kernel<<<(kParams + 255) / 256, 256, 0, m->stream>>>(m->master, m->wbf, m->grad, m->m, m->v, lr, b1, b2, 1e-8f,
                                                            c1, c2);
  g_launches++;
  MC_CUDA_TRY(cudaGetLastError());
  float *hl = (float *)m->h_small;
  MC_CUDA_TRY(cudaMemcpyAsync(hl, m->loss, 4, cudaMemcpyDeviceToHost, m->stream));
  MC_CUDA_TRY(cudaStreamSynchronize(m->stream));
  if (loss_out) *loss_out = *hl;
  return MC_OK;
}

}  // extern "C"
