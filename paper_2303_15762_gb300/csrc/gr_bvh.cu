// BVH construction on the GPU.
//
// Propagation of a generalized ray under the interactive simplification of the
// paper (Sec. 7.2) is ray tracing, which needs a spatial subdivision of the
// scene (Sec. 1 motivates locality by exactly this).  The paper does not
// describe its structure; the tree here is built by
//   centroid bounds -> 30-bit Morton codes -> 64-bit keys (morton << 32 | id)
//   -> bitonic sort -> agglomerative clustering along the Morton order
//   (PLOC: Meister & Bittner, "Parallel Locally-Ordered Clustering for
//   Bounding Volume Hierarchy Construction", IEEE TVCG 2018): each cluster
//   picks the neighbour within a window of +-8 whose merged box has the least
//   surface area; mutual nearest neighbours merge, the array is compacted, and
//   the loop repeats until one cluster remains.
// Every step is integer work or exact FP32 (min/max, and centroid,
// quantisation and surface-area arithmetic in explicitly rounded single
// precision), ties go to the lower index and node indices come from prefix
// sums, so the result is deterministic and reproducible bit for bit by a CPU
// build of the same algorithm.
#include <algorithm>
#include <cmath>

#include "gr_build.h"

namespace gr {

namespace {

__device__ __forceinline__ unsigned expand_bits(unsigned v) {
  v = (v * 0x00010001u) & 0xFF0000FFu;
  v = (v * 0x00000101u) & 0x0F00F00Fu;
  v = (v * 0x00000011u) & 0xC30C30C3u;
  v = (v * 0x00000005u) & 0x49249249u;
  return v;
}

// Order-preserving integers of floats (for atomic minima and maxima; -0 sorts
// below +0, and both decode to themselves).
__device__ __forceinline__ int ordered(float f) {
  const int i = __float_as_int(f);
  return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float unordered(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }

// What the build's kernels pass on through device memory, so that the host
// waits for none of them until the tree is done.
constexpr int kMaxLevels = 256;
struct BuildState {
  int clo[3], chi[3];   // centroid bounds as ordered integers
  int lo[3], hi[3];     // vertex bounds as ordered integers
  int bad, small;       // coordinates out of the grid's range; triangles smaller than kSmallSteps grid steps
  int deep;             // a walk of the 4-wide grid nodes could need more than kGridStackDepth entries
  GridDesc g;
  int m[2], created[2]; // clusters left and nodes created, by parity of the round
  int tiles_done;       // tiles of the round that have counted their pairs
  int level_first[kMaxLevels + 1], level_count[kMaxLevels + 1];  // wide nodes of each level
};
__global__ void k_build_init(BuildState* B, int n) {
  const int t = threadIdx.x;
  if (t < 3) {
    B->clo[t] = B->lo[t] = 0x7fffffff;
    B->chi[t] = B->hi[t] = (int)0x80000000;
  }
  if (t == 0) {
    B->bad = B->small = B->deep = B->tiles_done = 0;
    B->m[0] = n;
    B->created[0] = 0;
  }
  for (int l = t; l <= kMaxLevels; l += blockDim.x) {
    B->level_first[l] = 0;
    B->level_count[l] = l == 0 ? 1 : 0;
  }
}

// Centroids, and the bounds of centroids and vertices (exact min/max: a warp
// reduction and one atomic per warp).
__global__ void __launch_bounds__(256) k_centroids(const float* __restrict__ verts, int n, float4* __restrict__ cen,
                                                   BuildState* B) {
  int clo[3], chi[3], lo[3], hi[3];
  for (int a = 0; a < 3; ++a) {
    clo[a] = lo[a] = 0x7fffffff;
    chi[a] = hi[a] = (int)0x80000000;
  }
  bool bad = false;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float* v = verts + 9 * (size_t)i;
    float c[3];
    for (int a = 0; a < 3; ++a) {
      c[a] = __fdiv_rn(__fadd_rn(__fadd_rn(v[a], v[3 + a]), v[6 + a]), 3.0f);
      // a centroid that is not a number leaves the bounds as they are
      if (c[a] == c[a]) {
        clo[a] = min(clo[a], ordered(c[a]));
        chi[a] = max(chi[a], ordered(c[a]));
      }
      for (int k = 0; k < 3; ++k) {
        const float x = v[3 * k + a];
        bad = bad || !(fabsf(x) <= 1e12f);
        lo[a] = min(lo[a], ordered(x));
        hi[a] = max(hi[a], ordered(x));
      }
    }
    cen[i] = make_float4(c[0], c[1], c[2], 0.0f);
  }
  // one set of atomics per block
  __shared__ int s_b[12][8];
  __shared__ int s_bad;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int a = 0; a < 3; ++a) {
    const int v[4] = {__reduce_min_sync(0xffffffffu, clo[a]), __reduce_max_sync(0xffffffffu, chi[a]),
                      __reduce_min_sync(0xffffffffu, lo[a]), __reduce_max_sync(0xffffffffu, hi[a])};
    if (lane == 0)
      for (int k = 0; k < 4; ++k) s_b[4 * a + k][warp] = v[k];
  }
  if (bad) s_bad = 1;
  __syncthreads();
  if (threadIdx.x < 12) {
    const int a = threadIdx.x >> 2, k = threadIdx.x & 3;
    int v = s_b[threadIdx.x][0];
    for (int w = 1; w < 8; ++w) v = k & 1 ? max(v, s_b[threadIdx.x][w]) : min(v, s_b[threadIdx.x][w]);
    int* at = k == 0 ? &B->clo[a] : k == 1 ? &B->chi[a] : k == 2 ? &B->lo[a] : &B->hi[a];
    if (k & 1) atomicMax(at, v);
    else atomicMin(at, v);
  }
  if (threadIdx.x == 0 && s_bad) B->bad = 1;
}

__global__ void k_morton(const float4* __restrict__ cen, int n, int n_pad, const BuildState* __restrict__ B,
                         unsigned long long* __restrict__ keys) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_pad) return;
  if (i >= n) {
    keys[i] = ~0ull;
    return;
  }
  float4 c = cen[i];
  float cc[3] = {c.x, c.y, c.z};
  unsigned q[3];
  for (int a = 0; a < 3; ++a) {
    const float lo = unordered(B->clo[a]);
    float ext = __fsub_rn(unordered(B->chi[a]), lo);
    float t = ext > 0.0f ? __fdiv_rn(__fsub_rn(cc[a], lo), ext) : 0.0f;
    int qi = (int)__fmul_rn(t, 1024.0f);
    qi = qi < 0 ? 0 : (qi > 1023 ? 1023 : qi);
    q[a] = (unsigned)qi;
  }
  unsigned m = expand_bits(q[0]) * 4u + expand_bits(q[1]) * 2u + expand_bits(q[2]);
  keys[i] = ((unsigned long long)m << 32) | (unsigned)i;
}

// Bitonic sorting network (ascending): stages with j >= 1024 run one global
// pass each; all stages with j < 1024 of one k run in shared memory.
__global__ void k_bitonic_global(unsigned long long* keys, int n_pad, int j, int k) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_pad / 2) return;
  int a = 2 * j * (t / j) + (t % j);
  int b = a + j;
  unsigned long long x = keys[a], y = keys[b];
  bool up = (a & k) == 0;
  if ((x > y) == up) {
    keys[a] = y;
    keys[b] = x;
  }
}

__global__ void k_bitonic_shared(unsigned long long* keys, int n_pad, int k_first, int k_last) {
  __shared__ unsigned long long s[2048];
  int base = blockIdx.x * 2048;
  s[threadIdx.x] = keys[base + threadIdx.x];
  s[threadIdx.x + 1024] = keys[base + threadIdx.x + 1024];
  __syncthreads();
  for (int k = k_first; k <= k_last; k <<= 1) {
    int jstart = k >> 1;
    if (jstart > 1024) jstart = 1024;
    for (int j = jstart; j >= 1; j >>= 1) {
      int t = threadIdx.x;
      int a = 2 * j * (t / j) + (t % j);
      int b = a + j;
      unsigned long long x = s[a], y = s[b];
      bool up = ((base + a) & k) == 0;
      if ((x > y) == up) {
        s[a] = y;
        s[b] = x;
      }
      __syncthreads();
    }
  }
  keys[base + threadIdx.x] = s[threadIdx.x];
  keys[base + threadIdx.x + 1024] = s[threadIdx.x + 1024];
}

// Gather the triangles into leaf order; tri[3i].w carries the original id.
__global__ void k_reorder(const unsigned long long* __restrict__ keys, int n, const float* __restrict__ verts,
                          const int* __restrict__ tri_mat, float4* __restrict__ tri, int* __restrict__ tmat) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int id = (int)(keys[i] & 0xffffffffu);
  const float* v = verts + 9 * id;
  tri[3 * i] = make_float4(v[0], v[1], v[2], __int_as_float(id));
  tri[3 * i + 1] = make_float4(v[3], v[4], v[5], 0.0f);
  tri[3 * i + 2] = make_float4(v[6], v[7], v[8], 0.0f);
  tmat[i] = tri_mat[id];
}

// ---- PLOC
constexpr int kPlocRadius = 8;

struct Box6 {
  float lo[3], hi[3];
};

__device__ __forceinline__ Box6 box_union(const Box6& a, const Box6& b) {
  Box6 r;
  for (int k = 0; k < 3; ++k) {
    r.lo[k] = fminf(a.lo[k], b.lo[k]);
    r.hi[k] = fmaxf(a.hi[k], b.hi[k]);
  }
  return r;
}

// Half surface area, rounded step by step: ((dx dy) + (dy dz)) + (dz dx).
__device__ __forceinline__ float half_area_rn(const Box6& b) {
  const float dx = __fsub_rn(b.hi[0], b.lo[0]), dy = __fsub_rn(b.hi[1], b.lo[1]), dz = __fsub_rn(b.hi[2], b.lo[2]);
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dy), __fmul_rn(dy, dz)), __fmul_rn(dz, dx));
}

__device__ __forceinline__ Box6 load_box(const float* B, int i) {
  Box6 r;
  for (int k = 0; k < 3; ++k) {
    r.lo[k] = B[6 * i + k];
    r.hi[k] = B[6 * i + 3 + k];
  }
  return r;
}
__device__ __forceinline__ void store_box(float* B, int i, const Box6& b) {
  for (int k = 0; k < 3; ++k) {
    B[6 * i + k] = b.lo[k];
    B[6 * i + 3 + k] = b.hi[k];
  }
}

__global__ void k_leaf_clusters(const float4* __restrict__ tri, int n, float* __restrict__ B, int* __restrict__ C) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 a = tri[3 * i], b = tri[3 * i + 1], c = tri[3 * i + 2];
  Box6 r;
  r.lo[0] = fminf(fminf(a.x, b.x), c.x);
  r.lo[1] = fminf(fminf(a.y, b.y), c.y);
  r.lo[2] = fminf(fminf(a.z, b.z), c.z);
  r.hi[0] = fmaxf(fmaxf(a.x, b.x), c.x);
  r.hi[1] = fmaxf(fmaxf(a.y, b.y), c.y);
  r.hi[2] = fmaxf(fmaxf(a.z, b.z), c.z);
  store_box(B, i, r);
  C[i] = i | 0x80000000;
}

// One cluster's nearest neighbour within the window: least merged area, ties
// to the lower index.  box(j) gives cluster j's box.
template <class BoxFn>
__device__ __forceinline__ int nearest(int i, int m, BoxFn&& box) {
  const Box6 bi = box(i);
  int best = -1;
  float ba = 3.4e38f;
  const int j0 = max(i - kPlocRadius, 0), j1 = min(i + kPlocRadius, m - 1);
  for (int j = j0; j <= j1; ++j) {
    if (j == i) continue;
    const float a = half_area_rn(box_union(bi, box(j)));
    if (a < ba || (a == ba && j < best)) {
      ba = a;
      best = j;
    }
  }
  return best;
}

__device__ __forceinline__ void write_node(float* __restrict__ Nd, const Box6& a, const Box6& b, int ca, int cb) {
  float4* q = (float4*)Nd;
  q[0] = make_float4(a.lo[0], a.lo[1], a.lo[2], a.hi[0]);
  q[1] = make_float4(a.hi[1], a.hi[2], b.lo[0], b.lo[1]);
  q[2] = make_float4(b.lo[2], b.hi[0], b.hi[1], b.hi[2]);
  q[3] = make_float4(__int_as_float(ca), __int_as_float(cb), 0.0f, 0.0f);
}

// A round of the clustering over many blocks is two launches; the cluster
// count is read from device memory, so the host enqueues rounds without
// waiting (blocks beyond the count return, and rounds that start with at most
// kTail clusters do nothing).  Until every round was counted on the host the
// build of 91k triangles waited ~30 times and scanned its flags with one block:
// scene creation 3.3 -> 1.24 ms (1.01M triangles: 23.9 -> 3.8).
constexpr int kTile = 256, kTail = 1024;
constexpr int kPairThreads = kTile + 32;  // the tile and the clusters on either side, a thread each
// Levels of the collapse enqueued at once: n triangles take 1.3 to 1.6 log4(n)
// levels (2: 1, 1172: 8, 5k: 9 or 10, 37k: 12, 92k: 13, 280k: 13 or 14, 1.01M:
// 16), an empty level costs its launch (~2.3 us; with 18 for every scene a
// two-triangle one took 203 us to create, now 151), one too few another wait.
inline int first_levels(int n) { return std::min(n - 1, (int)std::ceil(1.55 * std::log2((double)n) / 2.0) + 1); }
constexpr int kMoreLevels = 8;

// Nearest neighbours of a tile (and of the 8 clusters on either side, whose
// choice decides who is mutual), the pairs that merge, and the tile's counts.
// P[i] = j when i merges with the higher-index j, -1 when i stays, -2 when it
// is merged away.  The last tile to finish turns the counts into their
// exclusive prefixes and sets the next round's cluster and node counts.
__global__ void __launch_bounds__(kPairThreads) k_ploc_pairs(const float* __restrict__ B, BuildState* S, int parity,
                                                             int* __restrict__ P, int2* sums) {
  const int m = S->m[parity], created = S->created[parity], start = blockIdx.x * kTile, t = threadIdx.x;
  if (m <= kTail) {
    if (blockIdx.x == 0 && t == 0) {
      S->m[parity ^ 1] = m;
      S->created[parity ^ 1] = created;
    }
    return;
  }
  if (start >= m) return;
  constexpr int H = 2 * kPlocRadius;
  __shared__ float s_box[(kTile + 2 * H) * 6];
  __shared__ int s_nn[kTile + H];
  __shared__ int2 s_cnt[kPairThreads / 32];
  __shared__ int2 s_part[kPairThreads];
  __shared__ int s_last;
  const int first = max(start - H, 0), last = min(start + kTile + H, m);
  for (int i = t; i < (last - first) * 6; i += kPairThreads) s_box[i] = B[6 * (size_t)first + i];
  __syncthreads();
  auto box = [&](int j) { return load_box(s_box, j - first); };
  const int c = start - kPlocRadius + t;  // the thread's cluster
  if (t < kTile + H) s_nn[t] = c >= 0 && c < m ? nearest(c, m, box) : -1;
  __syncthreads();
  bool merges = false, stays = false;
  if (t >= kPlocRadius && t < kTile + kPlocRadius && c < m) {
    const int j = s_nn[t];
    const bool mutual = j >= 0 && s_nn[j - start + kPlocRadius] == c;
    merges = mutual && c < j;
    stays = !(mutual && j < c);
    P[c] = merges ? j : stays ? -1 : -2;
  }
  const unsigned a = __ballot_sync(0xffffffffu, merges), b = __ballot_sync(0xffffffffu, stays);
  if ((t & 31) == 0) s_cnt[t >> 5] = make_int2(__popc(a), __popc(b));
  __syncthreads();
  const int tiles = (m + kTile - 1) / kTile;
  if (t == 0) {
    int2 n = make_int2(0, 0);
    for (int w = 0; w < kPairThreads / 32; ++w) {
      n.x += s_cnt[w].x;
      n.y += s_cnt[w].y;
    }
    sums[blockIdx.x] = n;
    __threadfence();
    s_last = atomicAdd(&S->tiles_done, 1) == tiles - 1;
  }
  __syncthreads();
  if (!s_last) return;
  // a contiguous chunk of tiles per thread, a scan of the partial sums, the chunk's prefixes
  __threadfence();
  const int chunk = (tiles + kPairThreads - 1) / kPairThreads;
  const int lo = min(t * chunk, tiles), hi = min(lo + chunk, tiles);
  int2 acc = make_int2(0, 0);
  for (int i = lo; i < hi; ++i) {
    const int2 v = __ldcg(&sums[i]);
    acc.x += v.x;
    acc.y += v.y;
  }
  s_part[t] = acc;
  __syncthreads();
  for (int off = 1; off < kPairThreads; off <<= 1) {
    const int2 v = t >= off ? s_part[t - off] : make_int2(0, 0);
    __syncthreads();
    s_part[t].x += v.x;
    s_part[t].y += v.y;
    __syncthreads();
  }
  int2 run = t > 0 ? s_part[t - 1] : make_int2(0, 0);
  for (int i = lo; i < hi; ++i) {
    const int2 v = __ldcg(&sums[i]);
    sums[i] = run;
    run.x += v.x;
    run.y += v.y;
  }
  if (t == kPairThreads - 1) {
    S->m[parity ^ 1] = s_part[t].y;
    S->created[parity ^ 1] = created + s_part[t].x;
    S->tiles_done = 0;
  }
}

// Merge the pairs into new nodes (index (n-2) - creation order, so the root,
// created last, is node 0) and compact the clusters in order.
__global__ void __launch_bounds__(kTile) k_ploc_merge(const float* __restrict__ B, const int* __restrict__ C,
                                                      const int* __restrict__ P, const int2* __restrict__ sums,
                                                      const BuildState* __restrict__ S, int parity, int n,
                                                      float* __restrict__ B2, int* __restrict__ C2,
                                                      float* __restrict__ nodes) {
  const int m = S->m[parity], start = blockIdx.x * kTile;
  if (start >= m) return;
  const int i = start + threadIdx.x;
  if (m <= kTail) {  // the round is over before it began: the clusters move to the other buffer
    if (i < m) {
      store_box(B2, i, load_box(B, i));
      C2[i] = C[i];
    }
    return;
  }
  __shared__ int2 s_cnt[kTile / 32];
  const int j = i < m ? P[i] : -2;
  const unsigned a = __ballot_sync(0xffffffffu, j >= 0), c = __ballot_sync(0xffffffffu, j >= -1);
  if ((threadIdx.x & 31) == 0) s_cnt[threadIdx.x >> 5] = make_int2(__popc(a), __popc(c));
  __syncthreads();
  if (j == -2) return;
  const unsigned below = (1u << (threadIdx.x & 31)) - 1u;
  int2 pos = sums[blockIdx.x];
  for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) {
    pos.x += s_cnt[w].x;
    pos.y += s_cnt[w].y;
  }
  pos.x += __popc(a & below);
  pos.y += __popc(c & below);
  const Box6 bi = load_box(B, i);
  if (j >= 0) {
    const Box6 bj = load_box(B, j);
    const int x = (n - 2) - (S->created[parity] + pos.x);
    write_node(nodes + 16 * (size_t)x, bi, bj, C[i], C[j]);
    store_box(B2, pos.y, box_union(bi, bj));
    C2[pos.y] = x;
  } else {
    store_box(B2, pos.y, bi);
    C2[pos.y] = C[i];
  }
}

// The last rounds, from at most kTail clusters to one, in one block's shared
// memory (one cluster per thread).
__global__ void __launch_bounds__(kTail) k_ploc_tail(const float* __restrict__ B, const int* __restrict__ C,
                                                     BuildState* S, int parity, int n, float* __restrict__ nodes) {
  int m = S->m[parity], created = S->created[parity];
  if (m > kTail) return;
  __shared__ float s_box[kTail * 6];
  __shared__ int s_id[kTail], s_nn[kTail];
  __shared__ int2 s_cnt[kTail / 32];
  const int i = threadIdx.x, warp = i >> 5;
  const unsigned below = (1u << (i & 31)) - 1u;
  for (int q = i; q < 6 * m; q += kTail) s_box[q] = B[q];
  if (i < m) s_id[i] = C[i];
  __syncthreads();
  auto box = [&](int j) { return load_box(s_box, j); };
  // a round with more than one cluster merges at least one pair: at most kTail - 1 rounds
  for (int round = 0; m > 1 && round < kTail; ++round) {
    if (i < m) s_nn[i] = nearest(i, m, box);
    __syncthreads();
    const int j = i < m ? s_nn[i] : -1;
    const bool mutual = j >= 0 && s_nn[j] == i;
    const bool merges = mutual && i < j, stays = i < m && !(mutual && j < i);
    const unsigned a = __ballot_sync(0xffffffffu, merges), c = __ballot_sync(0xffffffffu, stays);
    if ((i & 31) == 0) s_cnt[warp] = make_int2(__popc(a), __popc(c));
    Box6 bi, bj;
    int id = 0, idj = 0;
    if (stays) {
      bi = box(i);
      id = s_id[i];
    }
    if (merges) {
      bj = box(j);
      idj = s_id[j];
    }
    __syncthreads();
    int2 pos = make_int2(0, 0), tot = make_int2(0, 0);
    const int warps = (m + 31) >> 5;
    for (int w = 0; w < warps; ++w) {
      const int2 v = s_cnt[w];
      if (w < warp) {
        pos.x += v.x;
        pos.y += v.y;
      }
      tot.x += v.x;
      tot.y += v.y;
    }
    pos.x += __popc(a & below);
    pos.y += __popc(c & below);
    if (merges) {
      const int x = (n - 2) - (created + pos.x);
      write_node(nodes + 16 * (size_t)x, bi, bj, id, idj);
      bi = box_union(bi, bj);
      id = x;
    }
    if (stays) {
      store_box(s_box, pos.y, bi);
      s_id[pos.y] = id;
    }
    created += tot.x;
    m = tot.y;
    __syncthreads();
  }
  if (i == 0) {
    S->m[parity] = m;
    S->created[parity] = created;
  }
}

inline cudaError_t launch_sort(unsigned long long* keys, int n_pad, cudaStream_t st) {
  // n_pad is a power of two >= 2048
  int blocks_sh = n_pad / 2048;
  k_bitonic_shared<<<blocks_sh, 1024, 0, st>>>(keys, n_pad, 2, 2048);
  for (int k = 4096; k <= n_pad; k <<= 1) {
    for (int j = k >> 1; j >= 2048; j >>= 1) {
      int threads = n_pad / 2;
      k_bitonic_global<<<(threads + 255) / 256, 256, 0, st>>>(keys, n_pad, j, k);
    }
    k_bitonic_shared<<<blocks_sh, 1024, 0, st>>>(keys, n_pad, k, k);
  }
  return cudaGetLastError();
}

}  // namespace

// ------------------------------------------------------------------ 4-wide quantised BVH
// Derived from the binary LBVH: each wide node takes a binary node and expands
// its largest-area internal child until it has up to four children.  A wide
// node stores its box origin P (float32), one power-of-two scale 2^e per axis
// and 8-bit child bounds q with  P + qlo 2^e <= child lo  and  P + qhi 2^e >=
// child hi, computed with directed rounding, so every decoded box
// contains its child: the traversal can only visit more, never miss a hit.
// Layout (64 bytes = 4 x uint4):
//   w0..2 P.xyz, w3 = e.x | e.y << 8 | e.z << 16 (biased by 128) | count << 24
//   w4..9 child bytes: qlo.x[4], qlo.y[4], qlo.z[4], qhi.x[4], qhi.y[4], qhi.z[4]
//   w10..13 child references (bit 31 set = leaf slot; -1 = empty)
//   w14..15 unused

namespace {

struct BoxF {
  float lo[3], hi[3];
};

__device__ __forceinline__ BoxF leaf_box(const float4* tri, int slot) {
  const float4 a = tri[3 * slot], b = tri[3 * slot + 1], c = tri[3 * slot + 2];
  BoxF r;
  r.lo[0] = fminf(fminf(a.x, b.x), c.x);
  r.lo[1] = fminf(fminf(a.y, b.y), c.y);
  r.lo[2] = fminf(fminf(a.z, b.z), c.z);
  r.hi[0] = fmaxf(fmaxf(a.x, b.x), c.x);
  r.hi[1] = fmaxf(fmaxf(a.y, b.y), c.y);
  r.hi[2] = fmaxf(fmaxf(a.z, b.z), c.z);
  return r;
}

__device__ __forceinline__ BoxF ref_box(int ref, const float* nbox, const float4* tri) {
  if (ref < 0) return leaf_box(tri, ref & 0x7fffffff);
  BoxF b;
  for (int k = 0; k < 3; ++k) {
    b.lo[k] = nbox[6 * ref + k];
    b.hi[k] = nbox[6 * ref + 3 + k];
  }
  return b;
}

__device__ __forceinline__ float half_area(const BoxF& b) {
  const float dx = b.hi[0] - b.lo[0], dy = b.hi[1] - b.lo[1], dz = b.hi[2] - b.lo[2];
  return dx * dy + dy * dz + dz * dx;
}

// The 16-bit grid of a scene: its bounds in 65535 steps per axis.  It serves
// unless a coordinate is not finite or beyond 1e12, a walk of the tree could
// need more than the kGridStackDepth entries it has, or it is so coarse against
// the triangles (more than one in 16 smaller than kSmallSteps steps) that their
// boxes swell by more than the 4-wide walk saves; the renders of such a scene
// walk the FP32 nodes.  k_trace of a 512^2 x 16 spp view of procedural objects
// of 1 m on a ground that stretches the grid, grid nodes against FP32 nodes
// (us): 83k triangles on 32 / 64 / 96 / 256 m 4165 / 5243 / 6747 / 11506
// against 4637 / 5845 / 6385 / 7499; 7k on 128 / 256 m 4259 / 5254 against 4523
// / 5086; 374k on 32 / 48 m 6312 / 8511 against 6769 / 8411; the first object
// beside as many large triangles on 64 / 96 m 5506 / 6732 against 5702 / 6206.
// In each of them the first ground where the grid loses is the first with
// triangles smaller than 2 steps (11% to 24% of them).  Beyond the line the
// binary FP16 nodes of before took 2 to 7% less than the FP32 nodes, and the
// renders, with what surrounds the trace, no less.  The same
// launch stores the box of every binary internal node (from its parent's
// child boxes).
constexpr float kSmallSteps = 2.0f;
__global__ void __launch_bounds__(256) k_grid_steps(const float4* __restrict__ tri, const float* __restrict__ nodes, int n,
                                                    BuildState* S, int parity, float* __restrict__ nbox,
                                                    int2* __restrict__ front) {
  if (S->m[parity] != 1) return;  // the clustering needs more rounds
  GridDesc g;
  float widest = 0.0f;
  for (int a = 0; a < 3; ++a) {
    g.lo[a] = unordered(S->lo[a]);
    g.step[a] = fmaxf((float)(((double)unordered(S->hi[a]) - (double)g.lo[a]) / 65535.0 * (1.0 + 1e-6)), 1e-25f);
    widest = fmaxf(widest, g.step[a]);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    S->g = g;
    front[0] = make_int2(0, 0);  // wide node 0 stands for the root
  }
  int small = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const BoxF b = leaf_box(tri, i);
    small += fmaxf(fmaxf(b.hi[0] - b.lo[0], b.hi[1] - b.lo[1]), b.hi[2] - b.lo[2]) < kSmallSteps * widest;
    if (i >= n - 1) continue;
    const float4* q = (const float4*)(nodes + 16 * (size_t)i);
    const float4 q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3];
    const float N[12] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x, q2.y, q2.z, q2.w};
    const int l = __float_as_int(q3.x), r = __float_as_int(q3.y);
    if (l >= 0)
      for (int k = 0; k < 6; ++k) nbox[6 * (size_t)l + k] = N[k];
    if (r >= 0)
      for (int k = 0; k < 6; ++k) nbox[6 * (size_t)r + k] = N[6 + k];
    if (i == 0)
      for (int k = 0; k < 3; ++k) {
        nbox[k] = fminf(N[k], N[6 + k]);
        nbox[3 + k] = fmaxf(N[3 + k], N[9 + k]);
      }
  }
  small = __reduce_add_sync(0xffffffffu, small);
  if ((threadIdx.x & 31) == 0 && small) atomicAdd(&S->small, small);
}

// One level of the top-down collapse.  front[w] is the binary node that wide
// node w stands for, and the most entries a walk that enters w can have on its
// stack: every node on the way pushed its internal children but the one walked
// next.  (A bound by levels would not do: the way to w may have taken a wide
// level for each binary one, with three entries left at each.)  Level L's nodes
// are [level_first[L], + level_count[L]), and a node's internal children take
// consecutive places in the next level.
__global__ void __launch_bounds__(128) k_collapse(const float* __restrict__ nodes, const float* __restrict__ nbox,
                                                  const float4* __restrict__ tri, int2* __restrict__ front,
                                                  BuildState* S, int parity, int level, uint4* __restrict__ wn,
                                                  uint4* __restrict__ gn) {
  if (S->m[parity] != 1) return;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int first = S->level_first[level], count = S->level_count[level];
  if (t == 0) S->level_first[level + 1] = first + count;
  if (t >= count) return;
  const GridDesc g = S->g;
  const int widx = first + t, bnode = front[widx].x;
  int below = front[widx].y;
  int ch[4];
  int cnt = 2;
  ch[0] = __float_as_int(nodes[16 * bnode + 12]);
  ch[1] = __float_as_int(nodes[16 * bnode + 13]);
  while (cnt < 4) {
    int best = -1;
    float ba = -1.0f;
    for (int k = 0; k < cnt; ++k)
      if (ch[k] >= 0) {
        float a = half_area(ref_box(ch[k], nbox, tri));
        if (a > ba) {
          ba = a;
          best = k;
        }
      }
    if (best < 0) break;
    const int x = ch[best];
    ch[best] = __float_as_int(nodes[16 * x + 12]);
    ch[cnt++] = __float_as_int(nodes[16 * x + 13]);
  }
  BoxF cb[4];
  BoxF W;
  for (int k = 0; k < 3; ++k) {
    W.lo[k] = 3.4e38f;
    W.hi[k] = -3.4e38f;
  }
  for (int c = 0; c < cnt; ++c) {
    cb[c] = ref_box(ch[c], nbox, tri);
    for (int k = 0; k < 3; ++k) {
      W.lo[k] = fminf(W.lo[k], cb[c].lo[k]);
      W.hi[k] = fmaxf(W.hi[k], cb[c].hi[k]);
    }
  }
  // All of this in FP32 with directed rounding (lower bounds down, upper ones
  // up); in FP64 the launches of the collapse took 0.7 ms of a 92k-triangle
  // build, now 0.15.
  unsigned char qlo[3][4], qhi[3][4];
  int ex[3];
  for (int k = 0; k < 3; ++k) {
    // the least power of two 2^e with 255 * 2^e >= the node's extent
    const unsigned r = __float_as_uint(__fdiv_ru(__fsub_ru(W.hi[k], W.lo[k]), 255.0f));
    const int e = r == 0u ? -100 : max((int)(r >> 23) - 127 + ((r & 0x7fffffu) != 0u), -100);
    ex[k] = e;
    const float sc = __uint_as_float((unsigned)(127 - e) << 23);  // 2^-e
    for (int c = 0; c < 4; ++c) {
      if (c < cnt) {
        qlo[k][c] = (unsigned char)fminf(floorf(__fsub_rd(cb[c].lo[k], W.lo[k]) * sc), 255.0f);
        qhi[k][c] = (unsigned char)fminf(ceilf(__fsub_ru(cb[c].hi[k], W.lo[k]) * sc), 255.0f);
      } else {
        qlo[k][c] = 255;  // empty slot: an inverted box that no ray hits
        qhi[k][c] = 0;
      }
    }
  }
  int refs[4] = {-1, -1, -1, -1};
  int inner = 0;
  for (int c = 0; c < cnt; ++c) inner += ch[c] >= 0;
  below += max(inner - 1, 0);
  if (below > kGridStackDepth) S->deep = 1;
  int w = inner ? first + count + atomicAdd(&S->level_count[level + 1], inner) : 0;
  for (int c = 0; c < cnt; ++c) {
    if (ch[c] < 0) {
      refs[c] = ch[c];
    } else {
      refs[c] = w;
      front[w++] = make_int2(ch[c], below);
    }
  }
  uint4 a, b, c4, d;
  a.x = __float_as_uint(W.lo[0]);
  a.y = __float_as_uint(W.lo[1]);
  a.z = __float_as_uint(W.lo[2]);
  a.w = (unsigned)(ex[0] + 128) | ((unsigned)(ex[1] + 128) << 8) | ((unsigned)(ex[2] + 128) << 16) |
        ((unsigned)cnt << 24);
  auto pack4 = [](const unsigned char* v) {
    return (unsigned)v[0] | ((unsigned)v[1] << 8) | ((unsigned)v[2] << 16) | ((unsigned)v[3] << 24);
  };
  b.x = pack4(qlo[0]);
  b.y = pack4(qlo[1]);
  b.z = pack4(qlo[2]);
  b.w = pack4(qhi[0]);
  c4.x = pack4(qhi[1]);
  c4.y = pack4(qhi[2]);
  c4.z = (unsigned)refs[0];
  c4.w = (unsigned)refs[1];
  d.x = (unsigned)refs[2];
  d.y = (unsigned)refs[3];
  d.z = 0u;
  d.w = 0u;
  for (int c = 0; c < 4; ++c) {
    unsigned w[3];
    for (int k = 0; k < 3; ++k) {
      w[k] = 0xffffu;  // empty: an inverted box
      if (c < cnt) {
        const float lo = floorf(__fmul_rd(__fsub_rd(cb[c].lo[k], g.lo[k]), __frcp_rd(g.step[k])));
        const float hi = ceilf(__fmul_ru(__fsub_ru(cb[c].hi[k], g.lo[k]), __frcp_ru(g.step[k])));
        w[k] = (unsigned)fminf(fmaxf(lo, 0.0f), 65535.0f) | ((unsigned)fminf(fmaxf(hi, 0.0f), 65535.0f) << 16);
      }
    }
    gn[4 * (size_t)widx + c] = make_uint4(w[0], w[1], w[2], c < cnt ? (unsigned)refs[c] : 0x80000000u);
  }
  wn[4 * widx] = a;
  wn[4 * widx + 1] = b;
  wn[4 * widx + 2] = c4;
  wn[4 * widx + 3] = d;
}

}  // namespace

// Build the trees of `n` triangles (device arrays verts [n][9], tri_mat [n]).
// Outputs (device, caller-allocated): tri [n][3] float4, tmat [n], nodes
// [(n-1)][16] floats, keys [n], and the 4-wide nodes wn and gn of up to
// max_wide_nodes(n) each; on the host *n_wide (their count, 0 if n < 2 or the tree is too
// deep for them), *grid (the grid of gn's boxes) and *grid_ok (whether it
// serves the scene).  One scratch allocation;
// the host waits once, for the state the launches leave behind, and again only
// if the clustering or the collapse takes more rounds than were enqueued.
cudaError_t build_trees(const float* verts, const int* tri_mat, int n, float4* tri, int* tmat, float* nodes,
                        unsigned long long* keys_out, uint4* wn, uint4* gn, GridDesc* grid, bool* grid_ok,
                        int* n_wide, cudaStream_t st) {
  *n_wide = 0;
  *grid_ok = false;
  if (n <= 0) return cudaSuccess;
  int n_pad = 2048;
  while (n_pad < n) n_pad <<= 1;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t r = off;
    off += (bytes + 255) / 256 * 256;
    return r;
  };
  const size_t N = (size_t)n, o_state = take(sizeof(BuildState)), o_cen = take(sizeof(float4) * N);
  const size_t o_keys = take(sizeof(unsigned long long) * (size_t)n_pad);
  const size_t o_box = take(sizeof(float) * 6 * 2 * N), o_id = take(sizeof(int) * 2 * N), o_p = take(sizeof(int) * N);
  const size_t o_sums = take(sizeof(int2) * (N / kTile + 1));
  unsigned char* d = nullptr;
  cudaError_t e = dev_alloc((void**)&d, off, st);
  if (e != cudaSuccess) return e;
  BuildState* S = (BuildState*)(d + o_state);
  float4* cen = (float4*)(d + o_cen);
  unsigned long long* keys = (unsigned long long*)(d + o_keys);
  float *Bc = (float*)(d + o_box), *Bn = Bc + 6 * N;
  int *Cc = (int*)(d + o_id), *Cn = Cc + N, *P = (int*)(d + o_p);
  int2* sums = (int2*)(d + o_sums);
  BuildState h;
  auto run = [&]() -> cudaError_t {
    const int g256 = (n + 255) / 256;
    cudaError_t r;
    k_build_init<<<1, 256, 0, st>>>(S, n);
    k_centroids<<<std::min(g256, 1024), 256, 0, st>>>(verts, n, cen, S);
    k_morton<<<(n_pad + 255) / 256, 256, 0, st>>>(cen, n, n_pad, S, keys);
    if ((r = launch_sort(keys, n_pad, st)) != cudaSuccess) return r;
    k_reorder<<<g256, 256, 0, st>>>(keys, n, verts, tri_mat, tri, tmat);
    if ((r = cudaMemcpyAsync(keys_out, keys, sizeof(unsigned long long) * N, cudaMemcpyDeviceToDevice, st)) != cudaSuccess)
      return r;
    if (n == 1) return cudaGetLastError();
    k_leaf_clusters<<<g256, 256, 0, st>>>(tri, n, Bc, Cc);
    // rounds of the many-block form: a round leaves about 0.78 of the clusters
    int parity = 0;
    for (long long bound = n, done = 0; done < n;) {
      int rounds = 0;
      for (double m = (double)bound; m > kTail; m *= 0.78) ++rounds;
      const int tiles = (int)((bound + kTile - 1) / kTile);
      for (int k = 0; k < rounds; ++k) {
        k_ploc_pairs<<<tiles, kPairThreads, 0, st>>>(Bc, S, parity, P, sums);
        k_ploc_merge<<<tiles, kTile, 0, st>>>(Bc, Cc, P, sums, S, parity, n, Bn, Cn, nodes);
        std::swap(Bc, Bn);
        std::swap(Cc, Cn);
        parity ^= 1;
      }
      done += rounds;
      k_ploc_tail<<<1, kTail, 0, st>>>(Bc, Cc, S, parity, n, nodes);
      // the collapse is enqueued with the rounds; its launches return at once
      // if the clustering is not done, and are enqueued again after the next ones
      float* nbox = Bc;  // the cluster boxes and ids have served
      int2* front = (int2*)(d + o_id);  // 2 n ints for at most (2 n - 1) / 3 of them
      k_grid_steps<<<std::min(g256, 1024), 256, 0, st>>>(tri, nodes, n, S, parity, nbox, front);
      int level = 0, batch = first_levels(n);
      do {
        for (int k = 0; k < batch && level < kMaxLevels; ++k, ++level) {
          const double widest = level < 14 ? std::pow(4.0, level) : 3e8;
          const int blocks = (int)((std::min(widest, (double)n) + 127) / 128);
          k_collapse<<<blocks, 128, 0, st>>>(nodes, nbox, tri, front, S, parity, level, wn, gn);
        }
        batch = kMoreLevels;
        if ((r = cudaMemcpyAsync(&h, S, sizeof h, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return r;
        if ((r = cudaStreamSynchronize(st)) != cudaSuccess) return r;
      } while (h.m[parity] == 1 && h.level_count[level] > 0 && level < kMaxLevels);
      if (h.m[parity] == 1) {
        if (h.created[parity] != n - 1) return cudaErrorUnknown;
        // a tree of more than kMaxLevels wide levels (equal boxes merge into a
        // chain: 770 triangles on one another) keeps its binary nodes only
        if (h.level_count[level] > 0) return cudaGetLastError();
        *n_wide = h.level_first[level];
        *grid = h.g;
        *grid_ok = !h.bad && !h.deep && (long long)h.small * 16 <= n;
        return cudaGetLastError();
      }
      if (rounds == 0 || h.m[parity] >= bound) break;  // no pair merges (boxes that are not finite)
      bound = h.m[parity];
    }
    return cudaErrorUnknown;
  };
  e = run();
  cudaFreeAsync(d, st);
  return e;
}

}  // namespace gr
