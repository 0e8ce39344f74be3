// jet_kv_compact: commit of the accepted path.  One launch: a cluster of 8 CTAs per sequence copies the K and V rows of
// every accepted node of every layer behind the prefix (contiguous or paged cache) and, once every CTA of the cluster has
// read the old length, advances seq_len.  jet_kv_compact_tail: the same in place, for a cache that holds the tree's rows
// behind the prefix.
//
// Bound: latency (a step commits 0.1 - 3 MB).  The chain is lengths -> path and page table -> rows, three round trips; the rows of
// a sequence are spread over the warps of its cluster with all loads of a warp in flight at once.  (A block per row or
// (layer, K|V) with a second launch for the lengths, as before, cost a launch more: about 2 us of GPU time in a
// captured step and 2.3 us of host time in one issued call by call.)
#include "jet_common.cuh"
#include "sm100_ptx.cuh"

namespace jet {
namespace {

constexpr int kCommitCluster = 8;
constexpr int kCommitThreads = 512;
constexpr int kCommitWarps = kCommitCluster * kCommitThreads / 32;      // warps of a cluster

struct CommitParams {
  int64_t layer_stride16, batch_stride16;            // in 16-byte pieces
  const int32_t* page_table;
  const int32_t* path;
  const int32_t* accept_len;
  int32_t* seq_len;
  int max_pages, page_size, layers, batch, B, row16, N;
};

// The path of sequence b and where its rows lie, worked out once per CTA: node[i] (-1: not to be copied) and the cache row
// offsets (within a layer) of position seq_len + i and -- in-place layout -- seq_len + node[i].
struct CommitTable {
  int64_t dst[JET_MAX_DEPTH + 1], src[JET_MAX_DEPTH + 1];
  int node[JET_MAX_DEPTH + 1];
};

template <bool kTail>
__device__ __forceinline__ int commit_table(const CommitParams& p, int b, CommitTable& t) {
  const int a = min(p.accept_len[b], p.N);
  const int64_t len = p.seq_len[b];
  auto row_of = [&](int64_t pos) -> int64_t {        // -1: outside the page table (a length beyond it is the caller's error)
    if (pos < 0) return -1;
    if (!p.page_table) return b * p.batch_stride16 + pos * p.row16;
    if (pos / p.page_size >= p.max_pages) return -1;
    const int page = p.page_table[static_cast<size_t>(b) * p.max_pages + pos / p.page_size];
    return (static_cast<int64_t>(page) * p.page_size + pos % p.page_size) * p.row16;
  };
  for (int i = threadIdx.x; i <= a; i += kCommitThreads) {
    int node = p.path[static_cast<size_t>(b) * (p.N + 1) + i];
    if (node < 0 || node >= p.B) node = -1;
    const int64_t dst = row_of(len + i), src = kTail && node >= 0 ? row_of(len + node) : 0;
    if (dst < 0 || src < 0) node = -1;
    t.node[i] = node;
    t.dst[i] = dst;
    t.src[i] = src;
  }
  __syncthreads();
  // every CTA has read the length: one of them may advance it
  __syncwarp();
  ptx::cluster_sync_all();
  if (threadIdx.x == 0 && ptx::cluster_ctarank() == 0) p.seq_len[b] = static_cast<int32_t>(len) + p.accept_len[b] + 1;
  return a;
}

__global__ void __launch_bounds__(kCommitThreads)
kv_compact_kernel(const uint4* __restrict__ tree_k, const uint4* __restrict__ tree_v, uint4* __restrict__ k_cache,
                  uint4* __restrict__ v_cache, const CommitParams p) {
  grid_dependency_wait();
  __shared__ CommitTable t;
  const int b = blockIdx.x / kCommitCluster;
  const int a = commit_table<false>(p, b, t);
  if (a < 0) return;
  const int lane = threadIdx.x & 31;
  const int rows = 2 * p.layers * (a + 1);           // row r: path entry r mod (a + 1) of (layer, K | V) number r / (a + 1)
  for (int r = (blockIdx.x % kCommitCluster) * (kCommitThreads / 32) + (threadIdx.x >> 5); r < rows; r += kCommitWarps) {
    const int lk = r / (a + 1), i = r - lk * (a + 1), layer = lk >> 1;
    const int node = t.node[i];
    if (node < 0) continue;
    const uint4* src = ((lk & 1) ? tree_v : tree_k) + ((static_cast<int64_t>(layer) * p.batch + b) * p.B + node) * p.row16;
    uint4* dst = ((lk & 1) ? v_cache : k_cache) + layer * p.layer_stride16 + t.dst[i];
    int e = lane;
    for (; e + 96 < p.row16; e += 128) {
      uint4 x[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) x[k] = __ldg(src + e + 32 * k);
#pragma unroll
      for (int k = 0; k < 4; ++k) dst[e + 32 * k] = x[k];
    }
    for (; e < p.row16; e += 32) dst[e] = __ldg(src + e);
  }
}

// In place: row seq_len + path[i] moves to seq_len + i for i = 1 .. accept_len (path[i] >= i; the root stays where it is).
// One warp per (layer, K | V, 32 of the row's 16-byte columns); columns do not meet, so a lane's own order is all that
// counts: it reads kTailHeld rows into registers before it writes any, and never writes a row that it still has to read,
// because rows are taken in increasing i and path[i] >= i, path increasing.  (With a warp per (layer, K | V) few layers
// left most of the cluster idle: 36 layers of 8 heads of 128, four rows: 9.7 -> 7.0 us.)
constexpr int kTailHeld = 16;

__global__ void __launch_bounds__(kCommitThreads)
kv_compact_tail_kernel(uint4* k_cache, uint4* v_cache, const CommitParams p) {
  grid_dependency_wait();
  __shared__ CommitTable t;
  const int b = blockIdx.x / kCommitCluster;
  const int a = commit_table<true>(p, b, t);
  const int lane = threadIdx.x & 31, blocks = (p.row16 + 31) / 32;
  for (int u = (blockIdx.x % kCommitCluster) * (kCommitThreads / 32) + (threadIdx.x >> 5); u < 2 * p.layers * blocks; u += kCommitWarps) {
    const int lk = u / blocks, column = (u - lk * blocks) * 32 + lane;
    if (column >= p.row16) continue;
    uint4* cache = ((lk & 1) ? v_cache : k_cache) + (lk >> 1) * p.layer_stride16 + column;
    for (int i0 = 1; i0 <= a; i0 += kTailHeld) {
      uint4 held[kTailHeld];
#pragma unroll
      for (int k = 0; k < kTailHeld; ++k)
        if (i0 + k <= a && t.node[i0 + k] >= 0) held[k] = cache[t.src[i0 + k]];
#pragma unroll
      for (int k = 0; k < kTailHeld; ++k)
        if (i0 + k <= a && t.node[i0 + k] >= 0 && t.node[i0 + k] != i0 + k) cache[t.dst[i0 + k]] = held[k];
    }
  }
}

}  // namespace
}  // namespace jet

extern "C" jet_status jet_kv_compact(const void* tree_k, const void* tree_v, void* k_cache,
                                     void* v_cache, int64_t cache_layer_stride,
                                     int64_t kv_batch_stride, const int32_t* page_table,
                                     int max_pages_per_seq, int page_size, const int32_t* path,
                                     const int32_t* accept_len, int32_t* seq_len, int layers,
                                     int batch, int B, int Hkv, int D, int N, void* stream) {
  using namespace jet;
  if (!tree_k || !tree_v || !k_cache || !v_cache || !path || !accept_len || !seq_len)
    return JET_ERR_INVALID_ARG;
  if (layers < 1 || layers > 65535 || batch < 1 || batch > 65535 || B < 1 || B > JET_MAX_NODES ||
      Hkv < 1 || D < 1 || N < 1 || N > JET_MAX_DEPTH)
    return JET_ERR_INVALID_ARG;
  const int64_t row_elems = static_cast<int64_t>(Hkv) * D;
  if (row_elems % 8 != 0 || cache_layer_stride % 8 != 0) return JET_ERR_INVALID_ARG;   // 16-byte rows
  if (!aligned(tree_k, 16) || !aligned(tree_v, 16) || !aligned(k_cache, 16) || !aligned(v_cache, 16))
    return JET_ERR_INVALID_ARG;
  if (page_table) {
    if (page_size < 1 || max_pages_per_seq < 1) return JET_ERR_INVALID_ARG;
  } else if (kv_batch_stride % 8 != 0 || kv_batch_stride < 0) {
    return JET_ERR_INVALID_ARG;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int row16 = static_cast<int>(row_elems / 8);
  const CommitParams p{cache_layer_stride / 8, kv_batch_stride / 8, page_table, path, accept_len, seq_len,
                       max_pages_per_seq, page_size, layers, batch, B, row16, N};
  launch_dependent_cluster(kv_compact_kernel, dim3(kCommitCluster * batch), dim3(kCommitThreads), kCommitCluster, st,
      static_cast<const uint4*>(tree_k), static_cast<const uint4*>(tree_v), static_cast<uint4*>(k_cache),
      static_cast<uint4*>(v_cache), p);
  return launch_status();
}

extern "C" jet_status jet_kv_compact_tail(void* k_cache, void* v_cache, int64_t cache_layer_stride,
                                          int64_t kv_batch_stride, const int32_t* page_table,
                                          int max_pages_per_seq, int page_size, const int32_t* path,
                                          const int32_t* accept_len, int32_t* seq_len, int layers, int batch,
                                          int B, int Hkv, int D, int N, void* stream) {
  using namespace jet;
  if (!k_cache || !v_cache || !path || !accept_len || !seq_len) return JET_ERR_INVALID_ARG;
  if (layers < 1 || layers > 65535 || batch < 1 || B < 1 || B > JET_MAX_NODES || Hkv < 1 || D < 1 || N < 1 ||
      N > JET_MAX_DEPTH)
    return JET_ERR_INVALID_ARG;
  const int64_t row_elems = static_cast<int64_t>(Hkv) * D;
  if (row_elems % 8 != 0 || cache_layer_stride % 8 != 0) return JET_ERR_INVALID_ARG;   // 16-byte rows
  if (!aligned(k_cache, 16) || !aligned(v_cache, 16)) return JET_ERR_INVALID_ARG;
  if (page_table) {
    if (page_size < 1 || max_pages_per_seq < 1) return JET_ERR_INVALID_ARG;
  } else if (kv_batch_stride % 8 != 0 || kv_batch_stride < 0) {
    return JET_ERR_INVALID_ARG;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int row16 = static_cast<int>(row_elems / 8);
  const CommitParams p{cache_layer_stride / 8, kv_batch_stride / 8, page_table, path, accept_len, seq_len,
                       max_pages_per_seq, page_size, layers, batch, B, row16, N};
  launch_dependent_cluster(kv_compact_tail_kernel, dim3(kCommitCluster * batch), dim3(kCommitThreads), kCommitCluster, st,
      static_cast<uint4*>(k_cache), static_cast<uint4*>(v_cache), p);
  return launch_status();
}
