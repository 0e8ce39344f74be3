// jet_kv_compact: commit of the accepted path: the K and V rows of every accepted node of every layer are copied behind the
// prefix (contiguous or paged cache), then seq_len advances.  jet_kv_compact_tail: the same in place, for a cache that
// holds the tree's rows behind the prefix.
//
// Bound: latency (a step commits 0.1 - 3 MB).  The chain is lengths and path -> page table -> rows; the rows of all
// sequences are spread over the GPU, a warp per row, and a CTA works the path of its sequence out once.  No CTA may see an
// advanced length, so seq_len is advanced by a second launch, or, where one CTA per sequence is enough (kAloneRows), by that
// CTA: the second launch costs 1.7 us of host time.  It starts once all CTAs hold their lengths and runs beside the copies.  (While it
// waited for them before its load and store, a commit of several layers took 0.2 - 0.4 us more: acceptance and commit of 36 layers, 4
// rows, paged: 8.2 against 7.9 us; 32 sequences, 4 layers: 12.9 against 12.6.)
// us per call in a captured stream (a cluster of eight CTAs per sequence before; page size 16, 8 heads of 128 and 36 layers
// where not said otherwise; in place in brackets):
//   1 sequence, 6 rows                  5.3 -> 3.5   [8.1 -> 4.8]      1 sequence, 65 rows    28 -> 5.3  [50 -> 17]
//   32 sequences, 6 rows                11.6 -> 9.9  [22.4 -> 15.0]    128, one layer, 5 rows  10.2 -> 3.3 [23.5 -> 4.8]
//   8 sequences, 48 layers, 4 heads     5.3 -> 4.2   [7.4 -> 5.6]      128, 5 rows            39 -> 37  [61 -> 33]
// Left behind the clusters: 33 - 64 rows of 2 KB in one CTA, 0.4 us (two turns of its warps; a second launch costs a caller
// who issues call by call more than that).
#include "jet_common.cuh"
#include "sm100_ptx.cuh"

namespace jet {
namespace {

// Threads of a CTA; of one that has its sequence to itself.  (With 1024 the copy spills: 52 rows 0.5 us slower.)
constexpr int kCommitThreads = 256, kCommitThreadsAlone = 512;
constexpr int kTailHeld = 16;                        // rows a lane of the in-place form has in flight

struct CommitParams {
  int64_t layer_stride16, batch_stride16;            // in 16-byte pieces
  const int32_t* page_table;
  const int32_t* path;
  const int32_t* accept_len;
  int32_t* seq_len;
  int max_pages, page_size, layers, batch, B, row16, N;
  int ctas;                                          // per sequence
};

// The path of sequence b and where its rows lie: node[i] (-1: not to be copied) and the cache row offsets (within a layer) of
// position seq_len + i and -- in-place layout -- seq_len + node[i].
struct CommitTable {
  int64_t dst[JET_MAX_DEPTH + 1], src[JET_MAX_DEPTH + 1];
  int node[JET_MAX_DEPTH + 1];
};

// Waits for the kernels before this one, fills the table and returns a: entries 0 .. a of the path are committed.  A CTA that
// has its sequence to itself advances seq_len once all its threads have the length; else the launch behind this one does, and
// is let go only now: it starts when every CTA has got here, so that no CTA can read a length that it has advanced.
template <bool kTail>
__device__ __forceinline__ int commit_table(const CommitParams& p, int b, CommitTable& t) {
  const int i = threadIdx.x;
  if (p.ctas == 1) grid_dependency_wait();
  else ptx::grid_dep_wait();
  const int accepted = p.accept_len[b], len = p.seq_len[b];
  int node = i <= p.N ? p.path[static_cast<size_t>(b) * (p.N + 1) + i] : -1;      // (in flight with the lengths)
  const int a = min(accepted, p.N);
  auto row_of = [&](int64_t pos) -> int64_t {        // -1: outside the page table (a length beyond it is the caller's error)
    if (pos < 0) return -1;
    if (!p.page_table) return b * p.batch_stride16 + pos * p.row16;
    if (pos / p.page_size >= p.max_pages) return -1;
    const int page = p.page_table[static_cast<size_t>(b) * p.max_pages + pos / p.page_size];
    return (static_cast<int64_t>(page) * p.page_size + pos % p.page_size) * p.row16;
  };
  if (i <= a) {
    if (node < 0 || node >= p.B) node = -1;
    const int64_t dst = row_of(static_cast<int64_t>(len) + i), src = kTail && node >= 0 ? row_of(static_cast<int64_t>(len) + node) : 0;
    if (dst < 0 || src < 0) node = -1;
    t.node[i] = node;
    t.dst[i] = dst;
    t.src[i] = src;
  }
  __syncthreads();                                   // (the lengths have arrived: they went into the table and a)
  if (p.ctas != 1) ptx::grid_dep_launch();
  else if (threadIdx.x == 0) p.seq_len[b] = len + accepted + 1;
  return a;
}

// A warp per row, two rows in flight.  Row r: path entry r mod (a + 1) of (layer, K | V) number r / (a + 1).
__global__ void __launch_bounds__(kCommitThreadsAlone)
kv_compact_kernel(const uint4* __restrict__ tree_k, const uint4* __restrict__ tree_v, uint4* __restrict__ k_cache,
                  uint4* __restrict__ v_cache, const CommitParams p) {
  __shared__ CommitTable t;
  const int b = blockIdx.x / p.ctas;
  const int a = commit_table<false>(p, b, t);
  const int lane = threadIdx.x & 31, warps = p.ctas * (blockDim.x >> 5);
  const int rows = 2 * p.layers * (a + 1);           // (a below 0: none)
  for (int r0 = (blockIdx.x % p.ctas) * (blockDim.x >> 5) + (threadIdx.x >> 5); r0 < rows; r0 += 2 * warps) {
    const uint4* src[2];
    uint4* dst[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int r = r0 + k * warps, lk = r / (a + 1), i = r - lk * (a + 1), layer = lk >> 1;
      const int node = r < rows ? t.node[i] : -1;
      src[k] = node < 0 ? nullptr : ((lk & 1) ? tree_v : tree_k) + ((static_cast<int64_t>(layer) * p.batch + b) * p.B + node) * p.row16;
      dst[k] = ((lk & 1) ? v_cache : k_cache) + layer * p.layer_stride16 + t.dst[i];
    }
    for (int e0 = 0; e0 < p.row16; e0 += 128) {
      uint4 x[2][4];
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int e = e0 + j * 32 + lane;
          if (src[k] && e < p.row16) x[k][j] = __ldg(src[k] + e);
        }
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int e = e0 + j * 32 + lane;
          if (src[k] && e < p.row16) dst[k][e] = x[k][j];
        }
    }
  }
}

// In place: row seq_len + path[i] moves to seq_len + i for i = 1 .. accept_len (path[i] >= i; the root stays where it is).
// A unit is (layer, K | V, 32 of the row's 16-byte columns); columns do not meet, so a lane's own order is all that
// counts: it reads kTailHeld rows of a unit into registers before it writes any, and never writes a row that it still has to
// read, because rows are taken in increasing i and path[i] >= i, path increasing.  With few rows a warp holds several
// units at once, if there are more units than warps.
__global__ void __launch_bounds__(kCommitThreadsAlone, 1)
kv_compact_tail_kernel(uint4* k_cache, uint4* v_cache, const CommitParams p) {
  __shared__ CommitTable t;
  const int b = blockIdx.x / p.ctas;
  const int a = commit_table<true>(p, b, t);
  if (a < 1) return;
  const int lane = threadIdx.x & 31, warp = (blockIdx.x % p.ctas) * (blockDim.x >> 5) + (threadIdx.x >> 5), warps = p.ctas * (blockDim.x >> 5);
  const int columns = (p.row16 + 31) / 32, units = 2 * p.layers * columns;
  const int rows = min(a, kTailHeld);                // of a unit that are held at once
  const int per = max(1, min(kTailHeld / rows, (units + warps - 1) / warps));
  for (int first = warp * per; first < units; first += warps * per) {
    const int lk0 = first / columns, column0 = first - lk0 * columns;
    for (int i0 = 1; i0 <= a; i0 += kTailHeld) {     // (one pass unless per is 1)
      auto each = [&](auto&& piece) {
        int lk = lk0, column = column0, i = i0;
#pragma unroll
        for (int k = 0; k < kTailHeld; ++k) {
          if (k >= rows * per || lk >= 2 * p.layers || i > a) break;      // (warp-uniform)
          const int e = column * 32 + lane;
          if (t.node[i] >= 0 && t.node[i] != i && e < p.row16)
            piece(k, ((lk & 1) ? v_cache : k_cache) + (lk >> 1) * p.layer_stride16 + e, i);
          if (++i == i0 + rows && per > 1) {
            i = 1;
            if (++column == columns) { column = 0; ++lk; }
          }
        }
      };
      uint4 held[kTailHeld];
      each([&](int k, uint4* cache, int i) { held[k] = cache[t.src[i]]; });
      each([&](int k, uint4* cache, int i) { cache[t.dst[i]] = held[k]; });
    }
  }
}

// Runs beside the copies: by the time it starts (see commit_table) whatever wrote the two inputs has completed and every
// copying CTA has its length.  The stream's next kernel may be scheduled beside it at once, and, as this one ends behind the
// copies, finds both done when its own wait returns.  (Reads from L2: the kernel that wrote the inputs may have ended after
// this SM last cached the lines.)
__global__ void advance_seq_len_kernel(const int32_t* accept_len, int32_t* seq_len, int batch) {
  ptx::grid_dep_launch();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < batch) seq_len[b] = __ldcg(seq_len + b) + __ldcg(accept_len + b) + 1;
  ptx::grid_dep_wait();
}

// Sequences of at most this many rows get one CTA: 8 layers of 9 positions, 144 rows, 7.4 us that way instead of 4.3.
constexpr int kAloneRows = 64;
// CTAs of kCommitThreads that an SM holds: more rows than their warps cover are taken in turns, not in waves.
constexpr int kCopyResident = 3, kTailResident = 2;

struct CommitPlan {
  int ctas, threads;                                 // per sequence; of a CTA
  int launches() const { return ctas > 1 ? 2 : 1; }
};

// A warp per row of every layer, or, in place, per unit.
CommitPlan commit_plan(int layers, int batch, int row16, int N, bool tail) {
  const int64_t rows = static_cast<int64_t>(2 * layers) * (N + 1);
  if (rows <= kAloneRows) return {1, kCommitThreadsAlone};
  const int64_t work = tail ? static_cast<int64_t>(2 * layers) * ((row16 + 31) / 32) : rows;
  const int64_t fill = (work + kCommitThreads / 32 - 1) / (kCommitThreads / 32);
  const int64_t spread = (tail ? kTailResident : kCopyResident) * sm_count() / batch;
  return {static_cast<int>(fill < spread ? fill : spread > 1 ? spread : 1), kCommitThreads};
}

template <typename Kernel, typename... Args>
jet_status commit_launch(Kernel kernel, bool tail, CommitParams p, cudaStream_t st, Args... args) {
  const CommitPlan plan = commit_plan(p.layers, p.batch, p.row16, p.N, tail);
  p.ctas = plan.ctas;
  launch_dependent(kernel, dim3(static_cast<unsigned>(p.ctas) * p.batch), dim3(plan.threads), st, args..., p);
  if (plan.launches() > 1)
    launch_dependent(advance_seq_len_kernel, dim3((p.batch + 255) / 256), dim3(256), st, p.accept_len, p.seq_len, p.batch);
  return launch_status();
}

}  // namespace
}  // namespace jet

extern "C" int jet_kv_compact_launches(int layers, int batch, int Hkv, int D, int N, int tail) {
  if (layers < 1 || layers > 65535 || batch < 1 || Hkv < 1 || D < 1 || N < 1 || N > JET_MAX_DEPTH) return 0;
  return jet::commit_plan(layers, batch, static_cast<int>(static_cast<int64_t>(Hkv) * D / 8), N, tail != 0).launches();
}

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
                       max_pages_per_seq, page_size, layers, batch, B, row16, N, 1};
  return commit_launch(kv_compact_kernel, false, p, st, static_cast<const uint4*>(tree_k), static_cast<const uint4*>(tree_v),
                       static_cast<uint4*>(k_cache), static_cast<uint4*>(v_cache));
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
                       max_pages_per_seq, page_size, layers, batch, B, row16, N, 1};
  return commit_launch(kv_compact_tail_kernel, true, p, st, static_cast<uint4*>(k_cache), static_cast<uint4*>(v_cache));
}
