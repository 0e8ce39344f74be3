// jet_kv_compact: commit of the accepted path: the K and V rows of every accepted node of every layer are copied behind the
// prefix (contiguous or paged cache), then seq_len advances.  jet_kv_compact_tail: the same in place, for a cache that
// holds the tree's rows behind the prefix.
//
// Bound: latency (a step commits 0.1 - 3 MB).  The chain is lengths and path -> page table -> rows; the rows of all
// sequences are spread over the GPU, a warp per row, and a CTA works the path of its sequence out once.  No CTA may see an
// advanced length, so seq_len is advanced by a second launch, or, where one CTA per sequence is enough (kAloneRows), by that
// CTA: the second launch costs 1.7 us of host time.  It starts once all CTAs hold their lengths and runs beside the copies.  (While it
// waited for them before its load and store, a commit of several layers took 0.2 - 0.4 us more: acceptance and commit of 36 layers, 4
// rows, paged: 8.2 against 7.9 us; 32 sequences, 4 layers: 12.9 against 12.6.)  A step has counts that take its place (finish_commit), and
// with greedy acceptance the copying CTAs select the path themselves (accept_commit_kernel).
// us per call in a captured stream (a cluster of eight CTAs per sequence before; page size 16, 8 heads of 128 and 36 layers
// where not said otherwise; in place in brackets):
//   1 sequence, 6 rows                  5.3 -> 3.5   [8.1 -> 4.8]      1 sequence, 65 rows    28 -> 5.3  [50 -> 17]
//   32 sequences, 6 rows                11.6 -> 9.9  [22.4 -> 15.0]    128, one layer, 5 rows  10.2 -> 3.3 [23.5 -> 4.8]
//   8 sequences, 48 layers, 4 heads     5.3 -> 4.2   [7.4 -> 5.6]      128, 5 rows            39 -> 37  [61 -> 33]
// Left behind the clusters: 33 - 64 rows of 2 KB in one CTA, 0.4 us (two turns of its warps; a second launch costs a caller
// who issues call by call more than that).
#include "commit_rows.cuh"

namespace jet {
namespace {

// Waits for the kernels before this one, fills the table and returns a: entries 0 .. a of the path are committed.  Where a second launch
// advances seq_len it is let go only behind the lengths: it starts when every CTA has got here, so that no CTA can read a
// length that it has advanced.
template <bool kTail>
__device__ __forceinline__ int commit_table(const CommitParams& p, int b, CommitTable& t) {
  const int i = threadIdx.x;
  const bool second = p.ctas != 1 && !p.arrived;
  if (second) ptx::grid_dep_wait();
  else grid_dependency_wait();
  const int accepted = p.accept_len[b], len = p.seq_len[b];
  const int node = i <= p.N ? p.path[static_cast<size_t>(b) * (p.N + 1) + i] : -1;      // (in flight with the lengths)
  const int a = min(accepted, p.N);
  if (i <= a) commit_entry<kTail>(p, b, i, node, len, cache_row(p, b, static_cast<int64_t>(len) + i), t);
  __syncthreads();                                   // (the lengths have arrived: they went into the table and a)
  if (second) ptx::grid_dep_launch();
  finish_commit(p, b, len + accepted + 1);
  return a;
}

__global__ void __launch_bounds__(kCommitThreadsAlone, 1)
kv_compact_kernel(const CommitParams p) {
  __shared__ CommitTable t;
  const int b = blockIdx.x / p.ctas;
  const int a = commit_table<false>(p, b, t);
  copy_rows(p, b, a, t);
}

__global__ void __launch_bounds__(kCommitThreadsAlone, 1)
kv_compact_tail_kernel(const CommitParams p) {
  __shared__ CommitTable t;
  const int b = blockIdx.x / p.ctas;
  const int a = commit_table<true>(p, b, t);
  move_rows(p, a, t);
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

jet_status commit_launch(bool tail, CommitParams p, cudaStream_t st) {
  const CommitPlan plan = commit_plan(p.layers, p.batch, p.row16, p.N, tail);
  p.ctas = plan.ctas;
  launch_dependent(tail ? kv_compact_tail_kernel : kv_compact_kernel, dim3(static_cast<unsigned>(p.ctas) * p.batch), dim3(plan.threads), st, p);
  if (plan.launches() > 1 && !p.arrived)
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
  CommitParams p;
  const jet_status r = commit_params(tree_k, tree_v, k_cache, v_cache, cache_layer_stride, kv_batch_stride, page_table,
                                     max_pages_per_seq, page_size, path, accept_len, seq_len, layers, batch, B, Hkv, D, N, false, &p);
  return r != JET_OK ? r : commit_launch(false, p, static_cast<cudaStream_t>(stream));
}

extern "C" jet_status jet_kv_compact_tail(void* k_cache, void* v_cache, int64_t cache_layer_stride,
                                          int64_t kv_batch_stride, const int32_t* page_table,
                                          int max_pages_per_seq, int page_size, const int32_t* path,
                                          const int32_t* accept_len, int32_t* seq_len, int layers, int batch,
                                          int B, int Hkv, int D, int N, void* stream) {
  using namespace jet;
  CommitParams p;
  const jet_status r = commit_params(nullptr, nullptr, k_cache, v_cache, cache_layer_stride, kv_batch_stride, page_table,
                                     max_pages_per_seq, page_size, path, accept_len, seq_len, layers, batch, B, Hkv, D, N, true, &p);
  return r != JET_OK ? r : commit_launch(true, p, static_cast<cudaStream_t>(stream));
}

// Not part of the C ABI: either of the two with counts (one int per sequence, 0 between calls), which take the place of the second launch.
extern "C" JET_API jet_status jet_internal_kv_compact_step(const void* tree_k, const void* tree_v, void* k_cache, void* v_cache,
                                                           int64_t cache_layer_stride, int64_t kv_batch_stride,
                                                           const int32_t* page_table, int max_pages_per_seq, int page_size,
                                                           const int32_t* path, const int32_t* accept_len, int32_t* seq_len,
                                                           int layers, int batch, int B, int Hkv, int D, int N, int tail,
                                                           int32_t* arrived, void* stream) {
  using namespace jet;
  CommitParams p;
  const jet_status r = commit_params(tree_k, tree_v, k_cache, v_cache, cache_layer_stride, kv_batch_stride, page_table,
                                     max_pages_per_seq, page_size, path, accept_len, seq_len, layers, batch, B, Hkv, D, N, tail != 0, &p);
  if (r != JET_OK) return r;
  p.arrived = arrived;
  return commit_launch(tail != 0, p, static_cast<cudaStream_t>(stream));
}
