// Greedy acceptance walk (Sec. 2.1 verification phase) and KV commit (equivalence requirement of
// Sec. 2.1).  Both are latency-bound: one warp per sequence for the walk; the row copies of a sequence
// are spread over a thread-block cluster, so that a row of many heads is a few loads per thread (walk and
// commit of one sequence, 32 heads, 64 nodes: 6.4 us by one block, 3.7 by eight; then the nodes fetched at once,
// every node's accepted child found ahead of the walk and the pages fetched meanwhile: verify steps of 1 x 64 nodes 23.4 ->
// 22.6 us, of 4 x 64 with grouped heads 44.0 -> 43.0, of 1 x 16 14.7 -> 14.4).
#include <limits.h>

#include "clv_internal.cuh"

namespace clv {
namespace {

// ------------------------------------------------------------------------------------ walk
struct WalkSmem {
  int ids[CLV_MAX_NODES], next[CLV_MAX_NODES], path[CLV_MAX_NODES];
};
constexpr int kPerLane = CLV_MAX_NODES / 32;   // nodes of a lane

// The walk of sequence b by one warp; returns the accepted length (0 if the tree is malformed).
// The path is left in sm.path[0 .. len) for the caller (visible after a __syncwarp / barrier).
__device__ __forceinline__ int walk_sequence(WalkSmem& sm, int b, int lane, int N, int path_cap,
                                             const int32_t* parent, const int32_t* tokens,
                                             const int32_t* ids, int32_t* accept_len, int32_t* accept_idx,
                                             int32_t* next_token, int32_t* status, bool write) {
  const int64_t o = (int64_t)b * N;
  // Everything the walk needs is asked for at once: one load behind the other's store to shared memory cost a
  // round trip for every 32 nodes.
  int p[kPerLane], token[kPerLane], id[kPerLane];
#pragma unroll
  for (int k = 0; k < kPerLane; ++k) {
    const int i = lane + 32 * k;
    p[k] = i < N ? parent[o + i] : -1;
    token[k] = i < N ? tokens[o + i] : 0;
    id[k] = i < N ? ids[o + i] : 0;
  }
  bool bad = false;
#pragma unroll
  for (int k = 0; k < kPerLane; ++k) {
    const int i = lane + 32 * k;
    sm.ids[i] = id[k];
    sm.next[i] = INT_MAX;
    bad |= i < N && (i == 0 ? p[k] != -1 : p[k] < 0 || p[k] >= i);   // node 0 is the only root
  }
  bad = __any_sync(0xFFFFFFFFu, bad) || path_cap < 1;
  __syncwarp();
  // Every node's accepted child, the lowest that carries the target's choice there; the walk then is a load
  // per step (a search among the nodes at each step: five dependent instructions and a reduction).
  if (!bad) {
#pragma unroll
    for (int k = 0; k < kPerLane; ++k) {
      const int i = lane + 32 * k;
      if (i > 0 && i < N && token[k] == sm.ids[p[k]]) atomicMin(&sm.next[p[k]], i);
    }
  }
  __syncwarp();
  int len = 0, cur = 0;
  if (!bad) {
    if (lane == 0) sm.path[0] = 0;
    len = 1;
    for (int child = sm.next[0]; child != INT_MAX; child = sm.next[cur]) {   // a child's number is higher than its parent's
      if (len == path_cap || len == CLV_MAX_NODES) { bad = true; break; }
      if (lane == 0) sm.path[len] = child;
      ++len;
      cur = child;
    }
  }
  __syncwarp();
  if (bad) len = 0;
  if (!write) return len;
  for (int j = lane; j < path_cap; j += 32)
    accept_idx[(int64_t)b * path_cap + j] = (j < len) ? sm.path[j] : -1;
  if (lane == 0) {
    accept_len[b] = len;
    next_token[b] = bad ? -1 : sm.ids[cur];
    status[b] = bad ? CLV_ERR_TREE : CLV_OK;
  }
  return len;
}

__global__ void __launch_bounds__(32) walk_kernel(int N, int path_cap, const int32_t* parent,
                                                  const int32_t* tokens, const int32_t* ids,
                                                  int32_t* accept_len, int32_t* accept_idx,
                                                  int32_t* next_token, int32_t* status) {
  __shared__ WalkSmem sm;
  // Launched with programmatic stream serialisation: this grid may be set up while the previous
  // kernel of the stream is still draining, so wait for that kernel's results here, and let the
  // next kernel (the commit) start its own set-up right away.
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  walk_sequence(sm, blockIdx.x, threadIdx.x, N, path_cap, parent, tokens, ids, accept_len, accept_idx,
                next_token, status, true);
}

// ------------------------------------------------------------------------------------ commit
struct CommitParams {
  uint4* kc;
  uint4* vc;
  const uint4* k_tree;
  const uint4* v_tree;
  const int32_t* block_table;
  const int32_t* accept_idx;
  const int32_t* accept_len;
  const int32_t* ctx_len;
  int32_t* ctx_len_out;
  int32_t* status;
  int N, path_cap, paged, cap_tokens, n_pages, max_pages;
  int row_vec;  // 16-byte vectors per token row: Hkv * 128 * 2 / 16
};

constexpr int kPages = (CLV_MAX_NODES + CLV_PAGE_SIZE - 1) / CLV_PAGE_SIZE + 1;   // that a path may touch
struct CommitSmem {
  int pages[kPages];    // the block table's entries from the one that holds position L on
  int src[CLV_MAX_NODES];
  long long dst[CLV_MAX_NODES];  // destination token row (global row index)
  int L, len, ok;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// The pages that the rows behind position L go to, by a warp that has nothing else to do while the path is
// walked (paged caches: a round trip less before the copies).
__device__ __forceinline__ void fetch_pages(CommitSmem& sm, const CommitParams& p, int b, int lane) {
  if (!p.paged || lane >= kPages) return;
  const int L = p.ctx_len[b];
  const long long lp = (long long)(L / CLV_PAGE_SIZE) + lane;
  sm.pages[lane] = L >= 0 && lp < p.max_pages ? p.block_table[(int64_t)b * p.max_pages + lp] : -1;
}

// The commit of sequence b by `ranks` thread blocks, of which this is number `rank`.  path: the accepted
// nodes, sm.len of them (sm.len and sm.L are set by thread 0 of the caller).  kCluster: the blocks are a
// cluster; ctx_len_out may be ctx_len, so it is written when every block has read it.
template <bool kCluster, bool kWalked>
__device__ __forceinline__ void commit_sequence(CommitSmem& sm, const CommitParams& p, int b, int tid, const int32_t* path,
                                                int rank, int ranks) {
  // a path in memory is asked for beside its length and the context's, an entry per thread (the commit of 5 sequences
  // alone: 2.35 -> 2.15 us)
  const int entry = !kWalked && tid < min(p.path_cap, CLV_MAX_NODES) ? path[tid] : 0;
  __syncthreads();   // sm.L, sm.len (and the path and sm.pages, if this block walked it)
  if (kCluster) cluster_arrive();
  const int L = sm.L, len = sm.len;
  if (tid == 0) sm.ok = (L >= 0 && len >= 0 && len <= p.path_cap && len <= CLV_MAX_NODES) ? 1 : 0;
  __syncthreads();
  if (sm.ok) {
    for (int j = tid; j < len; j += blockDim.x) {
      const int a = kWalked ? path[j] : entry;   // (len <= 128 < the block's threads: j is tid)
      const long long t = (long long)L + j;
      long long row = -1;
      if (p.paged) {
        const long long lp = t / CLV_PAGE_SIZE;
        const int pg = kWalked ? sm.pages[lp - L / CLV_PAGE_SIZE]
                       : lp < p.max_pages ? p.block_table[(int64_t)b * p.max_pages + lp] : -1;
        if (pg >= 0 && pg < p.n_pages) row = (long long)pg * CLV_PAGE_SIZE + t % CLV_PAGE_SIZE;
      } else if (t < p.cap_tokens) {
        row = (long long)b * p.cap_tokens + t;
      }
      if (a < 0 || a >= p.N || row < 0) sm.ok = 0;  // benign race: every writer stores 0
      sm.src[j] = a;
      sm.dst[j] = row;
    }
  }
  __syncthreads();
  const bool ok = sm.ok != 0;
  if (ok) {
    const int per_row = 2 * p.row_vec;  // K then V
    const int total = len * per_row, step = (int)blockDim.x * ranks;
    auto addr = [&](int w, const uint4*& src, uint4*& dst) {
      const int j = w / per_row, r = w - j * per_row;
      const bool is_k = r < p.row_vec;
      const int c = is_k ? r : r - p.row_vec;
      src = (is_k ? p.k_tree : p.v_tree) + ((int64_t)b * p.N + sm.src[j]) * p.row_vec + c;
      dst = (is_k ? p.kc : p.vc) + sm.dst[j] * p.row_vec + c;
    };
    for (int w0 = rank * (int)blockDim.x + tid; w0 < total; w0 += 4 * step) {   // four 16-byte copies in flight
      uint4 v[4];
      uint4* dst[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (w0 + u * step >= total) continue;
        const uint4* src;
        addr(w0 + u * step, src, dst[u]);
        v[u] = *src;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (w0 + u * step < total) *dst[u] = v[u];
    }
  }
  __syncwarp();
  if (kCluster) cluster_wait();
  if (tid == 0 && rank == 0) {
    p.ctx_len_out[b] = ok ? L + len : L;
    p.status[b] = ok ? CLV_OK : CLV_ERR_TREE;
  }
}

// grid: sequence-major, `ranks` blocks (a cluster) per sequence
__global__ void __launch_bounds__(256) commit_kernel(CommitParams p, int ranks) {
  __shared__ CommitSmem sm;
  const int b = blockIdx.x / ranks, rank = blockIdx.x - b * ranks;
  cudaGridDependencySynchronize();  // programmatic launch: the walk's outputs are complete after this
  cudaTriggerProgrammaticLaunchCompletion();  // a following kernel may set up; it waits for this grid itself
  if (threadIdx.x == 0) { sm.L = p.ctx_len[b]; sm.len = p.accept_len[b]; }
  commit_sequence<true, false>(sm, p, b, threadIdx.x, p.accept_idx + (int64_t)b * p.path_cap, rank, ranks);
}

// Walk and commit of a sequence in one launch: warp 0 of every block walks (the first block's writes
// the results), then the blocks copy the rows together.
struct WalkArgs {
  int N, path_cap;
  const int32_t* parent;
  const int32_t* tokens;
  const int32_t* ids;
  int32_t* accept_len;
  int32_t* accept_idx;
  int32_t* next_token;
  int32_t* status;
};
__global__ void __launch_bounds__(256) walk_commit_kernel(WalkArgs w, CommitParams p, int ranks) {
  __shared__ WalkSmem wsm;
  __shared__ CommitSmem csm;
  const int b = blockIdx.x / ranks, rank = blockIdx.x - b * ranks;
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  if (threadIdx.x < 32) {
    const int L = threadIdx.x == 0 ? p.ctx_len[b] : 0;   // on its way during the walk
    const int len = walk_sequence(wsm, b, threadIdx.x, w.N, w.path_cap, w.parent, w.tokens, w.ids, w.accept_len,
                                  w.accept_idx, w.next_token, w.status, rank == 0);
    if (threadIdx.x == 0) { csm.L = L; csm.len = len; }
    __syncwarp();
  } else if (threadIdx.x < 64) {
    fetch_pages(csm, p, b, threadIdx.x - 32);
  }
  commit_sequence<true, true>(csm, p, b, threadIdx.x, wsm.path, rank, ranks);
}

// The commit of every layer of a model in one launch: blocks (b, layer, *) copy the accepted rows of
// sequence b in that layer's tree buffers into that layer's cache.  All layers share the accepted
// path, the context lengths (ctx_len_out is another array here) and (paged) the block table, so every
// block of a sequence reaches the same verdict; each layer's first one writes it.
__global__ void __launch_bounds__(256) commit_layers_kernel(CommitParams p, long long cache_stride_vec,
                                                            long long tree_stride_vec) {
  __shared__ CommitSmem sm;
  const int b = blockIdx.x;
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const long long layer = blockIdx.y;
  p.kc += layer * cache_stride_vec;
  p.vc += layer * cache_stride_vec;
  p.k_tree += layer * tree_stride_vec;
  p.v_tree += layer * tree_stride_vec;
  if (threadIdx.x == 0) { sm.L = p.ctx_len[b]; sm.len = p.accept_len[b]; }
  commit_sequence<false, false>(sm, p, b, threadIdx.x, p.accept_idx + (int64_t)b * p.path_cap, blockIdx.z, gridDim.z);
}

}  // namespace

cudaError_t launch_walk(const clv_shape& s, const int32_t* parent, const int32_t* tokens,
                        const int32_t* ids, int32_t* accept_len, int32_t* accept_idx,
                        int32_t* next_token, int32_t* status, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)s.batch, 1, 1);
  cfg.blockDim = dim3(32, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, walk_kernel, (int)s.n_nodes, (int)s.path_cap, parent, tokens, ids, accept_len,
                            accept_idx, next_token, status);
}

namespace {
// Blocks that share a sequence's rows: enough to cover the machine, up to the portable cluster size, and
// not more than leaves each thread a 16-byte copy of a path of four nodes (with 4 heads a second block only
// cost: 2.2 -> 2.5 us).
int commit_ranks(const clv_shape& s, int64_t groups) {
  int ranks = 1;
  while (ranks < 8 && groups * ranks * 2 <= sm_count() && ranks * 2 * 256 <= 4 * 2 * s.n_kv_heads * CLV_HEAD_DIM * 2 / 16) ranks *= 2;
  return ranks;
}

template <class K, class... A>
cudaError_t launch_clusters(K kernel, int batch, int ranks, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(batch * ranks), 1, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ranks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, args..., ranks);
}

CommitParams commit_params(const clv_shape& s, const clv_kv_cache& c, const void* k_tree, const void* v_tree,
                           const int32_t* accept_idx, const int32_t* accept_len, const int32_t* ctx_len,
                           int32_t* ctx_len_out, int32_t* status) {
  CommitParams p;
  p.kc = static_cast<uint4*>(c.k);
  p.vc = static_cast<uint4*>(c.v);
  p.k_tree = static_cast<const uint4*>(k_tree);
  p.v_tree = static_cast<const uint4*>(v_tree);
  p.block_table = c.block_table;
  p.accept_idx = accept_idx;
  p.accept_len = accept_len;
  p.ctx_len = ctx_len;
  p.ctx_len_out = ctx_len_out;
  p.status = status;
  p.N = s.n_nodes;
  p.path_cap = s.path_cap;
  p.paged = c.paged;
  p.cap_tokens = c.cap_tokens;
  p.n_pages = c.n_pages;
  p.max_pages = c.max_pages_per_seq;
  p.row_vec = s.n_kv_heads * CLV_HEAD_DIM * 2 / 16;
  return p;
}
}  // namespace

cudaError_t launch_commit(const clv_shape& s, const clv_kv_cache& c, const void* k_tree,
                          const void* v_tree, const int32_t* accept_idx, const int32_t* accept_len,
                          const int32_t* ctx_len, int32_t* ctx_len_out, int32_t* status,
                          cudaStream_t stream) {
  const CommitParams p = commit_params(s, c, k_tree, v_tree, accept_idx, accept_len, ctx_len, ctx_len_out, status);
  return launch_clusters(commit_kernel, s.batch, commit_ranks(s, s.batch), stream, p);
}

cudaError_t launch_walk_commit(const clv_shape& s, const clv_kv_cache& c, const int32_t* parent,
                               const int32_t* tokens, const int32_t* ids, const void* k_tree,
                               const void* v_tree, const int32_t* ctx_len, int32_t* accept_len,
                               int32_t* accept_idx, int32_t* next_token, int32_t* ctx_len_out,
                               int32_t* walk_status, int32_t* commit_status, cudaStream_t stream) {
  const CommitParams p =
      commit_params(s, c, k_tree, v_tree, accept_idx, accept_len, ctx_len, ctx_len_out, commit_status);
  WalkArgs w;
  w.N = s.n_nodes;
  w.path_cap = s.path_cap;
  w.parent = parent;
  w.tokens = tokens;
  w.ids = ids;
  w.accept_len = accept_len;
  w.accept_idx = accept_idx;
  w.next_token = next_token;
  w.status = walk_status;
  return launch_clusters(walk_commit_kernel, s.batch, commit_ranks(s, s.batch), stream, w, p);
}

cudaError_t launch_commit_layers(const clv_shape& s, const clv_kv_cache& c, int n_layers, int64_t cache_layer_stride,
                                 const void* k_tree, const void* v_tree, int64_t tree_layer_stride,
                                 const int32_t* accept_idx, const int32_t* accept_len, const int32_t* ctx_len,
                                 int32_t* ctx_len_out, int32_t* status, cudaStream_t stream) {
  const CommitParams p = commit_params(s, c, k_tree, v_tree, accept_idx, accept_len, ctx_len, ctx_len_out, status);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)s.batch, (unsigned)n_layers, (unsigned)commit_ranks(s, (int64_t)s.batch * n_layers));
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, commit_layers_kernel, p, (long long)(cache_layer_stride / 8),
                            (long long)(tree_layer_stride / 8));
}

}  // namespace clv
