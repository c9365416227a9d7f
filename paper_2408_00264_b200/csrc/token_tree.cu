// Token tree from speculated sequences (Sec. 2.1, Fig. 2 caption: several speculations are merged
// by prefix matching into a tree).  One thread block per sequence; the sizes are tiny (at most 128
// candidates of at most 16 tokens), so the kernel is latency bound like the walk.
//
// A node is a distinct non-empty prefix of some candidate; node 0 is the root (the token the target
// emitted last).  Nodes are numbered by depth first, then by the lowest candidate that contains
// the prefix, which makes the numbering unique and topological (parent[i] < i).  Unused slots up
// to node_cap become children of the root with token -1: they never match a target token, so the
// arrays can go into a verify step of fixed size as they are.
#include "clv_internal.cuh"

namespace clv {
namespace {

constexpr int kMaxCand = CLV_TREE_MAX_CAND;   // 128
constexpr int kMaxLen = CLV_TREE_MAX_LEN;     // 16
constexpr int kThreads = 1024;

struct Params {
  int n_cand, max_len, node_cap;
  const int32_t* root_token;
  const int32_t* cand;
  const int32_t* cand_len;
  int32_t* tokens;
  int32_t* parent;
  int32_t* n_nodes;
  int32_t* node_of;
  int32_t* status;
};

// What bounds it is the chain of barriers and shared-memory round trips, so nothing goes depth by depth:
// a warp takes a candidate and compares it with 32 earlier ones at a time over their whole length (one
// per lane; a ballot per depth finds the first that agrees so far, until none does), and nodes are numbered by a
// scan over bit masks of the candidates that start one.  4 x 32 candidates of 6 tokens: 6.9 -> 3.2 us;
// 8 x 128 of 16: 19.1 -> 7.3 us.
__global__ void __launch_bounds__(kThreads) token_tree_kernel(Params p) {
  constexpr int kWords = kMaxCand / 32, kStride = kMaxLen + 1;   // odd: a column of s_cand has no bank conflicts
  static_assert(kThreads / 32 >= kMaxLen, "a warp per depth");
  // rep[d][c]: lowest candidate whose first d+1 tokens equal those of candidate c (-1: c is shorter)
  __shared__ short s_rep[kMaxLen][kMaxCand];
  __shared__ int s_cand[kMaxCand * kStride];          // this sequence's candidates
  __shared__ int s_len[kMaxCand];
  __shared__ unsigned s_new[kMaxLen * kWords];        // bit c: candidate c is the first with its prefix of this depth
  __shared__ int s_before[kMaxLen * kWords];          // nodes in front of those of this word
  __shared__ int s_total;
  const int b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int C = p.n_cand, D = p.max_len;
  cudaGridDependencySynchronize();  // programmatic launch: the previous kernel's results are complete
  cudaTriggerProgrammaticLaunchCompletion();
  const int32_t* cand_g = p.cand + (int64_t)b * C * D;
  const int root = p.root_token[b];
  {
    const int d = tid % kMaxLen;
    if (d < D)
      for (int c = tid / kMaxLen; c < C; c += kThreads / kMaxLen) s_cand[c * kStride + d] = cand_g[c * D + d];
  }
  bool bad = false;
  for (int c = tid; c < C; c += kThreads) {
    const int len = p.cand_len[(int64_t)b * C + c];
    bad |= (len < 0 || len > D);
    s_len[c] = min(max(len, 0), D);
  }
  bad = __syncthreads_or(bad ? 1 : 0) != 0;

  // ---- prefix matching
  for (int c = warp; c < C; c += kThreads / 32) {
    const int len = s_len[c];
    int rep = -1;   // of lane d: rep[d][c]
    for (int o0 = 0; o0 < c; o0 += 32) {
      const int o = min(o0 + lane, C - 1);
      const int most = o0 + lane < c ? min(len, s_len[o]) : 0;   // tokens that can agree
      bool still = true;
#pragma unroll 2
      for (int d = 0; d < D; ++d) {
        still = still && d < most && s_cand[o * kStride + d] == s_cand[c * kStride + d];
        const unsigned agree = __ballot_sync(0xFFFFFFFFu, still);
        if (!agree) break;
        if (lane == d && rep < 0) rep = o0 + __ffs(agree) - 1;
      }
    }
    if (lane < D) s_rep[lane][c] = (short)(lane >= len ? -1 : rep < 0 ? c : rep);
  }
  __syncthreads();

  // ---- number the nodes: depth major, candidate minor
  if (warp < kMaxLen) {
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
      const int c = 32 * k + lane;
      const unsigned m = __ballot_sync(0xFFFFFFFFu, warp < D && c < C && s_rep[warp][c] == c);
      if (lane == 0) s_new[warp * kWords + k] = m;
    }
  }
  __syncthreads();
  if (warp == 0) {
    static_assert(kMaxLen * kWords == 64, "two words per lane");
    const int n0 = __popc(s_new[2 * lane]), n1 = __popc(s_new[2 * lane + 1]);
    int incl = n0 + n1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += up;
    }
    s_before[2 * lane] = 1 + incl - n0 - n1;   // node 0 is the root
    s_before[2 * lane + 1] = 1 + incl - n1;
    if (lane == 31) s_total = 1 + incl;
  }
  __syncthreads();
  const int total = s_total;
  const bool fail = bad || total > p.node_cap;
  auto node_at = [&](int d, int c) {   // of the prefix of depth d that candidate c starts
    const int w = d * kWords + (c >> 5);
    return s_before[w] + __popc(s_new[w] & ((1u << (c & 31)) - 1u));
  };

  int32_t* tokens = p.tokens + (int64_t)b * p.node_cap;
  int32_t* parent = p.parent + (int64_t)b * p.node_cap;
  int32_t* node_of = p.node_of + (int64_t)b * C * D;
  // the root, and padding that hangs off the root with a token nothing matches
  for (int i = tid; i < p.node_cap; i += kThreads)
    if (i == 0 || fail || i >= total) {
      tokens[i] = i == 0 ? root : -1;
      parent[i] = i == 0 ? -1 : 0;
    }
  const int d = tid % kMaxLen;
  if (d < D)
    for (int c = tid / kMaxLen; c < C; c += kThreads / kMaxLen) {
      const int rep = s_rep[d][c];
      int node = -1;
      if (!fail && rep >= 0) {
        node = node_at(d, rep);
        if (rep == c) {  // this candidate introduces the node
          tokens[node] = s_cand[c * kStride + d];
          parent[node] = d == 0 ? 0 : node_at(d - 1, s_rep[d - 1][c]);
        }
      }
      node_of[c * D + d] = node;
    }
  if (tid == 0) {
    p.n_nodes[b] = fail ? 1 : total;
    p.status[b] = fail ? CLV_ERR_TREE : CLV_OK;
  }
}

}  // namespace

cudaError_t launch_token_tree(int batch, int n_cand, int max_len, int node_cap, const int32_t* root_token,
                              const int32_t* cand, const int32_t* cand_len, int32_t* tokens, int32_t* parent,
                              int32_t* n_nodes, int32_t* node_of, int32_t* status, cudaStream_t stream) {
  Params p;
  p.n_cand = n_cand;
  p.max_len = max_len;
  p.node_cap = node_cap;
  p.root_token = root_token;
  p.cand = cand;
  p.cand_len = cand_len;
  p.tokens = tokens;
  p.parent = parent;
  p.n_nodes = n_nodes;
  p.node_of = node_of;
  p.status = status;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)batch, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, token_tree_kernel, p);
}

}  // namespace clv
