// Stochastic acceptance at temperature T > 0 (Sec. 4.1 / 4.2, Table 1 lower half: the paper adopts
// its baseline's tree sampling algorithm and prints no formula; taken here as speculative sampling
// for drafts that are proposed deterministically, one token per child).
//
// At the current node the target's distribution is p = softmax(logits / T).  The children are
// tried in increasing node index: child c with token x is accepted if
//   u[c] < p(x) / (1 - mass of the tokens rejected at this node so far);
// a rejected token is struck from the distribution; when every child is rejected (or there is
// none) the next token is the first v, in vocabulary order and not struck, whose running sum of p
// exceeds u[N] * (what is left).  The uniforms are the caller's.
//
// Two launches.  (1) One pass over all logits (an HBM stream like the argmax): every warp
// reduces a slice of 4096 consecutive logits of a row to (maximum, sum of exponentials relative
// to it) with an online update, in base-2 units.  (2) One block per sequence fetches what any level of
// the walk may need at once (every row's slices, every node's logit in its parent's row) and one
// thread runs the accept chain in shared memory; the final draw locates the slice by a running sum over
// the slices' weights (the weights of struck tokens taken out) and then scans that one slice with
// the whole block, 16 logits per thread.
#include <limits.h>
#include <math.h>

#include "clv_internal.cuh"

namespace clv {
namespace {

constexpr int kThreads = 256;
constexpr int kPiece = 32768;   // logits per block of the statistics pass (64 KB)
// Vectors of a batch of the statistics pass, whose registers let six blocks of it share an SM (eight vectors: three blocks,
// 16 x 64 rows of 128256 59 us instead of 54, or five with a few registers spilled, 55.5; 5 x 27 of 50257 the same).
constexpr int kUnroll = 4;
constexpr int kSlice = kPiece / (kThreads / 32);   // 4096 logits per warp: the unit of the running sums
constexpr int kPerThread = kSlice / kThreads;       // 16: what a thread scans of the chosen slice
static_assert(kSlice == 4096 && kPerThread == 16, "a slice is scanned in one round of the block");

__device__ __forceinline__ uint4 ld_stream16(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// A token's weight beside a maximum m: 2^(x k - m) in one rounding, as the statistics' packed form has it.  Wherever the same
// logit is weighed the number is the same, whatever the compiler makes of a product and a difference: m is rounded to 2^-24
// of itself, so a row's sum by one form and a weight by the other differ by that much of |x k| (T = 0.01 and a logit of 30:
// 1.7e-4 of a token that is certain).
//
// The rounding of m alone is up to 2^-24 |m|, which must not become a weight of its own: a slice of masked logits (-1e30) had
// weights of 2^(+-1e23), and infinity beside a rescale by 0 made the whole row's sum NaN.  From 2^20 on k and m are scaled by the
// power of two that brings m to [2^20, 2^21): an equal logit's weight stays within 2^(+-1/16), and any other bf16 logit, at
// least 2^-8 |m| below, has none either way.
struct Exponent {
  float k, m;
  __device__ __forceinline__ float weight(float x) const { return ex2(fmaf(x, k, -m)); }
};
__device__ __forceinline__ Exponent exponent_of(float k, float m) {
  const uint32_t e = (__float_as_uint(m) >> 23) & 255u;
  if (e < 127u + 20u || e == 255u) return {k, m};   // 255: infinite
  const float scale = __uint_as_float((2u * 127u + 20u - e) << 23);
  return {k * scale, m * scale};
}

// (m, s): s = sum of the weights beside m of the values seen so far, m their maximum (s = 0 while m = -inf)
struct Stat {
  float m, s;
};
__device__ __forceinline__ void stat_merge(Stat& a, const Stat& b) {
  const float m = fmaxf(a.m, b.m), ref = m == -INFINITY ? 0.f : m;
  a.s = a.s * ex2(a.m - ref) + b.s * ex2(b.m - ref);   // 2^(-inf) = 0 for an empty side
  a.m = m;
}
__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t u) { return *reinterpret_cast<__nv_bfloat162*>(&u); }
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  return (unsigned long long)__float_as_uint(y) << 32 | __float_as_uint(x);
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float low(unsigned long long v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float high(unsigned long long v) { return __uint_as_float((uint32_t)(v >> 32)); }

// A batch of kUnroll vectors at once: one maximum and at most one rescale for the 32 values, then
// their exponentials into four running sums (no long chain of dependent additions).  Beside the stream (DRAM 65 %) it is
// the issue slots, 61 % of the active cycles, and the exponentials, two thirds of theirs, that set the pace, so the maximum is taken of packed bf16 (a positive factor does not change which it is, and the
// maximum with -inf drops a NaN, which carries no mass), and products, differences and sums are packed fp32 (statistics and walk of
// 16 x 64 rows of 128256 64.3 -> 59.2 us, of 5 x 27 of 50257 11.8 -> 10.7 with the walk's changes).
__device__ __forceinline__ void stat_take_batch(Stat& st, uint4 (&w)[kUnroll], float k) {
  const __nv_bfloat162 none = as_bf162(0xFF80FF80u);
  __nv_bfloat162 top[2] = {none, none};
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    uint32_t* r = reinterpret_cast<uint32_t*>(&w[u]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const __nv_bfloat162 x = __hmax2(as_bf162(r[j]), none);
      r[j] = *reinterpret_cast<const uint32_t*>(&x);
      top[j & 1] = __hmax2(top[j & 1], x);
    }
  }
  const __nv_bfloat162 t = __hmax2(top[0], top[1]);
  const float mx = fmaxf(__low2float(t), __high2float(t)) * k;
  if (!(mx > -INFINITY)) return;   // nothing but -inf (or NaN): no mass
  if (mx > st.m) { st.s *= ex2(st.m - mx); st.m = mx; }
  const Exponent e = exponent_of(k, st.m);
  const unsigned long long kk = pack2(e.k, e.k), mm = pack2(-e.m, -e.m);
  unsigned long long acc[2] = {0ull, 0ull};
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    const uint32_t r[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned long long x = fma2(pack2(bf16_lo(r[j]), bf16_hi(r[j])), kk, mm);
      acc[j & 1] = add2(acc[j & 1], pack2(ex2(low(x)), ex2(high(x))));
    }
  }
  const unsigned long long sum = add2(acc[0], acc[1]);
  st.s += low(sum) + high(sum);
}

struct StatParams {
  const uint16_t* logits;
  int64_t ld;
  int vocab, pieces, rows;
  int rows_first;    // all rows' first pieces, then all second ones
  float k;           // log2(e) / T
  float2* partial;   // [rows][pieces * 8]: one (maximum, sum) per slice
};

__global__ void __launch_bounds__(kThreads, 6) softmax_stats_kernel(StatParams p) {
  const int row = p.rows_first ? blockIdx.x % p.rows : blockIdx.x / p.pieces;
  const int piece = p.rows_first ? blockIdx.x / p.rows : blockIdx.x - row * p.pieces;
  const int begin = piece * kPiece;
  const int end = min(p.vocab, begin + kPiece);
  const uint16_t* base = p.logits + (int64_t)row * p.ld;
  const int nvec = (end - begin) >> 3;
  const uint4* vp = reinterpret_cast<const uint4*>(base + begin);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();   // all of this grid has its place: the walk may be set up
  // warp w takes the vectors [512 w, 512 (w + 1)) of the piece: 4096 consecutive logits
  Stat st = {-INFINITY, 0.f};
  const int lim = min(nvec, (warp + 1) * (kSlice / 8));
  int i = warp * (kSlice / 8) + lane;
  for (; i < lim; i += kUnroll * 32) {
    // a short batch is filled up with -inf: one vector after the other it cost a round trip each
    // (6 x 109 rows of 16363 logits: 22.5 -> 20.1 us)
    uint4 w[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      w[u] = i + u * 32 < lim ? ld_stream16(vp + i + u * 32) : make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
    stat_take_batch(st, w, p.k);
  }
  {  // ragged end of the row: at most 7 scalars, taken by the warp whose slice holds them
    const int t0 = begin + 8 * nvec + lane;
    if (t0 < end && (t0 - begin) / kSlice == warp) {
      const float x = __uint_as_float((uint32_t)base[t0] << 16), m = x * p.k;
      if (m > -INFINITY) { Stat one = {m, m < INFINITY ? exponent_of(p.k, m).weight(x) : 1.f}; stat_merge(st, one); }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Stat other = {__shfl_xor_sync(0xFFFFFFFFu, st.m, o), __shfl_xor_sync(0xFFFFFFFFu, st.s, o)};
    stat_merge(st, other);
  }
  if (lane == 0) p.partial[((int64_t)row * p.pieces + piece) * (kThreads / 32) + warp] = make_float2(st.m, st.s);
}

struct WalkParams {
  const uint16_t* logits;
  int64_t ld;
  int vocab, pieces, N, path_cap;
  float k;
  const float2* partial;
  const int32_t* parent;
  const int32_t* tokens;
  const float* uniforms;   // [B][N + 1]
  int32_t* accept_len;
  int32_t* accept_idx;
  int32_t* next_token;
  int32_t* status;
};

// Slices that the walk's block keeps: 4 KB.  With room for those of every tree (32 KB) the block found no place beside
// what runs before and behind it: 4 x 109 nodes, 56488 logits, the whole step: 35 -> 43 us.
constexpr int kKept = 512;

constexpr int kMaskWords = CLV_MAX_NODES / 32;
// f(node) for every node of a mask below `end`, in increasing order
template <class F>
__device__ __forceinline__ void for_each_below(const uint32_t (&mask)[kMaskWords], int end, F f) {
#pragma unroll 1
  for (int w = 0; 32 * w < end; ++w) {
    uint32_t bits = mask[w];
    if (end - 32 * w < 32) bits &= (1u << (end - 32 * w)) - 1u;
    for (; bits; bits &= bits - 1u) f(32 * w + __ffs(bits) - 1);
  }
}

// One block per sequence.  What bounds it is the number of dependent round trips to memory, so everything
// that any level of the walk may need is fetched at once: every row's statistics, and every node's
// logit in its parent's row (statistics and walk, 5 sequences of 27 nodes, 50257 logits: 16.8 -> 12.8 us; 6 of 109 nodes:
// 42 -> 20).  The statistics are asked for ahead of the tree, from which the logits' addresses come, and kept for the
// draw (the whole step 35.0 -> 34.7).  Siblings are bits of their parent's mask; every node's test is made by a thread of its
// own ahead of the walk, which is then one load per level (one thread that tested and walked took 1.2 us for 27 nodes, 1.8
// for 109; now 0.3 and 0.4).
__global__ void __launch_bounds__(kThreads) sample_walk_kernel(WalkParams p) {
  __shared__ int st[CLV_MAX_NODES], path[CLV_MAX_NODES];
  __shared__ uint32_t s_kids[CLV_MAX_NODES][kMaskWords];           // a node's children
  __shared__ int s_accepted[CLV_MAX_NODES];                        // the first of them that its test accepts (INT_MAX: none)
  __shared__ float su[CLV_MAX_NODES + 1], se[CLV_MAX_NODES], s_m[CLV_MAX_NODES], s_S[CLV_MAX_NODES];
  __shared__ float s_slice[kThreads], s_before_slice[kThreads];
  __shared__ float2 s_stats[kKept];   // every row's slices, if they are few
  __shared__ float s_before, s_target;
  __shared__ int s_found, s_bad, s_pick, s_lastv, s_len, s_cur;
  static_assert(kThreads >= CLV_MAX_NODES, "a thread per node");
  const int b = blockIdx.x, tid = threadIdx.x, N = p.N;
  const int n_sl = p.pieces * (kPiece / kSlice);   // slices of a row
  const int64_t o = (int64_t)b * N;
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const int lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kThreads / 32, kRows = 4;   // a warp per row, four rows under way
  const bool keep = n_sl <= 32 && N * n_sl <= kKept;
  auto fetch = [&](int r0, float2 (&v)[kRows]) {
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const int r = r0 + u * kWarps;
      v[u] = (r < N && lane < n_sl) ? p.partial[(o + r) * n_sl + lane] : make_float2(-INFINITY, 0.f);
    }
  };
  float2 v[kRows];
  fetch(warp, v);   // under way before the tree, whose tokens the logits below wait for
  if (tid == 0) s_bad = (p.path_cap < 1) ? 1 : 0;
  if (tid < CLV_MAX_NODES) {
    s_accepted[tid] = INT_MAX;
#pragma unroll
    for (int w = 0; w < kMaskWords; ++w) s_kids[tid][w] = 0u;
  }
  __syncthreads();
  const int node = tid;
  int par = -1, tok = -1;
  if (node < N) {
    par = p.parent[o + node];
    tok = p.tokens[o + node];
    st[node] = tok;
    if ((node == 0) ? (par != -1) : (par < 0 || par >= node)) s_bad = 1;   // node 0 is the only root
  }
  for (int i = tid; i <= N; i += kThreads) su[i] = p.uniforms[(int64_t)b * (N + 1) + i];
  const bool child = node > 0 && node < N && par >= 0 && par < node;
  if (child) atomicOr(&s_kids[par][node >> 5], 1u << (node & 31));
  const bool in_vocab = child && tok >= 0 && tok < p.vocab;
  uint32_t logit = 0x7FC00000u;   // NaN: no mass
  if (in_vocab) logit = (uint32_t)p.logits[(o + par) * p.ld + tok] << 16;
  // ---- every row's maximum and sum from its slices
  {
    for (int r0 = warp; r0 < N; r0 += kWarps * kRows) {
      if (r0 != warp) fetch(r0, v);
      Stat a[kRows];
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int r = min(r0 + u * kWarps, N - 1);
        if (keep && r0 + u * kWarps < N && lane < n_sl) s_stats[(r0 + u * kWarps) * n_sl + lane] = v[u];
        a[u] = Stat{-INFINITY, 0.f};
        stat_merge(a[u], Stat{v[u].x, v[u].y});
        for (int i = lane + 32; i < n_sl; i += 32) {
          const float2 w = p.partial[(o + r) * n_sl + i];
          stat_merge(a[u], Stat{w.x, w.y});
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int u = 0; u < kRows; ++u)
          stat_merge(a[u], Stat{__shfl_xor_sync(0xFFFFFFFFu, a[u].m, off), __shfl_xor_sync(0xFFFFFFFFu, a[u].s, off)});
      }
#pragma unroll
      for (int u = 0; u < kRows; ++u)
        if (lane == 0 && r0 + u * kWarps < N) { s_m[r0 + u * kWarps] = a[u].m; s_S[r0 + u * kWarps] = a[u].s; }
    }
  }
  __syncthreads();
  bool bad = s_bad != 0;
  // ---- the weight of every node in its parent's row; a token that an earlier sibling carries was struck with
  //      that sibling and carries nothing
  if (!bad && child) {
    bool repeat = false;
    for_each_below(s_kids[par], node, [&](int d) { repeat |= st[d] == tok; });
    const float x = __uint_as_float(logit), m = s_m[par];
    se[node] = (!repeat && in_vocab && m > -INFINITY && x == x) ? exponent_of(p.k, m).weight(x) : 0.f;
  }
  __syncthreads();
  // ---- every node's test, should the walk come to its parent: what is left of that row when its earlier siblings were
  //      rejected, in node order
  if (!bad && child) {
    float rej = 0.f;
    for_each_below(s_kids[par], node, [&](int d) { rej += se[d]; });
    const float left = s_S[par] - rej;
    const float a = (left > 0.f) ? se[node] / left : 0.f;
    if (su[node] < a) atomicMin(&s_accepted[par], node);
  }
  __syncthreads();
  if (tid == 0) {   // the accept chain
    int len = 1, cur = 0;
    path[0] = 0;
    while (!bad) {
      const int found = s_accepted[cur];
      if (found == INT_MAX) break;
      if (len == p.path_cap || len == CLV_MAX_NODES) { bad = true; break; }
      path[len++] = found;
      cur = found;
    }
    s_len = len;
    s_cur = cur;
    s_bad = bad ? 1 : 0;
  }
  __syncthreads();
  bad = s_bad != 0;
  int len = s_len;
  const int cur = s_cur;
  if (!bad) {
    // ---- draw the next token from what is left of row `cur`: all of its children were rejected,
    //      their tokens are struck.  The slices' weights come from the statistics pass.
    const float m = s_m[cur];
    const uint16_t* row = p.logits + (o + cur) * p.ld;
    // what is left, slice by slice (the first pass's sums minus the struck weights differ from a
    // fresh sum by rounding only); thread 0 walks the slices in vocabulary order
    for (int j = tid; j < n_sl; j += kThreads) {
      const float2 sl = keep ? s_stats[cur * n_sl + j] : p.partial[(o + cur) * n_sl + j];
      float sum = (sl.x > -INFINITY && m > -INFINITY) ? sl.y * ex2(sl.x - m) : 0.f;
      const int v0 = j * kSlice, v1 = min(p.vocab, v0 + kSlice);
      for_each_below(s_kids[cur], N, [&](int c) {
        if (st[c] >= v0 && st[c] < v1) sum -= se[c];   // (a token carried by two siblings is struck once)
      });
      sum = fmaxf(sum, 0.f);
      if (j < kThreads) s_slice[j] = sum;
    }
    __syncthreads();
    if (warp == 0) {
      // the running sums in vocabulary order (one thread: the sums of all slices in this order are what is drawn from),
      // then every lane looks at slices of its own for the one that the target falls into
      float total = 0.f;
      if (lane == 0) {
#pragma unroll 8
        for (int j = 0; j < n_sl; ++j) {   // at most one slice per thread: larger vocabularies are refused by the host
          s_before_slice[j] = total;
          total += s_slice[j];
        }
      }
      __syncwarp();
      total = __shfl_sync(0xFFFFFFFFu, total, 0);
      const float target = su[N] * total;
      int pick = INT_MAX, last = -1;
      for (int j = lane; j < n_sl; j += 32) {
        const float here = s_slice[j];
        if (here > 0.f) {
          last = j;
          if (pick == INT_MAX && s_before_slice[j] + here > target) pick = j;
        }
      }
      pick = __reduce_min_sync(0xFFFFFFFFu, pick);
      last = __reduce_max_sync(0xFFFFFFFFu, last);
      if (lane == 0) {
        if (pick != INT_MAX) {
          s_before = s_before_slice[pick];
        } else {
          pick = last;   // rounding: the target lies at the very end (-1: a row without any mass)
          if (last >= 0) s_before = total - s_slice[last];
        }
        s_pick = pick;
        s_target = target;
        s_found = INT_MAX;   // first element of the slice whose running sum exceeds the target
        s_lastv = -1;        // last element of the slice that carries any weight
      }
    }
    __syncthreads();
    const int pick = s_pick;
    if (pick >= 0) {
      // ---- the whole block scans the chosen slice in one round: a thread takes 16 consecutive
      //      logits (two 16-byte reads), strikes the children's tokens among them, adds them up;
      //      a running sum across the block (warp scan + the warps' totals) gives every thread
      //      its start, and the first element whose running sum exceeds the target wins
      const float target = s_target;
      const int q0 = pick * kSlice, q1 = min(p.vocab, q0 + kSlice);
      const int v_base = q0 + tid * kPerThread;
      float e[kPerThread];
      {
        uint4 w[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)   // past the row's end: the last vector again (cut by index below)
          w[h] = ld_stream16(row + min(v_base + 8 * h, (q1 - 1) & ~7));
        const Exponent ex = exponent_of(p.k, m);   // (once: 16 times it took 0.4 us)
        uint32_t struck = 0;
        for_each_below(s_kids[cur], N, [&](int c) {
          if (st[c] >= v_base && st[c] < v_base + kPerThread) struck |= 1u << (st[c] - v_base);
        });
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float x[8] = {bf16_lo(w[h].x), bf16_hi(w[h].x), bf16_lo(w[h].y), bf16_hi(w[h].y),
                              bf16_lo(w[h].z), bf16_hi(w[h].z), bf16_lo(w[h].w), bf16_hi(w[h].w)};
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const bool in = (v_base + 8 * h + j < q1) && !((struck >> (8 * h + j)) & 1u) && x[j] == x[j] && m > -INFINITY;
            e[8 * h + j] = in ? ex.weight(x[j]) : 0.f;
          }
        }
      }
      float mine = 0.f;
#pragma unroll
      for (int j = 0; j < kPerThread; ++j) mine += e[j];
      float incl = mine;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const float up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += up;
      }
      if (lane == 31) s_slice[warp] = incl;
      __syncthreads();
      float run = s_before + (incl - mine);   // the running sum before this thread's first element
      for (int w = 0; w < warp; ++w) run += s_slice[w];
      int first = INT_MAX, lastv = -1;
#pragma unroll
      for (int j = 0; j < kPerThread; ++j) {
        run += e[j];
        if (e[j] > 0.f) {
          lastv = v_base + j;
          if (first == INT_MAX && run > target) first = v_base + j;
        }
      }
      if (lastv >= 0) atomicMax(&s_lastv, lastv);
      if (first != INT_MAX) atomicMin(&s_found, first);
      __syncthreads();
      if (tid == 0) p.next_token[b] = (s_found != INT_MAX) ? s_found : s_lastv;
    } else if (tid == 0) {
      p.next_token[b] = -1;   // a row without any mass
    }
  }
  __syncthreads();
  if (bad) len = 0;
  for (int j = tid; j < p.path_cap; j += kThreads)
    p.accept_idx[(int64_t)b * p.path_cap + j] = (j < len) ? path[j] : -1;
  if (tid == 0) {
    p.accept_len[b] = len;
    if (bad) p.next_token[b] = -1;
    p.status[b] = bad ? CLV_ERR_TREE : CLV_OK;
  }
}

int sample_pieces(int vocab) { return (vocab + kPiece - 1) / kPiece; }

}  // namespace

int sample_max_vocab() { return kThreads * kSlice; }   // one slice per thread of the walk's block

size_t sample_scratch_bytes(int rows, int vocab) {
  return sizeof(float2) * (size_t)rows * sample_pieces(vocab) * (kPiece / kSlice);
}

cudaError_t launch_accept_sample(const clv_shape& s, const void* logits, int64_t ld, const int32_t* parent,
                                 const int32_t* tokens, const float* uniforms, float temperature,
                                 int32_t* accept_len, int32_t* accept_idx, int32_t* next_token, int32_t* status,
                                 void* scratch, cudaStream_t stream) {
  const int rows = s.batch * s.n_nodes;
  const float k = 1.4426950408889634f / temperature;
  StatParams a;
  a.logits = static_cast<const uint16_t*>(logits);
  a.ld = ld;
  a.vocab = s.vocab;
  a.pieces = sample_pieces(s.vocab);
  a.rows = rows;
  // A row's last piece may be short.  If the pieces' number is even, as the SMs' is, blocks in the rows' order give the short
  // ones to the same SMs time and again (7 x 120 rows of 33000 27.8 us, by pieces 23.4; 4 x 110 of 33000 22.9, 20.1, of 50257
  // 25.1, 23.7; 1 x 128 of 100000 18.7, 17.8).  Otherwise rows stay together (16 x 64 of 128256 53.2, by pieces 53.6; 10 x 90 of
  // 70000 36.8, 37.5), and so they do where an SM has up to three blocks (5 x 36 of 50257 14.1, 14.6).
  const int last_piece = s.vocab - (a.pieces - 1) * kPiece;
  a.rows_first = a.pieces % 2 == 0 && 4 * last_piece < 3 * kPiece && (int64_t)rows * a.pieces > 3 * sm_count();
  a.k = k;
  a.partial = static_cast<float2*>(scratch);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((int64_t)rows * a.pieces), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  // (up to eight blocks per SM, of which registers let six run: the others do better behind an even share all the same, 7 x 128
  // rows of 32000 24.1 us instead of 27.9, 4 x 64 of 128256 22.8 instead of 23.6)
  cfg.dynamicSmemBytes = even_share_smem((int64_t)rows * a.pieces, 2048 / kThreads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  static OncePerDevice once;
  cudaError_t e = run_once_per_device(once, [] {
    return cudaFuncSetAttribute(softmax_stats_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  });
  if (e != cudaSuccess) return e;
  e = cudaLaunchKernelEx(&cfg, softmax_stats_kernel, a);
  if (e != cudaSuccess) return e;
  WalkParams w;
  w.logits = a.logits;
  w.ld = ld;
  w.vocab = s.vocab;
  w.pieces = a.pieces;
  w.N = s.n_nodes;
  w.path_cap = s.path_cap;
  w.k = k;
  w.partial = a.partial;
  w.parent = parent;
  w.tokens = tokens;
  w.uniforms = uniforms;
  w.accept_len = accept_len;
  w.accept_idx = accept_idx;
  w.next_token = next_token;
  w.status = status;
  cfg.gridDim = dim3((unsigned)s.batch, 1, 1);
  cfg.dynamicSmemBytes = 0;
  return cudaLaunchKernelEx(&cfg, sample_walk_kernel, w);
}

}  // namespace clv
