// One step of a Clover-2 draft head (Sec. 3.1; App. A.3 prints the Attention Decoder) for a few
// rows (one per sequence and candidate):
//   Attention Decoder:  x = RMSNorm(h; norm1);  q = x Wq^T + bq;  k = e Wk^T + bk;  v = e Wv^T + bv;
//     per head j: gate_j = <q_j, k_j> / max(|q_j| |k_j|, 1e-8);  a = h + v * gate   (no activation)
//   output projector:   p = [a, e] Wfc^T + bfc        (fully connected, over a and the token embedding)
//   proposals:          logits = RMSNorm(p; norm2) lm_head^T;  the k largest per row
// h = hidden state (of the target, or of the previous head), e = embedding of the last token.
// The five products run on the tensor cores (the row-block GEMM of the LM head kernel with its
// accumulators written out, fp32): with a handful of rows they stream their weights once, which
// is what bounds the step (1.22 GB at hidden 4096, vocabulary 128256).  The operands of a product
// are bf16 (x, a, e, RMSNorm(p) are rounded once, like the activations of a bf16 model); sums,
// gates and logits stay fp32.  The small kernels here do the rest: one block per row.
#include <limits.h>
#include <math.h>

#include "clv_internal.cuh"

namespace clv {
namespace {

constexpr int kThreads = 256;       // gate and top-k kernels
constexpr int kNormThreads = 512;
constexpr int kNormCache = 4;       // groups of 4 elements a thread keeps between the two passes

__device__ __forceinline__ uint32_t f2bf(float x) {
  const __nv_bfloat16 v = __float2bfloat16_rn(x);
  return (uint32_t)*reinterpret_cast<const uint16_t*>(&v);
}
__device__ __forceinline__ float4 bf16x4(uint2 b) {
  return make_float4(__uint_as_float(b.x << 16), __uint_as_float(b.x & 0xFFFF0000u), __uint_as_float(b.y << 16),
                     __uint_as_float(b.y & 0xFFFF0000u));
}
__device__ __forceinline__ uint2 to_bf16x4(float4 v) {
  return make_uint2(f2bf(v.x) | (f2bf(v.y) << 16), f2bf(v.z) | (f2bf(v.w) << 16));
}
// four elements of a bias, which may start anywhere
__device__ __forceinline__ uint2 load_bias4(const uint16_t* b, int i) {
  if ((reinterpret_cast<uintptr_t>(b) & 7u) == 0) return *reinterpret_cast<const uint2*>(b + i);
  return make_uint2(b[i] | ((uint32_t)b[i + 1] << 16), b[i + 2] | ((uint32_t)b[i + 3] << 16));
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// four neighbouring elements of a product whose K axis was cut in `parts` parts (up to 8): the
// parts added up in their order
struct Parts4 {
  float4 p[8];
};
__device__ __forceinline__ void load_parts4(Parts4& t, const float* x, int64_t i, int parts, int64_t stride) {
#pragma unroll
  for (int s = 0; s < 8; ++s)
    if (s < parts) t.p[s] = *reinterpret_cast<const float4*>(x + i + s * stride);
}
__device__ __forceinline__ float4 sum_parts4(const Parts4& t, int parts) {
  float4 v = t.p[0];
#pragma unroll
  for (int s = 1; s < 8; ++s)
    if (s < parts) v = add4(v, t.p[s]);
  return v;
}

// The kernels of a step are chained by programmatic launches: each lets its successor in at once, so
// that it finds its blocks in place and its weights on their way, and waits for its predecessor's
// results itself.  Only the step's first launch waits before it lets the next one in: from then on
// everything before the step is complete, and inputs of the step that no launch of it writes (weights,
// gains, biases, h, e) may be read without waiting.

// y = RMSNorm(x; gain) rounded to bf16.  kFirst: x is the step's input, bf16.  Otherwise a product in
// fp32 `parts` (+ bias); x itself is also written, rounded to bf16 (the head's hidden state, handed to
// the next head).  Bound by the latency of its loads: those that need not wait go ahead.
// One block per row; a thread keeps its first 16 elements in registers between the two passes
// (hidden sizes up to 8192 are read once), later ones are read again.  status: of the n_status products
// that follow, which write a word only when a wait runs out.
template <bool kFirst>
__global__ void __launch_bounds__(kNormThreads) rmsnorm_rows_kernel(int H, const uint16_t* x16, const float* x32,
                                                                    int parts, int64_t stride, const uint16_t* bias,
                                                                    const uint16_t* gain, float eps, uint16_t* y,
                                                                    uint16_t* x_out, int32_t* status, int n_status) {
  __shared__ float s_red[kNormThreads / 32];
  const int r = blockIdx.x, tid = threadIdx.x, n4 = H / 4;
  const int64_t row = (int64_t)r * H;
  if (!kFirst) cudaTriggerProgrammaticLaunchCompletion();
  else cudaGridDependencySynchronize();
  uint2 g[kNormCache], bs[kNormCache];
#pragma unroll
  for (int j = 0; j < kNormCache; ++j) {
    const int i = tid + j * kNormThreads;
    if (i >= n4) continue;
    g[j] = *reinterpret_cast<const uint2*>(gain + 4 * (int64_t)i);
    bs[j] = kFirst ? *reinterpret_cast<const uint2*>(x16 + row + 4 * (int64_t)i) : load_bias4(bias, 4 * i);
  }
  if (kFirst) cudaTriggerProgrammaticLaunchCompletion();
  else cudaGridDependencySynchronize();
  if (r == 0 && tid < n_status) status[tid] = CLV_OK;
  auto load = [&](int i) {
    if (kFirst) return bf16x4(*reinterpret_cast<const uint2*>(x16 + row + 4 * (int64_t)i));
    Parts4 t;
    load_parts4(t, x32, row + 4 * (int64_t)i, parts, stride);
    return add4(sum_parts4(t, parts), bf16x4(load_bias4(bias, 4 * i)));
  };
  float4 c[kNormCache];
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < kNormCache; ++j) {
    const int i = tid + j * kNormThreads;
    if (i >= n4) continue;
    c[j] = bf16x4(bs[j]);
    if (!kFirst) {
      Parts4 t;
      load_parts4(t, x32, row + 4 * (int64_t)i, parts, stride);
      c[j] = add4(sum_parts4(t, parts), c[j]);
    }
    ss += c[j].x * c[j].x + c[j].y * c[j].y + c[j].z * c[j].z + c[j].w * c[j].w;
  }
  for (int i = tid + kNormCache * kNormThreads; i < n4; i += kNormThreads) {
    const float4 v = load(i);
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
  if ((tid & 31) == 0) s_red[tid >> 5] = ss;
  __syncthreads();
  float total = 0.f;
#pragma unroll
  for (int w = 0; w < kNormThreads / 32; ++w) total += s_red[w];
  const float inv = rsqrtf(total / (float)H + eps);
  auto emit = [&](int i, float4 v, float4 gn) {
    *reinterpret_cast<uint2*>(y + row + 4 * (int64_t)i) =
        to_bf16x4(make_float4(v.x * inv * gn.x, v.y * inv * gn.y, v.z * inv * gn.z, v.w * inv * gn.w));
    if (!kFirst) *reinterpret_cast<uint2*>(x_out + row + 4 * (int64_t)i) = to_bf16x4(v);
  };
#pragma unroll
  for (int j = 0; j < kNormCache; ++j) {
    const int i = tid + j * kNormThreads;
    if (i < n4) emit(i, c[j], bf16x4(g[j]));
  }
  for (int i = tid + kNormCache * kNormThreads; i < n4; i += kNormThreads)
    emit(i, load(i), bf16x4(*reinterpret_cast<const uint2*>(gain + 4 * (int64_t)i)));
}

struct GateArgs {
  int H, n_heads, parts;
  int64_t stride;
  const float* prod[3];       // q, k, v in parts
  const uint16_t* bias[3];
  const uint16_t* h;
  const uint16_t* e;
  uint16_t* cat;
  int32_t* status;            // of the product that follows
};

// a = h + v * gate (per head: cosine of q and k), written with e behind it: cat[r] = [a, e] (bf16).
// One warp per head, eight heads per block; q, k, v arrive in `parts` parts without their bias; a lane
// takes four neighbouring elements at a time (the head size is a multiple of 4), the first four from
// registers (a head of 128 elements is read once).
__global__ void __launch_bounds__(kThreads) gate_residual_kernel(const GateArgs a) {
  const int r = blockIdx.x, hd = a.H / a.n_heads;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j = blockIdx.y * (kThreads / 32) + warp;
  const int i0 = 4 * lane;
  cudaTriggerProgrammaticLaunchCompletion();
  const bool have = j < a.n_heads, first = have && i0 < hd;
  const int64_t o = (int64_t)r * a.H + (int64_t)j * hd;
  uint2 in[5] = {};   // biases of q, k, v; h; e
  if (first) {
#pragma unroll
    for (int t = 0; t < 3; ++t) in[t] = load_bias4(a.bias[t], j * hd + i0);
    in[3] = *reinterpret_cast<const uint2*>(a.h + o + i0);
    in[4] = *reinterpret_cast<const uint2*>(a.e + o + i0);
  }
  cudaGridDependencySynchronize();
  if (r == 0 && blockIdx.y == 0 && threadIdx.x == 0) a.status[0] = CLV_OK;
  if (!have) return;
  float4 x[3] = {};
  if (first) {
    Parts4 t[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) load_parts4(t[m], a.prod[m], o + i0, a.parts, a.stride);
#pragma unroll
    for (int m = 0; m < 3; ++m) x[m] = add4(sum_parts4(t[m], a.parts), bf16x4(in[m]));
  }
  auto load = [&](int m, int i) {
    Parts4 t;
    load_parts4(t, a.prod[m], o + i, a.parts, a.stride);
    return add4(sum_parts4(t, a.parts), bf16x4(load_bias4(a.bias[m], j * hd + i)));
  };
  float qk = 0.f, qq = 0.f, kk = 0.f;
  auto dots = [&](float4 u, float4 w) {
    qk += u.x * w.x + u.y * w.y + u.z * w.z + u.w * w.w;
    qq += u.x * u.x + u.y * u.y + u.z * u.z + u.w * u.w;
    kk += w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
  };
  dots(x[0], x[1]);
  for (int i = i0 + 128; i < hd; i += 128) dots(load(0, i), load(1, i));
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    qk += __shfl_xor_sync(0xFFFFFFFFu, qk, s);
    qq += __shfl_xor_sync(0xFFFFFFFFu, qq, s);
    kk += __shfl_xor_sync(0xFFFFFFFFu, kk, s);
  }
  const float gate = qk / fmaxf(sqrtf(qq) * sqrtf(kk), 1e-8f);
  uint16_t* dst = a.cat + (int64_t)r * 2 * a.H + (int64_t)j * hd;
  auto emit = [&](int i, float4 hv, float4 vv, uint2 ev) {
    *reinterpret_cast<uint2*>(dst + i) =
        to_bf16x4(make_float4(hv.x + vv.x * gate, hv.y + vv.y * gate, hv.z + vv.z * gate, hv.w + vv.w * gate));
    *reinterpret_cast<uint2*>(dst + a.H + i) = ev;
  };
  if (first) emit(i0, bf16x4(in[3]), x[2], in[4]);
  for (int i = i0 + 128; i < hd; i += 128)
    emit(i, bf16x4(*reinterpret_cast<const uint2*>(a.h + o + i)), load(2, i), *reinterpret_cast<const uint2*>(a.e + o + i));
}

// ---- the k largest of a row: highest first, lower index first among equals ----------------------
// An entry is a 64-bit key whose unsigned order is that order (the upper half orders the values, the
// lower one is the index, inverted); 0 = no entry.  A row is cut in slices of 2048 entries, one block
// each: a thread sorts its 8 entries, each warp picks the k best of its 256 (k rounds of two warp-wide
// maxima over the lanes' best entries; the winning lane moves on to its next), warp 0 picks the k best
// of the 8 warps' picks.  The last block of the row to finish picks the k best of all slices' picks
// the same way.  (With shuffles in place of the warp-wide maxima and a second launch for the last
// step, 4 rows x 128256 took 13 us.)
constexpr int kPerThread = 8, kSliceLen = kThreads * kPerThread, kListK = 32;
static_assert((kThreads / 32) * kListK <= 32 * kPerThread, "warp 0 holds all warps' picks");

__device__ __forceinline__ unsigned long long topk_key(float v, int i) {
  if (v != v) v = -INFINITY;   // NaN: after everything else
  if (v == 0.f) v = 0.f;       // -0 and +0 are the same value
  const uint32_t f = __float_as_uint(v);
  const uint32_t ord = (f & 0x80000000u) ? ~f : (f | 0x80000000u);
  return ((unsigned long long)ord << 32) | (uint32_t)~i;
}
__device__ __forceinline__ float key_value(unsigned long long key) {
  const uint32_t ord = (uint32_t)(key >> 32);
  return __uint_as_float((ord & 0x80000000u) ? ord & 0x7FFFFFFFu : ~ord);
}
__device__ __forceinline__ void sort8(unsigned long long (&v)[kPerThread]) {   // largest first (Batcher's network)
  constexpr int net[19][2] = {{0, 1}, {2, 3}, {4, 5}, {6, 7}, {0, 2}, {1, 3}, {4, 6}, {5, 7}, {1, 2}, {5, 6},
                              {0, 4}, {1, 5}, {2, 6}, {3, 7}, {2, 4}, {3, 5}, {1, 2}, {3, 4}, {5, 6}};
#pragma unroll
  for (int c = 0; c < 19; ++c) {
    const unsigned long long x = v[net[c][0]], y = v[net[c][1]];
    v[net[c][0]] = x > y ? x : y;
    v[net[c][1]] = x > y ? y : x;
  }
}
// the k best of the warp's sorted lists, in order, to out[0 .. k)
__device__ __forceinline__ void warp_select(unsigned long long (&v)[kPerThread], int k, unsigned long long* out) {
  const int lane = threadIdx.x & 31;
  for (int t = 0; t < k; ++t) {
    const uint32_t hi = (uint32_t)(v[0] >> 32), lo = (uint32_t)v[0];
    const uint32_t best = __reduce_max_sync(0xFFFFFFFFu, hi);
    const uint32_t idx = __reduce_max_sync(0xFFFFFFFFu, hi == best ? lo : 0u);
    if (lane == 0) out[t] = ((unsigned long long)best << 32) | idx;
    if (hi == best && lo == idx) {   // entries are distinct: this lane won (or nobody has an entry left)
#pragma unroll
      for (int u = 0; u + 1 < kPerThread; ++u) v[u] = v[u + 1];
      v[kPerThread - 1] = 0ull;
    }
  }
}
// the k best of the block's keys, in order, to s_best (warp 0 has them when it returns; the others wait for nothing)
__device__ __forceinline__ void block_select(unsigned long long (&v)[kPerThread], int k, unsigned long long* s_picks,
                                             unsigned long long* s_best) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  sort8(v);
  warp_select(v, k, s_picks + warp * k);
  __syncthreads();
  if (warp != 0) return;
#pragma unroll
  for (int u = 0; u < kPerThread; ++u) {
    const int j = lane * kPerThread + u;
    v[u] = j < (kThreads / 32) * k ? s_picks[j] : 0ull;
  }
  sort8(v);
  warp_select(v, k, s_best);
  __syncwarp();
}

// cand: [rows][slices][k] keys; tickets: a counter per row, zero between calls
__global__ void __launch_bounds__(kThreads) topk_slices_kernel(int n, int64_t ld, const float* logits, int k,
                                                               unsigned long long* cand, unsigned* tickets,
                                                               int32_t* ids, float* vals) {
  __shared__ unsigned long long s_picks[(kThreads / 32) * kListK], s_best[kListK];
  __shared__ int s_last;
  const int r = blockIdx.x, slice = blockIdx.y, slices = gridDim.y, tid = threadIdx.x;
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  unsigned long long v[kPerThread];
  {
    const int j0 = slice * kSliceLen + tid * kPerThread;
    const float* at = logits + (int64_t)r * ld + j0;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (j0 < n) {   // rows are padded to a multiple of 8 entries: the loads stay inside
      a = *reinterpret_cast<const float4*>(at);
      b = *reinterpret_cast<const float4*>(at + 4);
    }
    const float x[kPerThread] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) v[u] = j0 + u < n ? topk_key(x[u], j0 + u) : 0ull;
  }
  block_select(v, k, s_picks, s_best);
  unsigned long long* mine = cand + (int64_t)r * slices * k;
  if (slices > 1) {
    if (tid < k) __stcg(mine + (int64_t)slice * k + tid, s_best[tid]);   // k <= 32: warp 0
    if (tid < 32) {
      __threadfence();
      __syncwarp();
      if (tid == 0) s_last = atomicInc(tickets + r, (unsigned)slices - 1) == (unsigned)slices - 1;   // wraps to 0
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // all slices' picks, a block's worth at a time; what has been picked so far comes along
    const int total = slices * k, step = kSliceLen - kListK;
    for (int base = 0; base < total; base += step) {
#pragma unroll
      for (int u = 0; u < kPerThread; ++u) {
        const int j = u * kThreads + tid;
        if (j < step) v[u] = base + j < total ? __ldcg(mine + base + j) : 0ull;
        else v[u] = base > 0 && j - step < k ? s_best[j - step] : 0ull;
      }
      __syncthreads();   // s_picks and s_best have been read
      block_select(v, k, s_picks, s_best);
      __syncthreads();
    }
  }
  if (tid < k) {
    const unsigned long long key = s_best[tid];
    ids[(int64_t)r * k + tid] = key ? (int32_t)~(uint32_t)key : -1;
    vals[(int64_t)r * k + tid] = key ? key_value(key) : -INFINITY;
  }
}

__device__ __forceinline__ bool before(float v, int i, float bv, int bi) {   // order: value desc, index asc
  return (v > bv) || (v == bv && i < bi);
}
// More than 32 per row: k passes over the row (it stays in L2), each taking the best of what
// comes after the previous pass's pick.
__global__ void __launch_bounds__(kThreads) topk_passes_kernel(int V, int64_t ld, int k_top, const float* logits,
                                                               int32_t* ids, float* vals) {
  __shared__ float s_v[kThreads / 32];
  __shared__ int s_i[kThreads / 32];
  __shared__ float s_last_v;
  __shared__ int s_last_i;
  const int r = blockIdx.x, tid = threadIdx.x;
  const float* row = logits + (int64_t)r * ld;
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  float last_v = INFINITY;
  int last_i = -1;
  for (int t = 0; t < k_top; ++t) {
    float bv = -INFINITY;
    int bi = INT_MAX;
    for (int i = tid; i < V; i += kThreads) {
      float x = row[i];
      if (x != x) x = -INFINITY;
      const bool after = (x < last_v) || (x == last_v && i > last_i);
      if (after && before(x, i, bv, bi)) { bv = x; bi = i; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
      const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
      if (before(ov, oi, bv, bi)) { bv = ov; bi = oi; }
    }
    if ((tid & 31) == 0) { s_v[tid >> 5] = bv; s_i[tid >> 5] = bi; }
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < kThreads / 32; ++w)
        if (before(s_v[w], s_i[w], bv, bi)) { bv = s_v[w]; bi = s_i[w]; }
      s_last_v = bv;
      s_last_i = bi;
      ids[(int64_t)r * k_top + t] = (bi == INT_MAX) ? -1 : bi;
      vals[(int64_t)r * k_top + t] = bv;
    }
    __syncthreads();
    last_v = s_last_v;
    last_i = s_last_i;
    if (last_i == INT_MAX) last_v = -INFINITY;
  }
}

template <class K, class... A>
cudaError_t launch_rows(K kernel, dim3 grid, int threads, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

size_t topk_slices(int vocab) { return ((size_t)vocab + kSliceLen - 1) / kSliceLen; }

}  // namespace

// scratch layout (after the workspace's fixed part): x bf16 [R,H] | q, k, v fp32 [S1][R,H] each |
// cat bf16 [R,2H] | p fp32 [S2][R,H] | y bf16 [R,H] | logits fp32 [R, ldl] | the slices' picks
// u64 [R, slices, 32]   (S1, S2: parts of the K axis)
size_t draft_head_scratch_bytes(int rows, int hidden, int vocab) {
  const size_t R = rows, H = hidden, ldl = (vocab + 7) / 8 * 8;
  const size_t s1 = rows_linear_splits(rows, hidden, hidden, 3), s2 = rows_linear_splits(rows, 2 * hidden, hidden, 1);
  return up256(R * H * 2) + 3 * up256(s1 * R * H * 4) + up256(R * 2 * H * 2) + up256(s2 * R * H * 4) +
         up256(R * H * 2) + up256(R * ldl * 4) + up256(R * topk_slices(vocab) * kListK * 8);
}

cudaError_t launch_draft_head_step(const clv_draft_head& w, int rows, const void* h, const void* e, int k_top,
                                   void* hidden_out, int32_t* top_ids, float* top_logits, int32_t* status,
                                   unsigned* tickets, void* scratch, cudaStream_t stream) {
  const int H = w.hidden_dim, V = w.vocab;
  const size_t R = rows, ldl = (V + 7) / 8 * 8;
  const int s1 = rows_linear_splits(rows, H, H, 3), s2 = rows_linear_splits(rows, 2 * H, H, 1);
  const int64_t part = (int64_t)R * H;   // elements between the parts of a product
  char* s = static_cast<char*>(scratch);
  uint16_t* x = reinterpret_cast<uint16_t*>(s); s += up256(R * H * 2);
  float* q = reinterpret_cast<float*>(s); s += up256(s1 * R * H * 4);
  float* k = reinterpret_cast<float*>(s); s += up256(s1 * R * H * 4);
  float* v = reinterpret_cast<float*>(s); s += up256(s1 * R * H * 4);
  uint16_t* cat = reinterpret_cast<uint16_t*>(s); s += up256(R * 2 * H * 2);
  float* p = reinterpret_cast<float*>(s); s += up256(s2 * R * H * 4);
  uint16_t* y = reinterpret_cast<uint16_t*>(s); s += up256(R * H * 2);
  float* logits = reinterpret_cast<float*>(s); s += up256(R * ldl * 4);
  unsigned long long* cand = reinterpret_cast<unsigned long long*>(s);
  const uint16_t* h16 = static_cast<const uint16_t*>(h);
  const uint16_t* e16 = static_cast<const uint16_t*>(e);
  const dim3 per_row((unsigned)rows);
  cudaError_t err;
#define CLV_TRY(call) if ((err = (call)) != cudaSuccess) return err
  // status words: one per product (a wait of its kernel that ran out)
  CLV_TRY(launch_rows(rmsnorm_rows_kernel<true>, per_row, kNormThreads, stream, H, h16, (const float*)nullptr, 1, (int64_t)0,
                      (const uint16_t*)nullptr, static_cast<const uint16_t*>(w.norm1), w.rms_eps, x, (uint16_t*)nullptr,
                      status, 3));
  {   // q = x wq^T, k = e wk^T, v = e wv^T: one launch
    const void* const xs[3] = {x, e16, e16};
    const void* const ws[3] = {w.wq, w.wk, w.wv};
    float* const outs[3] = {q, k, v};
    CLV_TRY(launch_rows_linear(3, xs, H, ws, H, rows, H, H, outs, H, true, part, true, status + 0, tickets, stream));
  }
  const GateArgs gate = {H, (int)w.n_heads, s1, part, {q, k, v},
                         {static_cast<const uint16_t*>(w.bq), static_cast<const uint16_t*>(w.bk), static_cast<const uint16_t*>(w.bv)},
                         h16, e16, cat, status + 3};
  CLV_TRY(launch_rows(gate_residual_kernel, dim3((unsigned)rows, (unsigned)((w.n_heads + 7) / 8)), kThreads, stream, gate));
  {
    const void* const xs[1] = {cat};
    float* const outs[1] = {p};
    CLV_TRY(launch_rows_linear(1, xs, 2 * H, &w.wfc, 2 * H, rows, 2 * H, H, outs, H, true, part, true, status + 3, tickets,
                               stream));
  }
  CLV_TRY(launch_rows(rmsnorm_rows_kernel<false>, per_row, kNormThreads, stream, H, (const uint16_t*)nullptr, (const float*)p,
                      s2, part, static_cast<const uint16_t*>(w.bfc), static_cast<const uint16_t*>(w.norm2), w.rms_eps, y,
                      static_cast<uint16_t*>(hidden_out), status + 4, 1));
  {
    const void* const xs[1] = {y};
    float* const outs[1] = {logits};
    CLV_TRY(launch_rows_linear(1, xs, H, &w.lm_head, H, rows, H, V, outs, (int64_t)ldl, false, 0, true, status + 4, tickets,
                               stream));
  }
  if (k_top > kListK) {
    CLV_TRY(launch_rows(topk_passes_kernel, per_row, kThreads, stream, V, (int64_t)ldl, k_top, (const float*)logits,
                        top_ids, top_logits));
  } else {
    // (the products' counters lie at the start of the tickets)
    CLV_TRY(launch_rows(topk_slices_kernel, dim3((unsigned)rows, (unsigned)topk_slices(V)), kThreads, stream, V, (int64_t)ldl,
                        (const float*)logits, k_top, cand, tickets + 1024, top_ids, top_logits));
  }
#undef CLV_TRY
  return cudaSuccess;
}

}  // namespace clv
