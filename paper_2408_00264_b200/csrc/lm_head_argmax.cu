// LM head fused with the per-node greedy choice (Sec. 3.1: final norm and LM head of the target;
// Sec. 4.2: greedy decoding at T = 0): ids[r] = argmax_v round_bf16(<hidden[r, :], W[v, :]>), lowest
// v on ties.  The logits are never written: each tile of them (up to 256 rows x 256 entries) lives in
// tensor memory only, and its row maxima go to one 64-bit key per row with atomicMax.
//
// A persistent block per SM takes (vocabulary tile, row block) pairs, with few rows from a queue.  Warp 0 streams
// 64-wide K chunks of the weight tile ([up to 256 vocabulary rows][64]) and of the hidden rows ([1 or 2 x
// 128][64]) through a TMA ring, warp 1 issues tcgen05.mma (M 128, N = the tile's width, K 16; two
// accumulators of 256 columns fill the tensor memory), warps 2..9 are the epilogue: one thread per row
// scans the accumulator for the row's best (value, lowest index).  The weight matrix is read from HBM
// once per row block; the hidden rows are re-read from L2 by every block.
// With a handful of rows the kernel is a stream over the weights, and what is in flight sets its rate:
// the ring is as deep as shared memory allows and holds only the rows there are (4 rows x 128256 x 4096:
// 172.9 -> 159.5 us, the measured copy rate).  The width of a tile is chosen so that the tiles divide
// evenly over the SMs (plan()).  With many rows the tensor core bounds it, at the power cap (1024 rows of
// 128256 x 4096 in a loop: 810 us), and its operands, 64 bytes per cycle and SM from L2 for a tile of 256 x 256.
#include <cuda_bf16.h>
#include <limits.h>
#include <math.h>

#include "clv_internal.cuh"
#include "tc_ptx.cuh"
#include "tmem_access.cuh"

namespace clv {
namespace {

constexpr int kThreads = 320;
constexpr int BM = 128;              // rows per accumulator
constexpr int MB = 2 * BM;           // rows per block step (two accumulators)
constexpr int BN = 256;              // columns of an accumulator: the most vocabulary entries per tile
constexpr int BK = 64;               // K elements per ring stage (one 128-byte swizzle row)
constexpr int kMaxStages = 12;
constexpr int kItems = 16;           // more than the ring, the accumulators and the producer's next item can hold at a time
constexpr int kMaxProb = 3;          // products of one shape that one launch can take
constexpr uint32_t kATile = BM * BK * 2;      // 16 KB
constexpr uint32_t kSmemMost = 232448 - 1024;   // the ring (its alignment included); static shared memory is small
constexpr uint32_t kTmemCols = 512;

struct Params {
  int M, K, V;
  int n_tiles, m_blocks;
  int bn;                     // vocabulary entries per tile, a multiple of 16
  uint32_t idesc;
  int stages;                 // depth of the ring
  uint32_t stage_bytes;       // row operand tile(s), then the weight tile
  int early_weights;          // no launch that may still be running writes the weights: ask for the first tiles before
                              //   the previous kernel's results are waited for
  int32_t* ids;
  float* out;                 // not NULL: the products are written here, fp32 [M, ld_out], and no argmax is taken
  int n_prob;                 // with `out`: up to kMaxProb products of one shape in one launch, each with its own
  float* outs[3];             //   operands (tensor maps) and destination; out == outs[0]
  int64_t ld_out;
  int k_splits;               // with `out`: the K axis is cut in this many parts, part s writes its partial
  int64_t out_split_stride;   //   products to out + s * out_split_stride (the reader adds the parts up)
  int out_vec;                // `out` and its strides allow 16-byte accesses
  int use_queue;              // a block's items after its first come from a queue, else every gridDim.x-th is its own
  int two_acc;                // M <= 128: the two accumulators alternate between tiles, so that the
                              //   epilogue of one tile runs under the MMAs of the next
  int weights_first;          // `out` and two_acc: the weights are the MMA's 128-row operand (see below)
  uint32_t a_tile_bytes;      // bytes one load of the row operand brings (a box of 8..128 rows)
  unsigned long long* keys;   // [M], zero between calls
  unsigned* queue;            // [0] items handed out beyond each block's first, [1] blocks that have stopped drawing; zero between calls
  unsigned* counter;          // zero between calls
  unsigned* aborts;           // blocks that gave up a wait; zero between calls
  int32_t* status;            // CLV_OK or CLV_ERR_TIMEOUT; with `out` one word per product, which holds CLV_OK before the launch
  long long wait_limit;       // SM cycles a bounded wait may last
};

__device__ __forceinline__ unsigned long long pack_key(float v, int i) {
  if (v == 0.0f) v = 0.0f;  // -0 and +0 are the same value: one bit pattern
  const uint32_t f = __float_as_uint(v);
  const uint32_t ord = (f & 0x80000000u) ? ~f : (f | 0x80000000u);
  return ((unsigned long long)ord << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)i);
}
// A row's best logit of a tile so far, after rounding to bf16, for each of eight column positions (two per
// register): the value and the group of eight columns in which it came first, 0xFFFF: nothing above -inf yet.
// Branch free, four instructions per pair of columns.  A search of every chunk of 32 columns for its rounded
// maximum took a warp some 350 instructions per chunk, and with more than 128 rows the tensor core waits for
// the epilogue (1024 rows x 128256 x 4096 in a loop: 844 -> 811 us; 551 x 18771 x 2176, back to back: 53.6 -> 45.8;
// 513 x 32000 x 4096: 149.6 -> 123.2).
struct Best {
  __nv_bfloat162 v[4];
  uint32_t at[4];
};
// columns [8 * group, 8 * group + 16) of the tile
__device__ __forceinline__ void take_columns(Best& b, const uint32_t (&x)[16], uint32_t group) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const __nv_bfloat162 r = __floats2bfloat162_rn(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1]));
    const uint32_t above = __hgt2_mask(r, b.v[j & 3]);   // strictly: the first of equals stays; false for NaN
    b.v[j & 3] = __hmax2(b.v[j & 3], r);                 // NaN operands are dropped
    b.at[j & 3] = (b.at[j & 3] & ~above) | ((group + (uint32_t)(j >> 2)) * 0x00010001u & above);
  }
}

// What a work item is: a vocabulary tile, a row block, with `out` also a part of the K axis and a
// product.  Products are innermost, so that blocks working side by side read different weights; the
// row blocks of a tile follow each other, so that a weight tile is read from HBM once and from L2
// afterwards.
struct Item {
  int col0, mb, prob, part;
};
__device__ __forceinline__ Item decode_item(const Params& p, int item) {
  const int per_tile = p.k_splits * p.n_prob;
  const int tile = item / per_tile, sub = item - tile * per_tile, n = tile / p.m_blocks;
  Item it;
  it.part = sub / p.n_prob;
  it.prob = sub - it.part * p.n_prob;
  it.mb = tile - n * p.m_blocks;
  it.col0 = n * p.bn;
  return it;
}

struct Maps {
  CUtensorMap a[kMaxProb], w[kMaxProb];
};

__global__ void __launch_bounds__(kThreads, 1)
lm_head_argmax_kernel(const __grid_constant__ Maps tm, const Params p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) unsigned long long s_bar[2 * kMaxStages + 5];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  __shared__ int s_last;
  __shared__ volatile int s_item[kItems];   // the block's items in turn, -1 behind the last

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bar0 = smem_u32(&s_bar[0]);
  auto bar_full = [&](int s) { return bar0 + 8u * s; };
  auto bar_empty = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
  // a tile's accumulators are complete / the epilogue has read them; index 1 only with two_acc
  auto bar_acc_full = [&](int b) { return bar0 + 8u * (2 * kMaxStages + b); };
  auto bar_acc_empty = [&](int b) { return bar0 + 8u * (2 * kMaxStages + 2 + b); };
  const uint32_t bar_drain = bar0 + 8u * (2 * kMaxStages + 4);
  if (tid == 0) {
    for (int i = 0; i < 2 * kMaxStages; ++i) mbar_init(bar0 + 8u * i, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_acc_full(b), 1);
      mbar_init(bar_acc_empty(b), p.two_acc ? BM : 2 * BM);
    }
    mbar_init(bar_drain, 1);
    s_abort = 0;
    fence_barrier_init();
    fence_async_smem();
  }
  if (warp == 1) tmem_alloc(smem_u32(&s_tmem), kTmemCols);
  if (tid >= 64 && tid < 64 + p.n_prob) {
    tma_prefetch_desc(&tm.a[tid - 64]);
    tma_prefetch_desc(&tm.w[tid - 64]);
  }
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  volatile int* abort_flag = &s_abort;
  const long long wlim = p.wait_limit;

  // Within a stage: the row operand, then the weight tile.  With fewer than 128 rows the operand takes the
  // box that was loaded; the rest of its 128 rows is whatever lies behind it (the weights): rows of
  // a product do not mix, and nobody reads those.
  const uint32_t w_at = p.two_acc ? p.a_tile_bytes : 2u * kATile;
  auto sA = [&](int s, int mt) { return smem_base + (uint32_t)s * p.stage_bytes + (uint32_t)mt * kATile; };
  auto sW = [&](int s) { return smem_base + (uint32_t)s * p.stage_bytes + w_at; };
  const int n_items = p.n_tiles * p.m_blocks * p.k_splits * p.n_prob;
  const int k_chunks = p.K / BK / p.k_splits;
  int issued = 0;  // ring stages filled by the producer (for the drain)
  if (!p.early_weights || warp != 0) cudaGridDependencySynchronize();  // programmatic launch: the previous kernel's results are complete
  cudaTriggerProgrammaticLaunchCompletion();

  if (warp == 0) {
    // =========================== TMA producer ===============================================
    // A block's first item is its number.  With few rows the others come from a queue, because the SMs do
    // not get equal shares of the memory's bandwidth (with equal numbers of tiles the fastest was done after
    // 0.75 of the time of the slowest).  With more than 128 the tensor core sets the pace, the same on every
    // SM, and the queue's end cost more than it brought: a block takes every gridDim.x-th item (551 rows x 18771 x
    // 2176: 54.7 -> 53.6 us, 513 x 32000 x 4096: 154.9 -> 149.6, 768 x 16384 x 1024: 31.0 -> 30.3).
    if (lane == 0) {
      bool ok = true;
      int s = 0, n = 0, item = blockIdx.x;
      uint32_t round = 0;
      auto load_w = [&](const Item& wi, int chunk, int st) {
        mbar_expect_tx(bar_full(st), (uint32_t)p.bn * BK * 2 + ((p.M - wi.mb * MB) > BM ? 2u : 1u) * p.a_tile_bytes);
        tma_load_2d(sW(st), &tm.w[wi.prob], (wi.part * k_chunks + chunk) * BK, wi.col0, bar_full(st));
      };
      int early = 0;
      if (p.early_weights) {   // the weights of the first item's first stages; the rows follow below
        const Item wi = decode_item(p, item);
        early = min(p.stages, k_chunks);
        s_item[0] = item;   // ahead of the arrivals by which its readers are ordered
        for (int i = 0; i < early; ++i) load_w(wi, i, i);
        cudaGridDependencySynchronize();
      }
      for (; ok; ++n) {
        const bool end = item >= n_items;
        if (end && !p.use_queue) break;
        unsigned ticket = 0;
        if (!end && p.use_queue) ticket = atomicAdd(p.queue, 1u);   // the next item, looked at when this one has been asked for
        const Item wi = decode_item(p, item);
        if (end) s_item[(n + 1) % kItems] = -1;
        s_item[n % kItems] = end ? -1 : item;
        for (int kc = 0; kc < (end ? 1 : k_chunks) && ok; ++kc) {
          if (issued >= p.stages) ok = mbar_wait(bar_empty(s), (round & 1u) ^ 1u, abort_flag, wlim);
          if (!ok) break;
          if (end) {
            mbar_arrive(bar_full(s));   // nothing to load: the issuer finds the end in s_item
          } else {
            if (issued >= early) load_w(wi, kc, s);
            for (int mt = 0; mt < ((p.M - wi.mb * MB) > BM ? 2 : 1); ++mt)
              tma_load_2d(sA(s, mt), &tm.a[wi.prob], (wi.part * k_chunks + kc) * BK, wi.mb * MB + mt * BM, bar_full(s));
          }
          ++issued;
          if (++s == p.stages) { s = 0; ++round; }
        }
        if (end) break;
        item = (p.use_queue ? (int)ticket : item) + (int)gridDim.x;
      }
      if (p.use_queue) {   // the last block to stop drawing leaves the queue empty for the next call
        __threadfence();
        if (atomicInc(p.queue + 1, gridDim.x - 1) == gridDim.x - 1) *p.queue = 0u;
      }
    }
  } else if (warp == 1) {
    // =========================== MMA issuer ===================================================
    // The whole warp walks the schedule and one elected lane issues.
    const uint32_t el = elect_one();
    bool ok = true;
    int s = 0;
    uint32_t round = 0;
    // accumulator (pair) of tile t is free: the epilogue has taken its previous tile out of tensor memory
    auto acc_free = [&](int t) {
      const int acc = p.two_acc ? (t & 1) : 0, use = p.two_acc ? (t >> 1) : t;
      if (use > 0 && !wait_warp(bar_acc_empty(acc), (use - 1) & 1, abort_flag, wlim)) return false;
      tc_fence_after();
      return true;
    };
    for (int tile = 0; ok; ++tile) {
      int item = (int)(blockIdx.x + tile * gridDim.x);
      if (!p.use_queue && item >= n_items) break;
      ok = wait_warp(bar_full(s), round & 1u, abort_flag, wlim);
      if (!ok) break;
      if (p.use_queue) item = __shfl_sync(0xFFFFFFFFu, (int)s_item[tile % kItems], 0);
      ok = acc_free(tile);
      if (!ok) break;
      const int acc = p.two_acc ? (tile & 1) : 0;
      if (item < 0) {   // tell the epilogue's groups: with two_acc each waits for an accumulator of its own
        umma_commit_if(el, bar_acc_full(acc));
        if (p.two_acc && acc_free(tile + 1)) umma_commit_if(el, bar_acc_full(acc ^ 1));
        break;
      }
      const int m_tiles = (p.M - decode_item(p, item).mb * MB) > BM ? 2 : 1;
      for (int kc = 0; kc < k_chunks && ok; ++kc) {
        if (kc > 0) ok = wait_warp(bar_full(s), round & 1u, abort_flag, wlim);
        if (!ok) break;
        tc_fence_after();
        const uint64_t wd = smem_desc(sW(s), 16, 1024);
        for (int mt = 0; mt < m_tiles; ++mt) {
          const uint64_t ad = smem_desc(sA(s, mt), 16, 1024);
          if (p.weights_first) {
            for (int v = 0; v < (p.bn > BM ? 2 : 1); ++v) {
              const uint64_t vd = wd + (uint64_t)((uint32_t)(v * (p.bn - BM)) * (BK * 2) >> 4);
#pragma unroll
              for (int ks = 0; ks < BK / 16; ++ks)
                umma_bf16_if(el, tmem + (uint32_t)(acc * BN + v * BM), vd + (uint64_t)((ks * 32) >> 4), ad + (uint64_t)((ks * 32) >> 4),
                             p.idesc, (kc > 0 || ks > 0) ? 1u : 0u);
            }
            continue;
          }
#pragma unroll
          for (int ks = 0; ks < BK / 16; ++ks)
            umma_bf16_if(el, tmem + (uint32_t)((mt + acc) * BN), ad + (uint64_t)((ks * 32) >> 4), wd + (uint64_t)((ks * 32) >> 4),
                         p.idesc, (kc > 0 || ks > 0) ? 1u : 0u);
        }
        umma_commit_if(el, bar_empty(s));  // the stage is free once these MMAs have read it
        if (++s == p.stages) { s = 0; ++round; }
      }
      if (ok) umma_commit_if(el, bar_acc_full(acc));
    }
  } else {
    // =========================== epilogue: one thread per row ==================================
    const int mt = (warp - 2) >> 2;          // accumulator of this group
    const int quarter = warp & 3;            // tensor-memory lanes this warp may touch
    const int row_in_tile = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    for (int tile = p.two_acc ? mt : 0;; tile += p.two_acc ? 2 : 1) {
      const int acc = p.two_acc ? mt : 0;
      int item = (int)(blockIdx.x + tile * gridDim.x);
      if (!p.use_queue && item >= n_items) break;
      if (!wait_warp(bar_acc_full(acc), (p.two_acc ? (tile >> 1) : tile) & 1, abort_flag, wlim)) break;
      if (p.use_queue) item = s_item[tile % kItems];
      if (item < 0) break;
      tc_fence_after();
      const Item wi = decode_item(p, item);
      const int row = wi.mb * MB + (p.two_acc ? 0 : mt * BM) + row_in_tile;
      const int lim = min(p.V, wi.col0 + p.bn);   // end of the tile's columns
      const bool row_valid = row < p.M;
      // the second accumulator is unused for a short row block
      const bool group_used = p.two_acc || (p.M - wi.mb * MB) > mt * BM;
      float best_v = -INFINITY;
      int best_i = INT_MAX;
      if (p.weights_first) {   // a lane per vocabulary entry, a column per row
        float* const out = (wi.prob == 0 ? p.outs[0] : wi.prob == 1 ? p.outs[1] : p.outs[2]) + wi.part * p.out_split_stride;
        for (int v = 0; v < (p.bn > BM ? 2 : 1); ++v) {
          const int entry = v * (p.bn - BM) + row_in_tile;
          const bool mine = wi.col0 + entry < lim && (v == 0 || entry >= BM);   // the two spans of 128 entries may overlap
#pragma unroll 1
          for (int c = 0; c < p.M; c += 16) {
            uint32_t x[16];
            tmem_ld_x16(tmem + lane_addr + (uint32_t)(mt * BN + v * BM + c), x);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (mine && c + j < p.M) out[(int64_t)(c + j) * p.ld_out + wi.col0 + entry] = __uint_as_float(x[j]);
          }
          __syncwarp();
        }
      } else if (group_used && p.out == nullptr) {   // a chunk of 16 columns is fetched while the one before it is taken
        // (chunks of 32 took 153 registers: the small kernels between the draft head's products found no room
        // beside this one, 1 x 119116 x 2048: 109.4 -> 113.1 us)
        Best best;
#pragma unroll
        for (int j = 0; j < 4; ++j) { best.v[j] = __float2bfloat162_rn(-INFINITY); best.at[j] = 0xFFFFFFFFu; }
        uint32_t x[2][16];
        const uint32_t acc_addr = tmem + lane_addr + (uint32_t)(mt * BN);
        tmem_ld_x16(acc_addr, x[0]);
#pragma unroll 1
        for (int c0 = 0; c0 < p.bn; c0 += 32) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int c = c0 + 16 * h;   // a tile's width is a multiple of 16
            if (c >= p.bn) continue;
            tmem_wait_ld();
            if (c + 16 < p.bn) tmem_ld_x16(acc_addr + (uint32_t)(c + 16), x[h ^ 1]);
            if (wi.col0 + c + 16 > lim) {   // the last of the vocabulary
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (wi.col0 + c + j >= lim) x[h][j] = 0xFF800000u;
            }
            take_columns(best, x[h], (uint32_t)c >> 3);
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t group = (j & 1) ? best.at[j >> 1] >> 16 : best.at[j >> 1] & 0xFFFFu;
          const float v = (j & 1) ? __high2float(best.v[j >> 1]) : __low2float(best.v[j >> 1]);
          const int i = wi.col0 + 8 * (int)group + j;
          if (group != 0xFFFFu && (v > best_v || (v == best_v && i < best_i))) { best_v = v; best_i = i; }
        }
      } else if (group_used) {
#pragma unroll 1
        for (int c = 0; c < p.bn; c += 32) {
          uint32_t x[32];
          tmem_ld_x32(tmem + lane_addr + (uint32_t)(mt * BN + c), x);
          tmem_wait_ld();
          if (row_valid) {   // plain product: this row's 32 values go to memory
            float* dst = (wi.prob == 0 ? p.outs[0] : wi.prob == 1 ? p.outs[1] : p.outs[2]) +
                         wi.part * p.out_split_stride + (int64_t)row * p.ld_out + wi.col0 + c;
#pragma unroll
            for (int j = 0; j < 8; ++j) {   // four values at a time; the last of a tile or row one by one
              const int at = wi.col0 + c + 4 * j;
              if (p.out_vec && at + 4 <= lim) {
                reinterpret_cast<uint4*>(dst)[j] = make_uint4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
              } else {
#pragma unroll
                for (int t = 0; t < 4; ++t)
                  if (at + t < lim) dst[4 * j + t] = __uint_as_float(x[4 * j + t]);
              }
            }
          }
        }
      }
      tc_fence_before();
      mbar_arrive(bar_acc_empty(acc));
      if (row_valid && best_i != INT_MAX) atomicMax(p.keys + row, pack_key(best_v, best_i));
    }
  }

  // ---- teardown --------------------------------------------------------------------------------
  __syncwarp();
  if (*abort_flag) {
    if (warp == 0 && lane == 0)
      for (int i = max(0, issued - p.stages); i < issued; ++i) mbar_drain(bar_full(i % p.stages), (i / p.stages) & 1);
    if (warp == 1) {
      umma_commit_if(elect_one(), bar_drain);
      mbar_drain(bar_drain, 0);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
  if (p.out != nullptr) {   // no keys were written
    if (tid == 0 && *abort_flag)
      for (int i = 0; i < p.n_prob; ++i) p.status[i] = CLV_ERR_TIMEOUT;
    return;
  }
  if (tid == 0) {
    if (*abort_flag) atomicAdd(p.aborts, 1u);
    __threadfence();
    const unsigned arrived = atomicInc(p.counter, gridDim.x - 1);  // wraps to 0
    s_last = (arrived == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return;
  // the last block turns the keys into indices and leaves keys and counters zero for the next call
  __threadfence();
  if (tid == 0) p.status[0] = atomicExch(p.aborts, 0u) ? (int)CLV_ERR_TIMEOUT : (int)CLV_OK;
  for (int r = tid; r < p.M; r += kThreads) {
    const unsigned long long key = atomicExch(p.keys + r, 0ull);
    const int idx = (int)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
    p.ids[r] = (key == 0ull) ? 0 : idx;  // a row of only -inf / NaN logits: first index
  }
}

bool make_map_2d(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t k, int64_t ld, uint32_t box_rows) {
  const cuuint64_t dims[2] = {(cuuint64_t)k, rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)BK, box_rows};
  return encode_tile_map(tm, base, 2, dims, strides, box);
}

}  // namespace

bool lm_head_supported(int rows, int hidden, int vocab) {
  // keys share the zero-initialised counter area of the workspace: 2 words per row after the counter
  return rows > 0 && vocab > 0 && hidden > 0 && (hidden % BK) == 0 && 2 * (int64_t)rows + 2 <= kTickets &&
         encode_fn() != nullptr;
}

namespace {
// How a product is cut: vocabulary entries per tile and parts of the K axis.  A tile of bn entries and
// k_chunks chunks takes about k_chunks * bn * 5.6 cycles when it streams weights from HBM (one SM's
// share of the bandwidth) or 4.3 of tensor core (16 columns more count for what a narrow tile costs: the
// rows are read more often), and some more per tile; what counts is the number of rounds over the SMs
// times that.  60 rows x vocabulary 32000 x 4096: 143 tiles of 224 keep 143 SMs busy where 125 tiles of
// 256 left 23 idle, 51.2 -> 47.4 us.  Below 128 entries a stage of the ring would bring too little.
// Every stage brings the rows again beside its weights: they count one and a half times, for the bandwidth
// and for the ring that they take (44 rows x 62745 x 2624: three rounds of tiles of 144 took 78 us, two
// of 256 take 64).
struct Cut {
  int bn, splits;
};
// rows one load of the row operand brings: the power of two that covers them, 8..128
int row_box(int rows) {
  int box = BM;
  while (box > 8 && box / 2 >= rows) box /= 2;
  return box;
}
Cut plan(int rows, int in_dim, int out_dim, int n, bool may_split) {
  const int m_blocks = (rows + MB - 1) / MB, chunks = in_dim / BK;
  const bool stream = rows <= BM;
  const int box = row_box(rows);
  Cut best = {BN, 1};
  double best_cost = 1e300;
  for (int sp = 1; sp <= (may_split ? 8 : 1); sp *= 2) {
    if (chunks % sp) break;
    for (int bn = BN; bn >= 128; bn -= 16) {
      const int64_t items = (int64_t)((out_dim + bn - 1) / bn) * m_blocks * n * sp;
      const double rounds = (double)((items + sm_count() - 1) / sm_count());
      const double cost = rounds * ((double)(chunks / sp) * (stream ? (bn + 1.5 * box) * 5.6 : (bn + 16) * 4.3) + (stream ? 700.0 : 4000.0)) + 200.0 * sp;
      if (cost < best_cost) { best_cost = cost; best = {bn, sp}; }
    }
  }
  return best;
}

struct Product {   // one product of a launch: rows x[rows, K] times weight[vocab, K]^T -> out
  const void* x;
  const void* weight;
  float* out;
};

cudaError_t launch_rows_times_weights(int n_prob, const Product* pr, int64_t ld_hidden, int64_t ld_weight, int rows,
                                      int hidden_dim, int vocab, int32_t* ids, int64_t ld_out, Cut cut,
                                      int64_t out_split_stride, bool early_weights, int32_t* status, unsigned* tickets,
                                      cudaStream_t stream) {
  static OncePerDevice once;
  cudaError_t e0 = run_once_per_device(once, [] {
    return cudaFuncSetAttribute(lm_head_argmax_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMost);
  });
  if (e0 != cudaSuccess) return e0;
  if (n_prob < 1 || n_prob > kMaxProb) return cudaErrorInvalidValue;
  Maps tm;
  const int a_box = row_box(rows);
  Params p;
  bool vec = (ld_out % 4) == 0 && (out_split_stride % 4) == 0;
  for (int i = 0; i < kMaxProb; ++i) {
    const Product& q = pr[i < n_prob ? i : 0];   // unused slots repeat the first product
    if (!make_map_2d(&tm.a[i], q.x, (uint64_t)rows, (uint64_t)hidden_dim, ld_hidden, (uint32_t)a_box) ||
        !make_map_2d(&tm.w[i], q.weight, (uint64_t)vocab, (uint64_t)hidden_dim, ld_weight, (uint32_t)cut.bn))
      return cudaErrorInvalidValue;
    p.outs[i] = q.out;
    vec = vec && (reinterpret_cast<uintptr_t>(q.out) % 16) == 0;
  }
  p.M = rows;
  p.K = hidden_dim;
  p.V = vocab;
  p.n_tiles = (vocab + cut.bn - 1) / cut.bn;
  p.bn = cut.bn;
  p.m_blocks = (rows + MB - 1) / MB;
  p.ids = ids;
  p.out = pr[0].out;
  p.n_prob = n_prob;
  p.ld_out = ld_out;
  p.k_splits = cut.splits;
  p.early_weights = early_weights;
  p.out_split_stride = out_split_stride;
  p.out_vec = p.out != nullptr && vec;
  p.two_acc = rows <= BM;
  p.use_queue = p.two_acc;
  // A few rows against many weights: with the rows as the 128-row operand every MMA multiplies 128 rows, most
  // of them whatever lies behind the real ones, and a step of the draft head runs into the power cap
  // (in a loop: 920 W, 1.43-1.6 GHz, 225-241 us by card).  With the weights there, an MMA has 16 columns for up
  // to 16 rows, and the step keeps 1.97 GHz at 800 W: 220 us.
  // (The fused argmax keeps a thread per row.)
  p.weights_first = p.two_acc && p.out != nullptr;
  p.idesc = p.weights_first ? make_idesc(BM, a_box > 16 ? a_box : 16, false) : make_idesc(BM, cut.bn, false);
  p.a_tile_bytes = (uint32_t)a_box * BK * 2;
  p.queue = ws_queue(tickets);
  p.counter = tickets;
  p.aborts = tickets + 1;
  p.keys = reinterpret_cast<unsigned long long*>(tickets + 2);
  p.status = status;
  p.wait_limit = wait_limit_cycles();
  p.stage_bytes = (p.two_acc ? p.a_tile_bytes : 2u * kATile) + (uint32_t)cut.bn * BK * 2;   // >= 16 KB: an operand ends inside
  p.stages = (int)((kSmemMost - 1024) / p.stage_bytes);
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  const int work = p.n_tiles * p.m_blocks * cut.splits * n_prob;
  const int grid = work < sm_count() ? work : sm_count();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = p.stages * p.stage_bytes + 1024;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lm_head_argmax_kernel, tm, p);
}
}  // namespace

cudaError_t launch_lm_head_argmax(const void* hidden, int64_t ld_hidden, const void* weight, int64_t ld_weight,
                                  int rows, int hidden_dim, int vocab, int32_t* ids, int32_t* status,
                                  unsigned* tickets, cudaStream_t stream) {
  const Product pr = {hidden, weight, nullptr};
  return launch_rows_times_weights(1, &pr, ld_hidden, ld_weight, rows, hidden_dim, vocab, ids, 0,
                                   plan(rows, hidden_dim, vocab, 1, false), 0, false, status, tickets, stream);
}

// How many parts the K axis of `n` products of one shape in one launch is cut into.
int rows_linear_splits(int rows, int in_dim, int out_dim, int n) { return plan(rows, in_dim, out_dim, n, true).splits; }

// out[i][part][r][o] = sum over part's share of k of x[i][r][k] * weight[i][o][k] for n products of one shape (n <= 3) in one launch: the same kernel with its
// accumulators written out (fp32) instead of reduced to an argmax.  in_parts: the reader adds
// rows_linear_splits() parts up (a fixed order: the result does not depend on scheduling); else there
// is one.  status: one word per product, CLV_OK before the launch.  early_weights: no launch that may
// still be running when this one starts writes any of the weights, so the first tiles of them are
// asked for without waiting.
cudaError_t launch_rows_linear(int n, const void* const* x, int64_t ld_x, const void* const* weight,
                               int64_t ld_weight, int rows, int in_dim, int out_dim,
                               float* const* out, int64_t ld_out, bool in_parts, int64_t split_stride, bool early_weights,
                               int32_t* status, unsigned* tickets, cudaStream_t stream) {
  if (n < 1 || n > kMaxProb) return cudaErrorInvalidValue;
  Product pr[kMaxProb];
  for (int i = 0; i < n; ++i) pr[i] = Product{x[i], weight[i], out[i]};
  return launch_rows_times_weights(n, pr, ld_x, ld_weight, rows, in_dim, out_dim, nullptr, ld_out,
                                   plan(rows, in_dim, out_dim, n, in_parts), split_stride, early_weights, status, tickets, stream);
}

}  // namespace clv
