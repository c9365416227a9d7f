// Tree attention (Sec. 2.1) on the 5th-generation tensor cores: tcgen05.mma with accumulators in
// tensor memory, K/V/Q tiles staged by TMA into 128-byte-swizzled shared memory.
//
// Query row = (tree node, head-in-group) pair, so all G heads of a GQA group and all tree nodes
// reuse every K/V byte.  A row tile of 128 rows holds whole nodes: 128 / G of them (rounded down;
// its other rows idle).  The key axis (cache keys first, then the tree's own) is walked in tiles of
// 128 keys that are loaded as 64-key pieces (also the page size of a paged cache).
//
// A thread block has two SLOTS, each with a score buffer and an output accumulator of its own in
// tensor memory (4 x 128 columns) and four softmax warps of its own, one thread per query row:
//   kRows2    the slots are two row tiles of the same (sequence, kv head); both take every key tile,
//             so a staged K/V tile serves 256 rows;
//   otherwise the slots share one row tile and take the key tiles in turn (even, odd); their two
//             partial results are combined like those of two blocks.
// If the row tile has 64 rows or fewer (kParts = 2; 32: kParts = 4), Q is loaded that many times, one copy
// below the other, and a row's keys are shared out over its copies: the softmax thread of a copy takes 64
// (32) of a tile's 128 scores, has zeros for the others, and ends up with a partial result of its own.
// The MMAs take what they take for 128 rows anyway; the softmax, which is what a short call waits for, is
// half (a quarter) as long and keeps all four of the SM's quadrants busy (whole steps in a loop, 1 x 16 nodes x
// 512 keys: 15.8 -> 14.8 us; 32 layers of 1 x 60 nodes x 1500 keys and LM head: 500 -> 470 us).
// What bounds a key tile of 128 x 128 scores: Q K^T and P V are 16 MMAs of 64 cycles, the
// exponentials 1024 cycles of the special-function units, and within a slot the two alternate (scores
// -> exponentials -> P V -> next scores).  With two slots the tensor core works for one while the
// other is in its exponentials, and P is handed over in two parts (96 and 32 keys), so that only the last
// quarter of P V is left when the exponentials are done.  (Three parts of 64, 32 and 32, the second after the
// last exponentials: half of it was left; 3 x 64 nodes x 16384 keys 64.8 -> 62.2 us, 8 x 128 x 32768 508 -> 500.)
// Leaving the exponentials out altogether does not shorten a call: what a tile takes is the chain through
// both units and the waits between them, so what counts is the length of a thread's instructions.
//
// Softmax: a thread takes its row's 128 scores into registers and writes P (bf16) back over the score
// columns.  The exponentials of the first 64 keys are computed with the row's reference as it stands,
// beside the maximum of the others; their sum, which the row needs anyway, says whether one of them is above
// 2^8 (their maximum besides: 3 x 64 x 16384 62.9 -> 60.7 us, 8 x 128 x 32768 500 -> 487).  The reference is replaced
// (O rescaled, those exponentials redone) only when a score exceeds it by 2^8 or their sum does: P is bf16 and the sums are fp32, so a probability above 1 costs
// no precision, only range (an accumulator holds |V| up to about 2^120), and after a row's first tile the
// replacement is a rare event.
// The tree columns are masked with ancestor bitsets derived from parent[]; masked scores are replaced
// by -inf, not added to, so they contribute exactly zero.
//
// Split-KV: the blocks that share row tiles form a thread-block cluster (1..8 along the key axis).
// Each sends the accumulator rows that another one finalises as fp16 (half a row scaled by a power of
// two of its own: 2^-11 relative, against the output's 2^-9) with their reference and sum, by bulk
// copies from its shared memory to the other's, into tile memory that is idle by then.  What is
// added up within a block (the slots; the parts of a row if the block is alone) stays fp32.
// No partial result touches global memory.
// Every wait is bounded: on expiry the block raises a flag, all roles leave their loops, in-flight
// copies and MMAs are drained and CLV_ERR_TIMEOUT is reported for the sequence.  That includes the
// waits of the merge (the last P V, the other ranks' rows): no rows are written behind one that ran out.
#include <cuda.h>
#include <cuda_fp16.h>
#include <math.h>

#include "clv_internal.cuh"
#include "seq_status.cuh"
#include "tc_ptx.cuh"
#include "tmem_access.cuh"

namespace clv {
namespace {

constexpr int PG = CLV_PAGE_SIZE;      // 64: keys per TMA piece (= page size)
constexpr int HD = CLV_HEAD_DIM;       // 128
constexpr int BM = 128;                // rows per slot
constexpr int BN = 128;                // keys per tile
constexpr int CH = 32;                 // keys whose scores one load brings
constexpr int kThreads = 384;          // warps 0-3 and 4-7: the slots' softmax; 8: TMA producer; 9: MMA issuer; 10 reports; 11 asks ahead
// Registers per thread: the launch's 168 cannot hold a row's 128 scores and the rest of a softmax
// thread, so the third warpgroup's go to the first two while the roles work (256 x 216 + 128 x 72 =
// 384 x 168; 4 x 64 nodes x 4096 keys, launch to launch: 28.0 -> 26.5 us).  No variant spills (-Xptxas -v).
constexpr int kSoftmaxRegs = 216, kOtherRegs = 72, kLaunchRegs = 168;
static_assert(2 * kSoftmaxRegs + kOtherRegs <= 3 * kLaunchRegs, "a block shares out the registers that it was launched with");
constexpr int kSoftmaxWarps = 8, kProducer = 8, kIssuer = 9, kWriter = 10, kScout = 11;
constexpr int kMaxSplits = 8;          // portable cluster size
constexpr uint32_t kQTile = BM * HD * 2;      // 32 KB: two [128 rows][64 d] swizzled halves
constexpr uint32_t kPiece = PG * 64 * 2;       // 8 KB: [64 keys][64 d] swizzled, one TMA box
constexpr uint32_t kStage = BN * HD * 2;       // 32 KB: a K (or V) tile, [64-wide half of d][128 keys][64 d]
constexpr uint32_t kHalf = kStage / 2;
constexpr uint32_t kTmemCols = 512;
constexpr float kRefSlack = 8.f;      // log2 units a score may exceed the row's reference by
constexpr float kTopP = 256.f;        // the same for its probability
constexpr uint32_t kIdescQK = make_idesc(BM, BN, false);  // S[128 rows x 128 keys] = Q K^T
constexpr uint32_t kIdescPV = make_idesc(BM, HD, true);   // O[128 rows x 128 d] += P V

template <bool kRows2, int kParts>
struct Cfg {
  static constexpr int kRows = BM / kParts;      // rows of a row tile
  static constexpr int kQ = kRows2 ? 2 : 1;      // row tiles
  static constexpr int NST = kRows2 ? 5 : 6;     // ring stages: K and V tiles in turn
  static constexpr int kStep = kRows2 ? 2 : 4;   // loads from one tile of a slot to its next
};

// What the merge sends of a row: its columns as fp16, and 16 bytes of reference, sum and scales (of either half of
// the columns, where different warps send them).
template <bool kRows2>
constexpr uint32_t kRowBytes = HD * 2 + (kRows2 ? 16 : 32);

// barriers: stage full [6] | stage empty [6] | S full [2] | part of P [2][2] | last P V done [2] | Q | merge | drain
constexpr int B_FULL = 0, B_EMPTY = 6, B_S = 12, B_P = 14, B_LAST = 18, B_Q = 20, B_RX = 21, B_DR = 22, NBAR = 23;

// What the merge needs to know about its block, the launch's constants among it (in shared memory meanwhile: see there).
struct __align__(16) Place {
  int b, split, kvh, users;
  int T, R, per, first;
  int mine, tile0, CS, N;
  int G, Hq, tile_nodes, tiles;
  int group_d;
  unsigned group_m, meta;              // by_group_heads; where a third idle stage starts in the ring
  uint16_t* out;
  float* lse;
  uint32_t rx[kMaxSplits];             // where each rank receives, in its ring
};
struct Misc {                           // behind the tiles in dynamic shared memory
  float2 ml[2 * BM];                    // (reference, sum) of every row of both slots
  unsigned long long bar[NBAR];
  uint32_t tmem;
  int abort_flag;                       // a wait of the roles ran out
  int late_flag;                        // the wait for the last P V did
  int seq;                              // the block's sequence, if they are handed out by length
  Place place;
  int issued;                           // loads issued (producer)
  signed char parent[CLV_MAX_NODES];    // as far as valid, -1 otherwise
};
constexpr uint32_t kMiscAt = 7 * kStage;   // either way: Q tiles + ring = 224 KB
constexpr uint32_t kSmem = kMiscAt + (uint32_t)sizeof(Misc);
static_assert(Cfg<true, 1>::kQ + Cfg<true, 1>::NST == 7 && Cfg<false, 1>::kQ + Cfg<false, 1>::NST == 7 && kSmem <= 232448, "shared memory");

// pieces of n >= 0 keys, up to the largest length there is (n + PG - 1 does not fit in an int for the last 63 of them)
__host__ __device__ __forceinline__ int pieces_of(int n) { return (int)(((unsigned)n + (unsigned)(PG - 1)) / PG); }

// n / d by a multiplication: m = ceil(2^32 / d), so the high word is n / d or one more.  (A division of
// the language is some 40 instructions that a block runs once, from a cold instruction cache.)
struct Divisor {
  unsigned d, m;   // m = 0: d = 1
  static Divisor of(unsigned d) { return Divisor{d, d > 1 ? (unsigned)(((1ull << 32) + d - 1) / d) : 0u}; }
  __device__ __forceinline__ unsigned divide(unsigned n) const {
    const unsigned q = m ? __umulhi(n, m) : n;
    return q - (q * d > n ? 1u : 0u);
  }
};

struct Params {
  const int32_t* block_table;
  const int32_t* parent;
  const int32_t* ctx_len;
  uint16_t* out;
  float* lse;
  int32_t* status;
  int B, N, Hq, Hkv, G;
  int paged, cap_tokens, n_pages, max_pages;
  int longest_first;  // hand out sequences in order of decreasing context length
  int ask_ahead;      // the first key tiles into L2 ahead of the previous kernel's end
  int pair_boxes;     // the 4-D tensor maps exist: a whole 128-key tile of a contiguous cache is one copy
  int tiles;          // row tiles per (sequence, kv head)
  int groups;         // blocks along the rows: tiles, or pairs of tiles (kRows2)
  int splits;         // blocks along the key axis = cluster size
  float scale_log2;
  long long wait_limit;   // SM cycles a bounded wait may last
  unsigned* tickets;      // per sequence: the word of seq_status.cuh; zero between calls
  int blocks_per_seq;
  int tile_nodes;         // whole nodes of a row tile
  Divisor by_splits, by_groups, by_kv_heads, by_group_heads;
};

struct Maps {
  CUtensorMap q, out;    // [B][N][Hq][128], box = 64 x G x 128/G nodes
  CUtensorMap kc, vc;    // cache rows, box = 64 x 1 head x 64 rows
  CUtensorMap kt, vt;    // tree rows, likewise
  CUtensorMap kc2, vc2;  // cache rows as [head][half of d][row][64], box = a whole key tile
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(c)));
  return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("mul.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
  return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
  return d;
}
// Natural log-sum-exp of a row from its reference (in base 2) and its sum, in effect rounded once: the
// sum is taken apart into 2^e * f, so that the logarithm is below 1, and ref + e keeps its remainder
// (Knuth's two-sum).  (Base 2 with a product at the end has two roundings of the size of this one.)
__device__ __forceinline__ float log_sum_exp(float ref, float total) {
  if (!(total > 0.f && total < INFINITY)) return total > 0.f ? ref + total : total == 0.f ? ref : total;   // no key: ref is -inf
  constexpr float kLn2 = 0x1.62e43p-1f, kLn2Rest = -0x1.05c61p-29f;
  const uint32_t u = __float_as_uint(total);
  const float e = (float)((int)(u >> 23) - 127), f = __uint_as_float((u & 0x007FFFFFu) | 0x3F800000u);
  const float x = __fadd_rn(ref, e), part = __fsub_rn(x, ref);
  const float rest = __fadd_rn(__fsub_rn(ref, __fsub_rn(x, part)), __fsub_rn(e, part));
  return fmaf(x, kLn2, fmaf(rest, kLn2, fmaf(x, kLn2Rest, logf(f))));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float2 half2_bits_to_float2(uint32_t u) {
  return __half22float2(*reinterpret_cast<const __half2*>(&u));
}
__device__ __forceinline__ void named_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
template <int kRegs>
__device__ __forceinline__ void more_registers() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegs)); }
template <int kRegs>
__device__ __forceinline__ void fewer_registers() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegs)); }
// Relaxed: the two arrivals say that shared memory may be overwritten or left, which needs no writes of
// this block to be visible to another (a release waits for all of them, here and with the divisions below:
// 11.2 -> 9.5 us for one sequence of 16 nodes and 512 keys).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// bulk copy to a peer's shared memory; its barrier counts the bytes
__device__ __forceinline__ void bulk_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "r"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* tm, uint32_t src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];"
               ::"l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(src)
               : "memory");
}
__device__ __forceinline__ void st_shared16(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ float4 ld_shared16(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_shared4(uint32_t a, uint32_t x) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(x) : "memory"); }
__device__ __forceinline__ void st_shared8(uint32_t a, float x, float y) {
  asm volatile("st.shared.v2.f32 [%0], {%1,%2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ uint32_t ld_shared4(uint32_t a) {
  uint32_t x;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x) : "r"(a) : "memory");
  return x;
}
__device__ __forceinline__ uint2 ld_shared8(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
  return v;
}

// a position in the ring of stages and the parity of its current round
template <int NST>
struct RingPos {
  int idx;
  uint32_t ph;
  __device__ __forceinline__ explicit RingPos(int n) : idx(n % NST), ph((uint32_t)(n / NST) & 1u) {}   // of load n
  __device__ __forceinline__ void advance(int k) {
    idx += k;
    if (idx >= NST) { idx -= NST; ph ^= 1u; }
  }
};

// What a thread knows about its block: its place in the grid, its share of the key axis, its row.
template <bool kRows2, int kParts>
struct Block {
  uint8_t* smem;
  uint32_t smem0, sRing, bar0, tmem;
  volatile int* abort_flag;
  int tid, warp, lane;
  int CS, split, group, kvh, b;            // cluster size, rank in the cluster, rows' group, kv head, sequence
  int N, G, tile_nodes, RT, tile0, users;  // whole nodes of a row tile and the rows they take; first row tile; slots that read one K/V tile
  int R, per, first, mine;                 // rows in use, numbered through the row tiles; rank d finalises [d * per, (d + 1) * per)
  int L, p_cache, p_total, pc_begin, pc_end, T, t_plain;
  bool len_bad;
  int slot, row, part, node_in_tile, node, my_tiles;     // of the softmax threads: accumulator row, share of a tile's keys
  bool row_valid;
  uint32_t lane_addr;

  __device__ __forceinline__ Misc& misc() const { return *reinterpret_cast<Misc*>(smem + kMiscAt); }
  __device__ __forceinline__ uint32_t bar(int idx) const { return bar0 + 8u * (uint32_t)idx; }
  __device__ __forceinline__ uint32_t tmem_S(int s) const { return tmem + (uint32_t)(s * BN); }   // P overwrites columns 0-63
  __device__ __forceinline__ uint32_t tmem_O(int s) const { return tmem + (uint32_t)(2 * BN + s * HD); }
  // real keys of piece g (0: not of this block)
  __device__ __forceinline__ int piece_keys(int g) const {
    return g >= pc_end ? 0 : g < p_cache ? min(PG, L - g * PG) : min(PG, N - (g - p_cache) * PG);
  }
  __device__ __forceinline__ int slot_tiles(int s) const { return kRows2 ? (s < users ? T : 0) : (T - s + 1) / 2; }

  // the place in the grid (blocks of a cluster are neighbours along x)
  __device__ __forceinline__ void place(const Params& p, uint8_t* sm, unsigned block, int thread) {
    smem = sm;
    smem0 = smem_u32(sm);
    sRing = smem0 + Cfg<kRows2, kParts>::kQ * kQTile;
    bar0 = smem_u32(&misc().bar[0]);
    abort_flag = &misc().abort_flag;
    tid = thread; warp = tid >> 5; lane = tid & 31;
    CS = p.splits;
    const unsigned cluster_id = p.by_splits.divide(block), unit = p.by_groups.divide(cluster_id);
    split = (int)(block - cluster_id * (unsigned)CS);
    group = (int)(cluster_id - unit * (unsigned)p.groups);
    b = (int)p.by_kv_heads.divide(unit);
    kvh = (int)unit - b * p.Hkv;
    N = p.N; G = p.G;
    tile_nodes = p.tile_nodes; RT = tile_nodes * G;
    tile0 = kRows2 ? 2 * group : group;
    users = (kRows2 && tile0 + 1 < p.tiles) ? 2 : 1;
    R = (kRows2 ? (users - 1) * BM : 0) + min(RT, (N - (tile0 + users - 1) * tile_nodes) * G);
    per = ((int)p.by_splits.divide((unsigned)(R + CS - 1)) + 7) & ~7;
    first = min(R, split * per);
    mine = min(R, first + per) - first;
  }
  // The sequence's length and this block's range of the key axis.  The axis is cut in 64-key pieces:
  // p_cache pieces of context, then the tree's own pieces.  A split takes a contiguous range of pieces
  // and walks it in tiles of two; the last tile of a range may hold one piece only.  A bad length
  // reads the tree's own rows only.  Tiles [0, t_plain) consist of two complete pieces of context.
  __device__ __forceinline__ void range(const Params& p, int len) {
    L = len;
    len_bad = (L < 0) || (p.paged ? (pieces_of(L) > p.max_pages) : (L > p.cap_tokens));
    p_cache = len_bad ? 0 : pieces_of(L);
    p_total = p_cache + pieces_of(N);
    pc_begin = (int)p.by_splits.divide((unsigned)split * (unsigned)p_total);
    pc_end = (int)p.by_splits.divide((unsigned)(split + 1) * (unsigned)p_total);
    T = (pc_end - pc_begin + 1) / 2;
    t_plain = max(0, (min(pc_end, len_bad ? 0 : L / PG) - pc_begin) / 2);
    tmem = misc().tmem;
    slot = (warp >> 2) & 1;
    row = (warp & 3) * 32 + lane;   // a warp may touch the 32 tensor-memory lanes of its number modulo 4
    lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const int rtile = kRows2 ? tile0 + slot : tile0;
    part = row / Cfg<kRows2, kParts>::kRows;
    const int tile_row = row % Cfg<kRows2, kParts>::kRows;
    node_in_tile = (int)p.by_group_heads.divide((unsigned)tile_row);
    node = rtile * tile_nodes + node_in_tile;
    row_valid = warp < kSoftmaxWarps && tile_row < RT && rtile < p.tiles && node < N;
    my_tiles = slot_tiles(slot);
  }
};

// ---- the roles' work on the block's share of the keys

// A tile's P is handed over in parts: keys 0-95, 96-127 if a thread has all keys of its row, else
// the first and the second 32 of every thread's, or all at once.
template <int kParts>
__host__ __device__ constexpr int hand_overs() { return kParts <= 2 ? 2 : 1; }
template <int kParts>
__host__ __device__ constexpr int handed_over_in(int c) { return kParts == 1 ? (c < 3 ? 0 : 1) : kParts == 2 ? (c & 1) : 0; }   // 32 keys c

// Q needs nothing that is read from memory, so it is asked for ahead of the context length.
template <bool kRows2, int kParts>
__device__ __forceinline__ void load_q(const Block<kRows2, kParts>& k, const Maps& tm) {
  mbar_expect_tx(k.bar(B_Q), (uint32_t)(k.users * kParts * k.RT * HD * 2));   // a box holds RT rows, absent nodes as zeros
#pragma unroll
  for (int m = 0; m < Cfg<kRows2, kParts>::kQ * kParts; ++m) {
    if (kRows2 && m >= k.users) break;
    const uint32_t dst = k.smem0 + (uint32_t)m * (kRows2 ? kQTile : kQTile / 2 / kParts);
    const int node0 = (k.tile0 + (kRows2 ? m : 0)) * k.tile_nodes;
    tma_load_4d(dst, &tm.q, 0, k.kvh * k.G, node0, k.b, k.bar(B_Q));
    tma_load_4d(dst + kQTile / 2, &tm.q, 64, k.kvh * k.G, node0, k.b, k.bar(B_Q));
  }
}

// Ahead of the previous kernel's end, by an idle warp: the block's first key tiles of context are asked for into L2, a lane
// per piece.  Length and block table are read as hints (an earlier kernel may still be writing them): whatever they say,
// the addresses are in range, and what is loaded in the end goes by what they say then.  For the short variants, whose
// loads would otherwise start from nothing when the previous grid is gone (1 x 64 nodes x 2048 keys, whole step: 20.5 -> 18.9
// us; 32 layers of 1 x 60 x 1500 and LM head: 450 -> 432; with three tiles 1 % less, with four or eight 2; attention behind a
// kernel that is not launched ahead of its end: 15.2 -> 14.9).  The other variants lost: where their loop is bound by the
// tensor core, or the memory is busy anyway, it is traffic in the way (one tile, 32 layers of 4 x 64 x 4096: 985 -> 995;
// 32 x 32 paged: 137.4 -> 138.4).
constexpr int kAhead = 2;
constexpr int kAheadFrom = 3;   // key tiles of a block, by the bound of the lengths: with fewer there is nothing to gain
template <bool kRows2, int kParts>
__device__ __forceinline__ void scout(const Block<kRows2, kParts>& k, const Maps& tm, const Params& p) {
  const int len = max(0, ld_hint(p.ctx_len + k.b));
  const int p_cache = p.paged ? min(pieces_of(len), p.max_pages) : pieces_of(min(len, p.cap_tokens)), p_total = p_cache + pieces_of(k.N);
  const int begin = (int)p.by_splits.divide((unsigned)k.split * (unsigned)p_total);
  const int end = min(min(p_cache, begin + 2 * kAhead), (int)p.by_splits.divide((unsigned)(k.split + 1) * (unsigned)p_total));
  for (int g = begin + k.lane; g < end; g += 32) {
    int row = k.b * p.cap_tokens + g * PG;
    if (p.paged) {
      const int pg = ld_hint(p.block_table + (int64_t)k.b * p.max_pages + g);
      if (pg < 0 || pg >= p.n_pages) continue;
      row = pg * PG;
    }
    tma_prefetch_3d(&tm.kc, 0, k.kvh, row);
    tma_prefetch_3d(&tm.kc, 64, k.kvh, row);
    tma_prefetch_3d(&tm.vc, 0, k.kvh, row);
    tma_prefetch_3d(&tm.vc, 64, k.kvh, row);
  }
  __syncwarp();
}

template <bool kRows2, int kParts>
__device__ __forceinline__ void produce(const Block<kRows2, kParts>& k, const Maps& tm, const Params& p) {
  constexpr int NST = Cfg<kRows2, kParts>::NST;
  if (k.T == 0) mbar_drain(k.bar(B_Q), 0);   // nobody else waits for the Q that is on its way
  int page = 0, page_base = -64;   // lane j: pool page of context piece (page_base + j)
  RingPos<NST> pos(0);
  int issued = 0;
  bool ok = true;
  for (int t = 0; t < k.T && ok; ++t) {
    const int g0 = k.pc_begin + 2 * t;
    if (p.paged && g0 < k.p_cache && g0 + 2 > page_base + 32) {
      page_base = g0;
      const int pc = g0 + k.lane;
      page = (pc < k.p_cache) ? p.block_table[(int64_t)k.b * p.max_pages + pc] : 0;
    }
    int row0[2];
    bool is_tree[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int g = g0 + j;
      int pg = __shfl_sync(0xFFFFFFFFu, page, (g - page_base) & 31);
      is_tree[j] = g >= k.p_cache;
      if (g >= k.pc_end) row0[j] = -1;     // the range ended inside this tile
      else if (is_tree[j]) row0[j] = k.b * k.N + (g - k.p_cache) * PG;
      else if (p.paged) {
        if (pg < 0 || pg >= p.n_pages) pg = 0;   // the reporter flags the sequence; any page will do
        row0[j] = pg * PG;
      } else row0[j] = k.b * p.cap_tokens + g * PG;
    }
#pragma unroll
    for (int kv = 0; kv < 2; ++kv) {   // K, then V
      if (issued >= NST) ok = wait_warp(k.bar(B_EMPTY + pos.idx), pos.ph ^ 1u, k.abort_flag, p.wait_limit);
      if (!ok) break;
      if (k.lane == 0) {
        const uint32_t full = k.bar(B_FULL + pos.idx), stage = k.sRing + (uint32_t)pos.idx * kStage;
        if (p.pair_boxes && row0[0] >= 0 && !is_tree[1] && row0[1] == row0[0] + PG) {
          // both pieces are neighbours in the cache: the whole tile, both halves of d, in one copy
          mbar_expect_tx(full, kStage);
          tma_load_4d(stage, kv == 0 ? &tm.kc2 : &tm.vc2, 0, row0[0], 0, k.kvh, full);
        } else {
          mbar_expect_tx(full, (row0[1] >= 0 ? 2u : 1u) * 2u * kPiece);
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            if (row0[j] < 0) continue;
            const CUtensorMap* m = is_tree[j] ? (kv == 0 ? &tm.kt : &tm.vt) : (kv == 0 ? &tm.kc : &tm.vc);
            const uint32_t dst = stage + (uint32_t)j * kPiece;
            tma_load_3d(dst, m, 0, k.kvh, row0[j], full);
            tma_load_3d(dst + kHalf, m, 64, k.kvh, row0[j], full);
          }
        }
      }
      ++issued;
      pos.advance(1);
    }
  }
  if (k.lane == 0) k.misc().issued = issued;   // for the drain of an aborted block
}

// The whole warp walks the schedule and one elected lane issues: inside a divergent branch every
// operand is moved to the uniform registers for each MMA, and an MMA of 64 cycles took 110 to 200 to
// issue (long contexts, 8 x 32768 keys: 1090 -> 740 us for the branch under elect.sync alone).  Fixed
// order: Q K^T of both slots, then per tile and slot P V of the tile's parts as they are handed over and
// Q K^T of the slot's next tile.  The tensor core queues a few MMAs, so what lies between two groups
// of them is hidden.
template <bool kRows2, int kParts>
__device__ __forceinline__ void issue(const Block<kRows2, kParts>& k, const Params& p) {
  constexpr int NST = Cfg<kRows2, kParts>::NST;
  const uint32_t el = elect_one();
  if (k.T == 0 || !wait_warp(k.bar(B_Q), 0, k.abort_flag, p.wait_limit)) return;
  const uint64_t q_desc = smem_desc(k.smem0, 16, 1024);
  const uint64_t k_desc = smem_desc(k.sRing, 16, 1024);
  const uint64_t v_desc = smem_desc(k.sRing, kHalf, 1024);   // lbo: the other half of d
  RingPos<NST> kpos[2] = {RingPos<NST>(0), RingPos<NST>(kRows2 ? 0 : 2)};
  uint32_t ph = 0u;   // bit 2 s + h: parity of the next use of the barrier for part h of slot s's P
  auto issue_qk = [&](int s) -> bool {
    if (!wait_warp(k.bar(B_FULL + kpos[s].idx), kpos[s].ph, k.abort_flag, p.wait_limit)) return false;
    tc_fence_after();
    const uint64_t qd = q_desc + (uint64_t)(((kRows2 ? s : 0) * kQTile) >> 4);
    const uint64_t kd = k_desc + (uint64_t)((uint32_t)(kpos[s].idx * (int)kStage) >> 4);
#pragma unroll
    for (int ks = 0; ks < HD / 16; ++ks) {
      const uint32_t qo = (ks >> 2) * (kQTile / 2) + (ks & 3) * 32;
      const uint32_t ko = (ks >> 2) * kHalf + (ks & 3) * 32;
      umma_bf16_if(el, k.tmem_S(s), qd + (qo >> 4), kd + (ko >> 4), kIdescQK, ks > 0 ? 1u : 0u);
    }
    umma_commit_if(el, k.bar(B_S + s));
    umma_commit_if(el, k.bar(B_EMPTY + kpos[s].idx));
    return true;
  };
  bool ok = issue_qk(0);
  if (ok && k.slot_tiles(1) > 0) ok = issue_qk(1);
#pragma unroll 1
  for (int r = 0; r < k.slot_tiles(0) && ok; ++r) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (!ok || r >= k.slot_tiles(s)) continue;
      const int g0 = k.pc_begin + 2 * (kRows2 ? r : 2 * r + s);
      RingPos<NST> vpos = kpos[s];
      vpos.advance(1);
      ok = wait_warp(k.bar(B_FULL + vpos.idx), vpos.ph, k.abort_flag, p.wait_limit);
      const uint64_t vd = v_desc + (uint64_t)((uint32_t)(vpos.idx * (int)kStage) >> 4);
      const int keys[2] = {k.piece_keys(g0), k.piece_keys(g0 + 1)};
#pragma unroll
      for (int h = 0; h < hand_overs<kParts>(); ++h) {
        if (!ok || (kParts == 1 && h > 0 && keys[1] <= CH)) continue;
        ok = wait_warp(k.bar(B_P + 2 * s + h), (ph >> (2 * s + h)) & 1u, k.abort_flag, p.wait_limit);
        if (!ok) continue;
        ph ^= 1u << (2 * s + h);
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < BN / CH; ++c) {
          if (handed_over_in<kParts>(c) != h || keys[c >> 1] <= (c & 1) * CH) continue;
#pragma unroll
          for (int kk = 2 * c; kk < 2 * c + 2; ++kk)
            umma_bf16_ts_if(el, k.tmem_O(s), k.tmem_S(s) + (uint32_t)(kk * 8), vd + (uint64_t)((kk * 16 * 128) >> 4), kIdescPV,
                            (r > 0 || kk > 0) ? 1u : 0u);
        }
      }
      if (!ok) continue;
      umma_commit_if(el, k.bar(B_EMPTY + vpos.idx));
      kpos[s].advance(Cfg<kRows2, kParts>::kStep);
      if (r + 1 < k.slot_tiles(s)) ok = issue_qk(s);
      else umma_commit_if(el, k.bar(B_LAST + s));
    }
  }
}

// By an idle warp, meanwhile: what the merge needs to know, so that nothing but shared memory is read ahead of its copies.
// Two neighbouring stages of the ring receive and a third holds this block's own sums: any but those of the last V tiles.
template <bool kRows2, int kParts>
__device__ __forceinline__ void note_place(const Block<kRows2, kParts>& k, const Params& p) {
  constexpr int NST = Cfg<kRows2, kParts>::NST;
  Place& at = k.misc().place;
  if (k.lane < kMaxSplits) {   // other ranks write there, so the place is a function of the receiver's number of tiles
    const unsigned d = min((unsigned)k.lane, (unsigned)k.CS - 1u);
    const int tiles_of_rank = ((int)(p.by_splits.divide((d + 1u) * (unsigned)k.p_total) - p.by_splits.divide(d * (unsigned)k.p_total)) + 1) / 2;
    const int i = (2 * tiles_of_rank) % NST, idx = i == NST - 1 ? 0 : i;
    at.rx[k.lane] = (uint32_t)idx * kStage;
    if ((int)d == k.split) at.meta = (uint32_t)((idx + 2) % NST) * kStage;
  }
  if (k.lane == 0) {
    at.b = k.b; at.split = k.split; at.kvh = k.kvh;
    at.users = k.users; at.T = k.T; at.R = k.R; at.per = k.per;
    at.first = k.first; at.mine = k.mine; at.tile0 = k.tile0; at.CS = k.CS;
    at.N = k.N; at.G = k.G; at.Hq = p.Hq; at.tile_nodes = k.tile_nodes;
    at.tiles = p.tiles; at.group_d = (int)p.by_group_heads.d; at.group_m = p.by_group_heads.m;
    at.out = p.out; at.lse = p.lse;
  }
}

template <bool kRows2, int kParts>
__device__ __forceinline__ void softmax(const Block<kRows2, kParts>& k, const Params& p, int par) {
  constexpr int NST = Cfg<kRows2, kParts>::NST;
  Misc& ms = k.misc();
  const int tid = k.tid, lane = k.lane, slot = k.slot, row = k.row;
  if (tid < CLV_MAX_NODES) {
    bool bad = false;
    if (par < -1 || par >= tid) { bad = true; par = -1; }
    ms.parent[tid] = (signed char)par;
    // one block per sequence reports what is wrong with it: the length, the tree, the block table
    if (k.group == 0 && k.split == 0 && k.kvh == 0) {
      bad |= k.len_bad;
      if (p.paged && k.warp == 0)
        for (int pg = lane; pg < k.p_cache; pg += 32) {
          const int e = p.block_table[(int64_t)k.b * p.max_pages + pg];
          bad |= (e < 0 || e >= p.n_pages);
        }
      if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) {
        atomicOr(p.tickets + 2 * k.b + 1, 1u);
        __threadfence();   // before this block's ticket
      }
    }
  }
  __syncwarp();
  named_barrier(1, 32 * kSoftmaxWarps);
  uint32_t anc[4] = {0u, 0u, 0u, 0u};   // row of the tree's topology matrix: the node and its ancestors
  if (k.row_valid) {
    for (int j = k.node; j >= 0; j = ms.parent[j]) {
#pragma unroll
      for (int w = 0; w < 4; ++w) anc[w] |= (j >> 5) == w ? 1u << (j & 31) : 0u;
    }
  }
  __syncwarp();
  const bool warp_active = __any_sync(0xFFFFFFFFu, k.row_valid);
  const uint32_t s_addr = k.tmem_S(slot) + k.lane_addr;   // this row's scores, then its P
  const float sc = p.scale_log2;
  float m_ref = k.row_valid ? -INFINITY : 0.f, l_run = 0.f;
  auto hand_over = [&](int h) {   // part h of P
    tmem_wait_st();
    tc_fence_before();
    __syncwarp();
    mbar_arrive_if(lane == 0 ? 1u : 0u, k.bar(B_P + 2 * slot + h));
  };
  RingPos<NST> vpos(kRows2 || slot == 0 ? 1 : 3);   // V stage of the current tile
#pragma unroll 1
  for (int r = 0; r < k.my_tiles; ++r) {
    const int t = kRows2 ? r : 2 * r + slot;
    if (!wait_warp(k.bar(B_S + slot), (uint32_t)r & 1u, k.abort_flag, p.wait_limit)) break;
    tc_fence_after();
    int keys0 = PG, keys1 = PG;    // real keys of the tile's pieces
    const bool plain = t < k.t_plain;
    if (!plain) {
      keys0 = k.piece_keys(k.pc_begin + 2 * t);
      keys1 = k.piece_keys(k.pc_begin + 2 * t + 1);
      // Rows of V beyond a piece's real keys hold whatever lies behind them in memory; their
      // probabilities are exactly 0, but 0 * NaN would poison O: clear them, up to the end of the
      // last 32 keys that P V takes.
      if ((keys0 | keys1) & (CH - 1)) {
        if (!wait_warp(k.bar(B_FULL + vpos.idx), vpos.ph, k.abort_flag, p.wait_limit)) break;
        uint8_t* vt = k.smem + (k.sRing - k.smem0) + (uint32_t)vpos.idx * kStage;
#pragma unroll 1
        for (int j = 0; j < 2; ++j) {
          const int v = j ? keys1 : keys0;
          const int n = ((v + CH - 1) & ~(CH - 1)) - v;
          for (int i = row; i < n * 16; i += BM) {
            const int vr = j * PG + v + (i >> 4), chk = i & 15;
            *reinterpret_cast<uint4*>(vt + (chk >> 3) * kHalf + vr * 128 + (chk & 7) * 16) = make_uint4(0, 0, 0, 0);
          }
        }
        fence_async_smem();   // cleared V rows visible to the tensor core's reads
        __syncwarp();
      }
    }
    vpos.advance(Cfg<kRows2, kParts>::kStep);
    if (kParts == 1 && !warp_active) {   // no row of this warp exists: its lanes of P may hold anything
      hand_over(0);
      if (keys1 > CH) hand_over(1);
      continue;
    }
    const bool masked = !plain;   // rows that do not exist compute what nobody reads
    auto mask = [&](int c, uint32_t (&a)[CH]) {   // columns that this row may not see become -inf
      const int g = k.pc_begin + 2 * t + (c >> 1), keys = ((c >> 1) ? keys1 : keys0) - (c & 1) * CH;
      uint32_t bits = 0u;
      if (k.row_valid && keys > 0) {
        if (g < k.p_cache) bits = keys >= CH ? 0xFFFFFFFFu : (1u << keys) - 1u;
        else bits = g == k.p_cache ? ((c & 1) ? anc[1] : anc[0]) : ((c & 1) ? anc[3] : anc[2]);
      }
#pragma unroll
      for (int j = 0; j < CH; ++j)
        if (!((bits >> j) & 1u)) a[j] = 0xFF800000u;
    };
    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
    auto take_max = [&](const uint32_t (&a)[CH]) {
#pragma unroll
      for (int j = 0; j < CH; j += 2) mx[(j >> 1) & 3] = max3(mx[(j >> 1) & 3], __uint_as_float(a[j]), __uint_as_float(a[j + 1]));
    };
    float2 sum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    float neg_m = m_ref == -INFINITY ? 0.f : -m_ref;
    auto exps = [&](uint32_t (&a)[CH]) {   // the first half of `a` becomes P
      const float2 sc2 = make_float2(sc, sc), nm2 = make_float2(neg_m, neg_m);
#pragma unroll
      for (int j = 0; j < CH / 2; ++j) {
        const float2 e = fma2(make_float2(__uint_as_float(a[2 * j]), __uint_as_float(a[2 * j + 1])), sc2, nm2);
        const float2 pr = make_float2(ex2(e.x), ex2(e.y));
        sum[j & 1] = add2(sum[j & 1], pr);
        a[j] = pack_bf16(pr.x, pr.y);
      }
    };
    auto new_reference = [&](float m_new, bool need) {   // O is at rest: these scores were asked for after P V of the slot's previous tile
      const float alpha = need ? ex2(m_ref - m_new) : 1.f;   // ex2(-inf) = 0
      if (need) { m_ref = m_new; l_run *= alpha; }
      neg_m = m_ref == -INFINITY ? 0.f : -m_ref;
      if (r > 0) {
#pragma unroll 1
        for (int cc = 0; cc < HD; cc += 16) {
          uint32_t ov[16];
          tmem_ld_x16(k.tmem_O(slot) + k.lane_addr + (uint32_t)cc, ov);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 16; ++j) ov[j] = __float_as_uint(__uint_as_float(ov[j]) * alpha);
          tmem_st_x16(k.tmem_O(slot) + k.lane_addr + (uint32_t)cc, ov);
        }
      }
    };
    auto load = [&](int c, uint32_t (&a)[CH]) { tmem_ld_x32(s_addr + (uint32_t)(c * CH), a); };
    auto store_p = [&](int c, const uint32_t (&a)[CH]) {
      tmem_st_x16(s_addr + (uint32_t)(c * (CH / 2)), *reinterpret_cast<const uint32_t(*)[CH / 2]>(&a[0]));
    };
    if constexpr (kParts > 1) {   // one or two loads' worth of keys
      constexpr int kLoads = 4 / kParts;
      const int c0 = k.part * kLoads;
      uint32_t x[kLoads][CH];
#pragma unroll
      for (int c = 0; c < kLoads; ++c) load(c0 + c, x[c]);
      tmem_wait_ld();
      {
        uint32_t none[CH / 2];
#pragma unroll
        for (int j = 0; j < CH / 2; ++j) none[j] = 0u;
#pragma unroll
        for (int c = kLoads; c < 4; ++c) tmem_st_x16(s_addr + (uint32_t)(((c0 + c) & 3) * (CH / 2)), none);   // the other parts' keys
      }
#pragma unroll
      for (int c = 0; c < kLoads; ++c) {
        if (masked) mask(c0 + c, x[c]);
        take_max(x[c]);
      }
      const float m_new = fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]) * sc;
      const bool need = m_new > m_ref + kRefSlack;
      if (__any_sync(0xFFFFFFFFu, need)) new_reference(m_new, need);
#pragma unroll
      for (int c = 0; c < kLoads; ++c) {
        exps(x[c]);
        store_p(c0 + c, x[c]);
        hand_over(c);
      }
      const float2 tot = add2(sum[0], sum[1]);
      l_run += tot.x + tot.y;
      continue;
    }
    uint32_t x0[CH], x1[CH], x2[CH], x3[CH];
    load(0, x0);
    tmem_wait_ld();
    load(1, x1);
    load(2, x2);
    load(3, x3);
    if (masked) mask(0, x0);
    exps(x0);
    tmem_wait_ld();
    if (masked) {
      mask(1, x1);
      mask(2, x2);
      mask(3, x3);
    }
    take_max(x2);
    take_max(x3);
    exps(x1);
    float m_new = fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]) * sc;   // scale > 0; no allowed key: -inf
    const float s01 = (sum[0].x + sum[0].y) + (sum[1].x + sum[1].y);   // no less than the largest of its 64 terms
    bool need = s01 > kTopP || m_new > m_ref + kRefSlack || m_ref == -INFINITY;
    if (__any_sync(0xFFFFFFFFu, need)) {
      load(0, x0);   // the scores of the first 64 keys are still in place
      load(1, x1);
      tmem_wait_ld();
      if (masked) {
        mask(0, x0);
        mask(1, x1);
      }
      take_max(x0);
      take_max(x1);
      m_new = fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]) * sc;
      need = need && m_new > m_ref;
      new_reference(m_new, need);
      sum[0] = sum[1] = make_float2(0.f, 0.f);
      exps(x0);
      exps(x1);
    }
    store_p(0, x0);
    store_p(1, x1);
    if (keys1 > CH) {
      exps(x2);
      store_p(2, x2);
      hand_over(0);
      exps(x3);
      store_p(3, x3);
      hand_over(1);
    } else if (keys1 > 0) {
      exps(x2);
      store_p(2, x2);
      hand_over(0);
    } else {
      hand_over(0);
    }
    const float2 tot = add2(sum[0], sum[1]);
    l_run += tot.x + tot.y;
  }
  ms.ml[slot * BM + row] = make_float2(m_ref, l_run);
}

// The words of a sequence for seq_status.cuh.  The wait for its publisher outlasts the publisher's own.
struct TallyWords {
  unsigned long long* tally;
  int32_t* status;
  long long wait_limit, since = 0;
  __device__ __forceinline__ unsigned long long add(unsigned long long v) { return atomicAdd(tally, v); }
  __device__ __forceinline__ unsigned count() { return *reinterpret_cast<volatile unsigned*>(tally); }
  __device__ __forceinline__ void clear() { *const_cast<volatile unsigned long long*>(tally) = 0ull; }
  __device__ __forceinline__ void put(int s) { *const_cast<volatile int32_t*>(status) = s; }
  __device__ __forceinline__ void fence() { __threadfence(); }
  __device__ __forceinline__ void correct() { atomicCAS(status, CLV_OK, CLV_ERR_TIMEOUT); }
  __device__ __forceinline__ bool expired() {
    const long long now = clock64();
    if (since == 0) since = now;
    return now - since > wait_limit + kWaitLimitCycles;
  }
};

// ------------------------------------------------------------------------------------ kernel
// kOneBlock: of the variants with several threads per row, the one for a block that is not part of a cluster
// (the code of neither case lies in the other's way: 1 x 16 nodes x 512 keys took 0.13 us longer in one kernel).
template <bool kRows2, int kParts, bool kOneBlock>
__global__ void __launch_bounds__(kThreads, 1) tree_attn_kernel(const __grid_constant__ Maps tm, const __grid_constant__ Params p) {
  constexpr int NST = Cfg<kRows2, kParts>::NST;
  extern __shared__ __align__(1024) uint8_t smem[];
  Misc& ms = *reinterpret_cast<Misc*>(smem + kMiscAt);
  {
  Block<kRows2, kParts> k;
  k.place(p, smem, blockIdx.x, threadIdx.x);
  const int tid = k.tid, warp = k.warp;
  auto bar = [&](int idx) { return k.bar(idx); };

  // ---- set-up that reads no global memory: barriers, tensor memory, descriptor prefetch.  The
  //      kernel is launched with programmatic stream serialisation, so this part may run while the
  //      previous kernel of the stream drains.
  if (tid == 0) {
    for (int i = 0; i < NST; ++i) { mbar_init(bar(B_FULL + i), 1); mbar_init(bar(B_EMPTY + i), (uint32_t)k.users); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar(B_S + i), 1); mbar_init(bar(B_LAST + i), 1); }
    for (int i = 0; i < 4; ++i) mbar_init(bar(B_P + i), 4);
    mbar_init(bar(B_Q), 1);
    mbar_init(bar(B_RX), 1);
    mbar_init(bar(B_DR), 1);
    if (kParts > 1 ? !kOneBlock : k.CS > 1) mbar_expect_tx(bar(B_RX), (uint32_t)((k.CS - 1) * kParts * k.mine) * kRowBytes<kRows2>);   // what the other ranks will send
    ms.abort_flag = 0;
    ms.late_flag = 0;
    ms.issued = 0;
    fence_barrier_init();
    fence_async_smem();
  }
  if (warp == kIssuer) tmem_alloc(smem_u32(&ms.tmem), kTmemCols);
  if (tid == 32 * kProducer) {
    tma_prefetch_desc(&tm.q);
    if (p.pair_boxes) { tma_prefetch_desc(&tm.kc2); tma_prefetch_desc(&tm.vc2); }
    tma_prefetch_desc(&tm.kc); tma_prefetch_desc(&tm.vc);
    tma_prefetch_desc(&tm.kt); tma_prefetch_desc(&tm.vt);
  }
  tc_fence_before();
  if (kParts > 1 && p.ask_ahead && warp == kScout) scout(k, tm, p);
  __syncthreads();
  tc_fence_after();
  cudaGridDependencySynchronize();

  if (p.longest_first) {
    // More blocks than SMs and contexts of different lengths (ragged batch): hand the sequences
    // out longest first, so that the block scheduler packs the short ones into the gaps.  Block
    // group `b` takes the sequence whose length has rank b (ties by index).
    int* len = reinterpret_cast<int*>(smem);   // the tiles are not in use yet
    for (int i = tid; i < p.B; i += kThreads) len[i] = p.ctx_len[i];
    __syncthreads();
    for (int i = tid; i < p.B; i += kThreads) {
      const int Li = len[i];
      int rank = 0;
      for (int j = 0; j < p.B; ++j) rank += (len[j] > Li) || (len[j] == Li && j < i);
      if (rank == k.b) ms.seq = i;
    }
    __syncthreads();
    k.b = ms.seq;
    fence_async_smem();   // the tiles are written by TMA next
    __syncthreads();
  }
  // what the block reads of global memory before its tiles: all under way at once
  if (tid == 32 * kProducer) load_q<kRows2, kParts>(k, tm);
  __syncwarp();
  const int par = tid < k.N ? p.parent[(int64_t)k.b * k.N + tid] : -1;   // of node tid
  k.range(p, p.ctx_len[k.b]);
  if (warp == kWriter) note_place(k, p);
  if (warp < kSoftmaxWarps) {
    more_registers<kSoftmaxRegs>();
    softmax<kRows2, kParts>(k, p, par);
    __syncwarp();
    fewer_registers<kLaunchRegs>();   // before the third warpgroup takes its own back
    named_barrier(2, kThreads);
  } else {
    fewer_registers<kOtherRegs>();
    if (warp == kProducer) produce<kRows2, kParts>(k, tm, p);
    else if (warp == kIssuer) issue<kRows2, kParts>(k, p);
    __syncwarp();
    named_barrier(2, kThreads);
    more_registers<kLaunchRegs>();
  }
  }

  // ---- every role has met here ------------------------------------------------------------------
  // What follows runs once per block, from a cold instruction cache, and that is what it takes its time by: compact
  // loops, few instructions ahead of the copies.  What is known about the block comes from shared memory: kept in
  // registers it would push the softmax threads' scores out of theirs (4 x 64 nodes x 4096 keys: 29.8 -> 27.7 us), and
  // worked out once more it took 570 cycles instead of 90.
  const Place& at = ms.place;
  int tid;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
  const int warp = tid >> 5, lane = tid & 31, CS = at.CS, split = at.split, users = at.users, b = at.b, T = at.T;
  const int R = at.R, per = at.per, first = at.first, mine = at.mine;
  const uint32_t smem0 = smem_u32(smem), sRing = smem0 + Cfg<kRows2, kParts>::kQ * kQTile, tmem = ms.tmem;
  auto bar = [&](int idx) { return smem_u32(&ms.bar[0]) + 8u * (uint32_t)idx; };
  // Calls this short lose a tenth of their time between two launches.  The next kernel may be set up on the
  // SMs that this grid leaves idle or has left, and waits for this grid's results itself (32 layers of
  // 1 x 60 nodes x 1500 keys and LM head, in a loop: 486 -> 470 us).  The other variants do not: what follows a long call is a
  // stream over the logits at full occupancy, whose blocks then pile up on the idle SMs (4 x 64 nodes x
  // 4096 keys with 256 rows of logits: 44.7 -> 45.9 us).
  if (kParts > 1) cudaTriggerProgrammaticLaunchCompletion();
  const bool clustered = kParts > 1 ? !kOneBlock : CS > 1;
  const bool alone = kParts == 1 && !clustered;   // nothing to be added to this block's accumulators
  const bool aborted = *const_cast<volatile int*>(&ms.abort_flag) != 0;
  if (clustered) cluster_arrive();   // all Q K^T of this block are done: what the merge uses is idle (see there)
  if (aborted) {
    // copies that were issued land on their own, MMAs that were issued finish: wait for both
    if (warp == kProducer && lane == 0) {
      const int issued = ms.issued;
      for (int i = max(0, issued - NST); i < issued; ++i) {
        const RingPos<NST> pos(i);
        mbar_drain(bar(B_FULL + pos.idx), pos.ph);
      }
      mbar_drain(bar(B_Q), 0);
    }
    if (warp == kIssuer) {
      umma_commit_if(elect_one(), bar(B_DR));
      mbar_drain(bar(B_DR), 0);
    }
    __syncthreads();
  }
  // The status is settled by one thread (see seq_status.cuh).  The block is counted here, so that the addition's round trip
  // ends while the rows are staged; the waits of the merge come after it.
  TallyWords words = {reinterpret_cast<unsigned long long*>(p.tickets + 2 * b), p.status + b, p.wait_limit};
  const bool clerk = tid == 32 * kWriter;
  unsigned long long found = 0;
  if (clerk) found = add_block(words, aborted);

  // ---- merge.  Idle once all Q K^T of a block are done, which is when it arrives at the cluster
  //      barrier: the Q tiles (staging of the rows to be sent), and all ring stages but those of the
  //      last V tiles.  Two neighbouring stages receive; a third one holds what goes with this block's
  //      own rows (reference, sum, scales) | where each row's output starts | the sources' weights.
  //      Rows are 128 bytes per half of their columns, 16-byte piece c of row r at c ^ (r & 7).
  //      What counts is the number of instructions of one thread's chain, at about four cycles each: the same code, run
  //      again with warm caches, takes as long.  Packed arithmetic, each warp's rows sent as they are staged, a lane per
  //      source for the weights, addresses by increments: from where the roles meet to the end 6500 -> 5900 cycles for
  //      1 x 16 nodes x 512 keys (MHA), 5600 -> 5400 for 4 x 64 x 4096 (8 KV heads); the step of 32 layers of 1 x 60 x 1500
  //      and LM head 464 -> 451 us, of 4 x 64 x 4096 1010 -> 998.  (Stores from registers into the peers instead of staged
  //      copies: 130 cycles each, 478 us; sums sent ahead and weights worked out by the other warps while rows are
  //      staged, one copy per peer: 447 and 1010.)
  constexpr int kRows = Cfg<kRows2, kParts>::kRows, kSlotRows = kRows2 ? 2 * BM : BM;   // rows of a part; of a staged half
  constexpr uint32_t kHalfRows = (uint32_t)kSlotRows * 128u;
  const int received = (CS - 1) * kParts, sources = CS * kParts;
  auto rx_meta = [&](uint32_t rx_base) { return rx_base + (uint32_t)(received * per) * 256u; };   // behind the rows
  const uint32_t rx = sRing + at.rx[split], meta = sRing + at.meta;
  const uint32_t row_at = meta + 4096u, weights = meta + 8192u, lse_at = meta + 16384u;
  __syncwarp();
  if (warp < kSoftmaxWarps) {
    const int slot = (warp >> 2) & 1, row = (warp & 3) * 32 + lane, part = row / kRows, tile_row = row % kRows;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const int rtile = kRows2 ? at.tile0 + slot : at.tile0;
    const int node_in_tile = (int)Divisor{(unsigned)at.group_d, at.group_m}.divide((unsigned)tile_row), node = rtile * at.tile_nodes + node_in_tile;
    const bool row_valid = tile_row < at.tile_nodes * at.G && rtile < at.tiles && node < at.N;
    const int row_in_out = (b * at.N + node) * at.Hq + at.kvh * at.G + (tile_row - node_in_tile * at.G);
    const int seq_row = (kRows2 ? slot * BM : 0) + row;   // number of this row within the block
    float2 ml = ms.ml[slot * BM + row];
    float w0 = 1.f, w1 = 0.f;
    if (!kRows2) {   // combine the slots' shares of the keys
      const float2 a = ms.ml[row], c = ms.ml[BM + row];
      ml.x = fmaxf(a.x, c.x);
      const float mu = ml.x == -INFINITY ? 0.f : ml.x;
      w0 = ex2(a.x - mu);   // ex2(-inf) = 0
      w1 = ex2(c.x - mu);
      ml.y = a.y * w0 + c.y * w1;
    }
    if (alone) {
      const float inv = ml.y > 0.f ? 1.f / ml.y : 0.f;
      w0 *= inv;
      w1 *= inv;
      if (at.lse != nullptr && row_valid && (kRows2 || slot == 0)) at.lse[row_in_out] = log_sum_exp(ml.x, ml.y);
    }
    // what the warp's lane d will send to rank d
    int to_send = 0, send_from = 0;
    uint32_t their_rows = 0u, their_sums = 0u, their_bar = 0u;
    if (clustered && lane < CS && lane != split) {
      const int d = lane, row0 = row - lane - part * kRows + (kRows2 ? slot * BM : 0);   // the warp's first row, as the ranks share them out
      const int f = max(row0, d * per);
      to_send = min(min(R, d * per + per), row0 + 32) - f;
      send_from = f + part * kRows;
      const int src = (split < d ? split : split - 1) * kParts + part, to = f - d * per;
      const uint32_t base = cluster_map(sRing + at.rx[d], (uint32_t)d);
      their_bar = cluster_map(bar(B_RX), (uint32_t)d);
      their_rows = base + (uint32_t)(src * 2 * per + to) * 128u;
      their_sums = rx_meta(base) + (uint32_t)((kRows2 ? src : src * 2 + slot) * per + to) * 16u;
    }
    __syncwarp();
    // the last P V of the accumulators this thread reads
    const bool has0 = kRows2 ? slot < users && T > 0 : T > 0, has1 = !kRows2 && T > 1;
    if (!aborted) {
      const uint32_t bar0 = bar(B_LAST + (kRows2 ? slot : 0));
      bool done = (!has0 || mbar_test(bar0, 0)) & (!has1 || mbar_test(bar(B_LAST + 1), 0));   // both under way at once
      if (!__all_sync(0xFFFFFFFFu, done)) {
        done = !has0 || wait_warp(bar0, 0, &ms.late_flag, p.wait_limit);
        if (has1 && done) wait_warp(bar(B_LAST + 1), 0, &ms.late_flag, p.wait_limit);
      }
    }
    __syncwarp();
    tc_fence_after();
    // Half a row (64 columns) at a time: bf16 output if the block is alone (into the Q tile's place and layout; TMA
    // stores it), fp32 if its parts are all there is to add up (512 bytes per row where a cluster would receive), else
    // fp16 for the rank that finalises the row.
    const uint32_t acc0 = tmem + (uint32_t)(2 * BN + (kRows2 ? slot * HD : 0)) + lane_addr, acc1 = tmem + (uint32_t)(2 * BN + HD) + lane_addr;
    float downs[2] = {0.f, 0.f};   // what undoes the scales of the halves
#pragma unroll 1
    for (int half = kRows2 ? 0 : slot; half < (kRows2 ? 2 : slot + 1); ++half) {
      float2 v[32];
      {
        const float2 ww0 = make_float2(w0, w0), ww1 = make_float2(w1, w1);
        if (has1) {
          uint32_t u[64], u1[64];
          tmem_ld_x64(acc0 + (uint32_t)(half * 64), u);
          tmem_ld_x64(acc1 + (uint32_t)(half * 64), u1);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 32; ++j)
            v[j] = fma2(make_float2(__uint_as_float(u1[2 * j]), __uint_as_float(u1[2 * j + 1])), ww1,
                        mul2(make_float2(__uint_as_float(u[2 * j]), __uint_as_float(u[2 * j + 1])), ww0));
        } else if (has0) {
          uint32_t u[64];
          tmem_ld_x64(acc0 + (uint32_t)(half * 64), u);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = mul2(make_float2(__uint_as_float(u[2 * j]), __uint_as_float(u[2 * j + 1])), ww0);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = make_float2(0.f, 0.f);
        }
      }
      if (kOneBlock) {
        const uint32_t to = rx + (uint32_t)row * 512u;
#pragma unroll
        for (int c = 0; c < 16; ++c)   // 16-byte piece c of row r sits at c ^ (r & 31)
          st_shared16(to + (uint32_t)(((half * 16 + c) ^ (row & 31)) << 4), __float_as_uint(v[2 * c].x), __float_as_uint(v[2 * c].y),
                      __float_as_uint(v[2 * c + 1].x), __float_as_uint(v[2 * c + 1].y));
        continue;
      }
      uint32_t h[32], to;
      if (alone) {
#pragma unroll
        for (int j = 0; j < 32; ++j) h[j] = pack_bf16(v[j].x, v[j].y);
        to = smem0 + (kRows2 ? slot * kQTile : 0u) + (uint32_t)half * (kQTile / 2) + (uint32_t)row * 128u;
      } else {
        float top[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 32; ++j) top[j & 3] = max3(top[j & 3], fabsf(v[j].x), fabsf(v[j].y));
        const float amax = fmaxf(max3(top[0], top[1], top[2]), top[3]);
        // scale 2^lc with amax * 2^lc in [2^13, 2^14), up to the largest fp32 number; lc is clamped so that
        // the scale and its inverse are normal numbers (zeros stay zeros, inf or NaN stay what they are)
        const int lc = max(-114, min(100, 140 - (int)((__float_as_uint(amax) >> 23) & 255u)));
        const float up = __uint_as_float((uint32_t)(127 + lc) << 23), down = __uint_as_float((uint32_t)(127 - lc) << 23);
        if (half) downs[1] = down; else downs[0] = down;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float2 x = mul2(v[j], make_float2(up, up));
          const __half2 hv = __floats2half2_rn(x.x, x.y);
          h[j] = *reinterpret_cast<const uint32_t*>(&hv);
        }
        to = smem0 + (uint32_t)half * kHalfRows + (uint32_t)seq_row * 128u;
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) st_shared16(to + (uint32_t)((c ^ (row & 7)) << 4), h[4 * c], h[4 * c + 1], h[4 * c + 2], h[4 * c + 3]);
    }
    if (!alone) {   // (of the scales, a reader takes the one of the half that it reads)
      const float d0 = downs[0], d1 = downs[1];
      st_shared16(meta + (uint32_t)((kRows2 ? 0 : slot * BM) + seq_row) * 16u, __float_as_uint(ml.x), __float_as_uint(ml.y), __float_as_uint(d0), __float_as_uint(d1));
    }
    if (alone || clustered) fence_async_smem();
    tc_fence_before();
    __syncwarp();
    if (clustered) {   // each warp sends its rows, a lane per peer
      cluster_wait();   // every rank's receiving stages are idle
      if (to_send > 0) {
#pragma unroll
        for (int half = 0; half < 2; ++half)
          if (kRows2 || half == slot)
            bulk_to_peer(their_rows + (uint32_t)(half * per) * 128u, smem0 + (uint32_t)half * kHalfRows + (uint32_t)send_from * 128u, (uint32_t)to_send * 128u, their_bar);
        bulk_to_peer(their_sums, meta + (uint32_t)((kRows2 ? 0 : slot * BM) + send_from) * 16u, (uint32_t)to_send * 16u, their_bar);
      }
      __syncwarp();
    }
    if (!alone && (kRows2 || slot == 0))   // where the row's output starts (in rows of 128), -1: the row does not exist
      st_shared4(row_at + (uint32_t)seq_row * 4u, (uint32_t)(row_valid ? row_in_out : -1));
  } else if (clustered) {
    cluster_wait();
  }
  __syncthreads();
  bool failed = aborted || *reinterpret_cast<volatile int*>(&ms.late_flag) != 0;   // neither flag is written any more
  if (warp == kIssuer) {
    if (failed && !aborted) {   // the last P V is still under way
      umma_commit_if(elect_one(), bar(B_DR));
      mbar_drain(bar(B_DR), 0);
    }
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }

  if (clerk) publish_if_last(words, found, (unsigned)p.blocks_per_seq);
  __syncwarp();
  if (alone) {
    if (tid == 0 && !failed) {
#pragma unroll
      for (int m = 0; m < Cfg<kRows2, kParts>::kQ; ++m) {
        if (m >= users) break;
        tma_store_4d(&tm.out, smem0 + m * kQTile, 0, at.kvh * at.G, (at.tile0 + m) * at.tile_nodes, b);
        tma_store_4d(&tm.out, smem0 + m * kQTile + kQTile / 2, 64, at.kvh * at.G, (at.tile0 + m) * at.tile_nodes, b);
      }
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
    if (clerk && failed && !aborted) report_late(words, (unsigned)p.blocks_per_seq);
    return;
  }

  if (clustered) {
    if (!mbar_drain_within(bar(B_RX), 0, p.wait_limit)) ms.late_flag = 1;   // looked at again behind the next barrier
    __syncwarp();
    cluster_arrive();   // what this block was sent has arrived: its peers may leave
  }
  // ---- final rows.  A source of a row is a part of a block's accumulators: first what was received, by
  //      rank, then this block's own, always in this order, so that the result does not depend on timing.
  int rows = failed ? 0 : mine;
  if constexpr (kOneBlock) {   // this block's parts, fp32, eight columns of a row per item
    const uint32_t own_sums = meta + (uint32_t)first * 16u;
#pragma unroll 1
    for (int it = tid; it < rows * 16; it += kThreads) {
      const int i = it >> 4, c = it & 15, o = (int)ld_shared4(row_at + (uint32_t)(first + i) * 4u);
      float M = -INFINITY;
#pragma unroll
      for (int j = 0; j < kParts; ++j) M = fmaxf(M, ld_shared16(own_sums + (uint32_t)(j * kRows + i) * 16u).x);
      const float mu = M == -INFINITY ? 0.f : M;
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, total = 0.f;
#pragma unroll
      for (int j = 0; j < kParts; ++j) {
        const uint32_t r = (uint32_t)(j * kRows + i), from = rx + r * 512u;
        const float4 m = ld_shared16(own_sums + r * 16u);
        const float w = ex2(m.x - mu);   // ex2(-inf) = 0
        const float4 lo = ld_shared16(from + (((uint32_t)(2 * c) ^ (r & 31u)) << 4));
        const float4 hi = ld_shared16(from + (((uint32_t)(2 * c + 1) ^ (r & 31u)) << 4));
        const float x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        total = fmaf(m.y, w, total);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = fmaf(x[e], w, acc[e]);
      }
      const float inv = total > 0.f ? 1.f / total : 0.f;
      if (o < 0) continue;
      *reinterpret_cast<uint4*>(at.out + (int64_t)o * HD + c * 8) = make_uint4(pack_bf16(acc[0] * inv, acc[1] * inv), pack_bf16(acc[2] * inv, acc[3] * inv),
                                                                           pack_bf16(acc[4] * inv, acc[5] * inv), pack_bf16(acc[6] * inv, acc[7] * inv));
      if (c == 0 && at.lse != nullptr) at.lse[o] = log_sum_exp(M, total);
    }
  } else {
    // The sources' weights, a lane per source (2^n lanes per row, so that a row is a chain of two short reductions),
    // for either half of the columns.
    constexpr int kMetaStep = kRows2 ? 16 : 32;   // times per: from a source's to the next's
    const int lanes_log = sources <= 2 ? 1 : sources <= 4 ? 2 : sources <= 8 ? 3 : sources <= 16 ? 4 : 5;
#pragma unroll 1
    for (int it0 = warp * 32; it0 < rows << lanes_log; it0 += kThreads) {
      const int i = (it0 + lane) >> lanes_log, j = (it0 + lane) & ((1 << lanes_log) - 1);
      const bool here = i < rows && j < sources;
      float4 m0 = make_float4(-INFINITY, 0.f, 0.f, 0.f), m1 = m0;
      if (here) {
        const uint32_t at0 = j < received ? rx_meta(rx) + (uint32_t)(j * per * kMetaStep + i * 16) : meta + (uint32_t)((j - received) * kRows + first + i) * 16u;
        m0 = ld_shared16(at0);
        m1 = kRows2 ? m0 : ld_shared16(at0 + (j < received ? (uint32_t)per * 16u : (uint32_t)BM * 16u));
      }
      float M = m0.x;
#pragma unroll
      for (int d = 1; d < 32; d *= 2)
        if (d < 1 << lanes_log) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, d));
      const float w = ex2(m0.x - (M == -INFINITY ? 0.f : M));   // ex2(-inf) = 0
      float total = m0.y * w;
#pragma unroll
      for (int d = 1; d < 32; d *= 2)
        if (d < 1 << lanes_log) total += __shfl_xor_sync(0xFFFFFFFFu, total, d);
      const float inv = total > 0.f ? 1.f / total : 0.f;
      if (here) {
        const uint32_t to = weights + (uint32_t)(i * 2 * sources + j) * 4u;
        st_shared4(to, __float_as_uint(w * m0.z * inv));
        st_shared4(to + (uint32_t)sources * 4u, __float_as_uint(w * m1.w * inv));
        if (j == 0) st_shared8(lse_at + (uint32_t)i * 8u, M, total);
      }
    }
    __syncthreads();
    if (clustered && *reinterpret_cast<volatile int*>(&ms.late_flag) != 0) {
      failed = true;
      rows = 0;
    }
    if (at.lse != nullptr)   // by the last warps, which have fewer items below
      for (int i = kThreads - 1 - tid; i < rows; i += kThreads) {
        const int o = (int)ld_shared4(row_at + (uint32_t)(first + i) * 4u);
        const uint2 m = ld_shared8(lse_at + (uint32_t)i * 8u);
        if (o >= 0) at.lse[o] = log_sum_exp(__uint_as_float(m.x), __uint_as_float(m.y));
      }
    // kCols columns of a row per item, so that there are items for all threads; a source is a load, its weight another
    constexpr int kCols = kParts > 2 ? 4 : 8, kItems = HD / kCols;
#pragma unroll 1
    for (int it = tid; it < rows * kItems; it += kThreads) {
      const int i = it / kItems, c = it % kItems, half = c / (kItems / 2);
      const uint32_t piece = (uint32_t)(((c * kCols / 8) & 7) ^ (i & 7)) * 16u + (kCols == 4 ? (uint32_t)(c & 1) * 8u : 0u);   // first and per are multiples of 8
      float acc[kCols];
#pragma unroll
      for (int e = 0; e < kCols; ++e) acc[e] = 0.f;
      auto take = [&](uint32_t from, uint32_t w_at) {
        uint32_t h[kCols / 2];
        if constexpr (kCols == 8) {
          const float4 u = ld_shared16(from);
          h[0] = __float_as_uint(u.x); h[1] = __float_as_uint(u.y); h[2] = __float_as_uint(u.z); h[3] = __float_as_uint(u.w);
        } else {
          const uint2 u = ld_shared8(from);
          h[0] = u.x; h[1] = u.y;
        }
        const float w = __uint_as_float(ld_shared4(w_at));
#pragma unroll
        for (int x = 0; x < kCols / 2; ++x) {
          const float2 f = half2_bits_to_float2(h[x]);
          acc[2 * x] = fmaf(f.x, w, acc[2 * x]);
          acc[2 * x + 1] = fmaf(f.y, w, acc[2 * x + 1]);
        }
      };
      uint32_t w_at = weights + (uint32_t)((i * 2 + half) * sources) * 4u;
      uint32_t from = rx + (uint32_t)(half * per + i) * 128u + piece;
      const uint32_t step = (uint32_t)per * 256u;
#pragma unroll 4
      for (int j = 0; j < received; ++j, from += step, w_at += 4u) take(from, w_at);
      from = smem0 + (uint32_t)half * kHalfRows + (uint32_t)(first + i) * 128u + piece;
#pragma unroll
      for (int j = 0; j < kParts; ++j) take(from + (uint32_t)(j * kRows) * 128u, w_at + 4u * (uint32_t)j);
      const int o = (int)ld_shared4(row_at + (uint32_t)(first + i) * 4u);
      if (o < 0) continue;
      uint16_t* out = at.out + (int64_t)o * HD + c * kCols;
      if constexpr (kCols == 8)
        *reinterpret_cast<uint4*>(out) = make_uint4(pack_bf16(acc[0], acc[1]), pack_bf16(acc[2], acc[3]), pack_bf16(acc[4], acc[5]), pack_bf16(acc[6], acc[7]));
      else
        *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16(acc[0], acc[1]), pack_bf16(acc[2], acc[3]));
    }
  }
  __syncwarp();
  if (clustered) cluster_wait();   // no block may leave while a copy still reads its shared memory
  if (clerk && failed && !aborted) report_late(words, (unsigned)p.blocks_per_seq);
}

// ------------------------------------------------------------------------------------ host side
// bf16 tensor [rows][heads][128]; box = 64 elements x 1 head x box_rows, 128-byte swizzle
bool make_map(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t heads, uint32_t box_rows) {
  const cuuint64_t dims[3] = {(cuuint64_t)HD, heads, rows};
  const cuuint64_t strides[2] = {(cuuint64_t)HD * 2, (cuuint64_t)HD * 2 * heads};
  const cuuint32_t box[3] = {64, 1, box_rows};
  return encode_tile_map(tm, base, 3, dims, strides, box);
}

// Q and the output: [B][N][Hq][128], box = 64 elements x G heads x `nodes` nodes of one sequence, so
// that nodes beyond the sequence's last are read as zeros and never written
bool make_map_nodes(CUtensorMap* tm, const void* base, const clv_shape& s, uint32_t G, uint32_t nodes) {
  const cuuint64_t dims[4] = {(cuuint64_t)HD, (cuuint64_t)s.n_q_heads, (cuuint64_t)s.n_nodes, (cuuint64_t)s.batch};
  const cuuint64_t row = (cuuint64_t)HD * 2 * s.n_q_heads;
  const cuuint64_t strides[3] = {(cuuint64_t)HD * 2, row, row * s.n_nodes};
  const cuuint32_t box[4] = {64, G, nodes, 1};
  return encode_tile_map(tm, base, 4, dims, strides, box);
}

// The cache seen as [rows][heads][2 halves of d][64]: a box of 64 x box_rows x 2 x 1 in the order
// (d, row, half, head) lands in shared memory as [half][row][64], the layout of a K or V stage, so a
// tile of 128 neighbouring rows is one copy instead of four.
bool make_map_halves(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t heads, uint32_t box_rows) {
  const cuuint64_t dims[4] = {64, rows, 2, heads};
  const cuuint64_t strides[3] = {(cuuint64_t)HD * 2 * heads, 128, (cuuint64_t)HD * 2};
  const cuuint32_t box[4] = {64, box_rows, 2, 1};
  return encode_tile_map(tm, base, 4, dims, strides, box);
}

using Kernel = void (*)(Maps, Params);
Kernel kernel_of(bool rows2, int parts, int splits) {
  if (rows2) return tree_attn_kernel<true, 1, false>;
  if (parts == 1) return tree_attn_kernel<false, 1, false>;
  if (splits == 1) return parts == 4 ? tree_attn_kernel<false, 4, true> : tree_attn_kernel<false, 2, true>;
  return parts == 4 ? tree_attn_kernel<false, 4, false> : tree_attn_kernel<false, 2, false>;
}

// Once per device: the kernels' shared memory, and how many clusters of each size run at once (one
// block per SM; a cluster lives inside one GPC, so sizes that do not divide a GPC's SMs leave some idle).
int g_clusters[kMaxDevices][kMaxSplits + 1];

cudaError_t set_up() {
  const Kernel all[] = {kernel_of(true, 1, 1), kernel_of(false, 1, 1), kernel_of(false, 2, 1),
                        kernel_of(false, 4, 1), kernel_of(false, 2, 2), kernel_of(false, 4, 2)};
  for (const Kernel kernel : all) {
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, kernel);
    if (e == cudaSuccess && a.numRegs < kLaunchRegs) e = cudaErrorInvalidKernelImage;   // a block would wait for registers that it was not launched with
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  for (int s = 1; s <= kMaxSplits; ++s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(s * sm_count()), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)s;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, kernel_of(false, 1, 1), &cfg);
    if (e != cudaSuccess) return e;
    g_clusters[dev][s] = n > 0 ? n : 1;
  }
  return cudaSuccess;
}

struct AttnPlan {
  bool rows2;
  int parts, tiles, groups, splits;
};

// Blocks along the rows and along the keys: the cheapest choice by a cost in SM cycles, rounds of
// clusters over the machine times (key tiles of a block x cycles per tile + what a block takes
// besides).  The figures are fitted to measurements of 22 shapes (batch 1-32, 1-8 row tiles, 350-16424
// keys).  Lengths are data of the device, so every sequence counts as long as the bound.  A pool's pages are no
// measure of their mean: with n_pages / batch taken for it, ragged batches gained where the pool just held them (10 x 42 nodes,
// 28/4 heads, 3019-13316 keys: 115.2 -> 74.1 us; not in a pool of three times the pages), but equally long ones lost with shared pages
// (32 x 32, 8192 keys, 750 pages: 133.6 -> 147.1) or a loose bound (16 x 64, 4000 keys, bound 16384: 70.2 -> 98.5), and calls
// of blocks alone, whose partial sums stay fp32, went to clusters, which exchange theirs as fp16.
AttnPlan make_plan(const clv_shape& s, int max_ctx_len, const int* clusters) {
  const int G = s.n_q_heads / s.n_kv_heads;
  const int rows = s.n_nodes * G;
  const int parts = rows <= BM / 4 ? 4 : rows <= BM / 2 ? 2 : 1;
  const int tiles = (s.n_nodes + BM / G - 1) / (BM / G);   // row tiles of BM / G whole nodes
  const int pieces = pieces_of(max_ctx_len) + pieces_of(s.n_nodes);
  const int64_t units = (int64_t)s.batch * s.n_kv_heads;
  AttnPlan best = {false, parts, tiles, tiles, 1};
  double best_cost = 1e300;
  for (int r = 0; r < 2; ++r) {
    if (r && tiles < 2) break;
    const int groups = r ? (tiles + 1) / 2 : tiles;
    for (int sp = 1; sp <= kMaxSplits; ++sp) {
      if (sp > 1 && pieces < 2 * sp) break;   // at least one key tile per block
      const double rounds = (double)((units * groups + clusters[sp] - 1) / clusters[sp]);
      const double key_tiles = (double)((pieces + sp - 1) / sp) * 0.5;
      const double tile = r ? 3200.0 : parts > 1 ? 1200.0 : 1650.0;
      const double besides = sp == 1 ? 18000.0 : r ? 36000.0 : parts > 1 ? 19500.0 : 22500.0;
      const double cost = rounds * (key_tiles * tile + besides);
      if (cost < best_cost) { best_cost = cost; best = {r != 0, parts, tiles, groups, sp}; }
    }
  }
  return best;
}

}  // namespace

bool tree_attn_supported(const clv_shape& s, const clv_kv_cache& c) {
  const int G = s.n_q_heads / s.n_kv_heads;
  if (G > BM) return false;                            // a row tile must hold at least one whole node
  const int64_t cache_rows = c.paged ? (int64_t)c.n_pages * CLV_PAGE_SIZE : (int64_t)s.batch * c.cap_tokens;
  if (cache_rows >= (1ll << 31) || (int64_t)s.batch * s.n_nodes * s.n_q_heads >= (1ll << 31)) return false;
  return encode_fn() != nullptr;
}

cudaError_t launch_tree_attn(const clv_shape& s, const clv_kv_cache& c, const void* q, const void* k_tree,
                             const void* v_tree, const int32_t* parent, const int32_t* ctx_len, int max_ctx_len,
                             float scale, void* out, float* lse, int32_t* status, unsigned* tickets,
                             cudaStream_t stream) {
  static OncePerDevice once;
  cudaError_t e = run_once_per_device(once, set_up);
  if (e != cudaSuccess) return e;
  int dev = 0;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const AttnPlan plan = make_plan(s, max_ctx_len, g_clusters[dev]);
  const int G = s.n_q_heads / s.n_kv_heads;
  alignas(64) Maps tm;
  const uint64_t cache_rows = c.paged ? (uint64_t)c.n_pages * CLV_PAGE_SIZE : (uint64_t)s.batch * c.cap_tokens;
  const uint64_t tree_rows = (uint64_t)s.batch * s.n_nodes;
  if (!make_map_nodes(&tm.q, q, s, (uint32_t)G, (uint32_t)(BM / plan.parts / G)) ||
      !make_map_nodes(&tm.out, out, s, (uint32_t)G, (uint32_t)(BM / G)) ||
      !make_map(&tm.kc, c.k, cache_rows, s.n_kv_heads, PG) || !make_map(&tm.vc, c.v, cache_rows, s.n_kv_heads, PG) ||
      !make_map(&tm.kt, k_tree, tree_rows, s.n_kv_heads, PG) || !make_map(&tm.vt, v_tree, tree_rows, s.n_kv_heads, PG))
    return cudaErrorInvalidValue;
  // whole-tile copies: only if the driver accepts the 4-D view (else the piece-wise copies do it all)
  const bool pair_boxes = make_map_halves(&tm.kc2, c.k, cache_rows, s.n_kv_heads, BN) &&
                          make_map_halves(&tm.vc2, c.v, cache_rows, s.n_kv_heads, BN);
  if (!pair_boxes) { tm.kc2 = tm.kc; tm.vc2 = tm.vc; }

  Params p;
  p.pair_boxes = pair_boxes ? 1 : 0;
  p.block_table = c.block_table;
  p.parent = parent;
  p.ctx_len = ctx_len;
  p.out = static_cast<uint16_t*>(out);
  p.lse = lse;
  p.status = status;
  const int64_t clusters = (int64_t)s.batch * s.n_kv_heads * plan.groups;
  p.B = s.batch; p.N = s.n_nodes; p.Hq = s.n_q_heads; p.Hkv = s.n_kv_heads; p.G = G;
  p.paged = c.paged; p.cap_tokens = c.cap_tokens; p.n_pages = c.n_pages; p.max_pages = c.max_pages_per_seq;
  p.tiles = plan.tiles;
  p.groups = plan.groups;
  p.splits = plan.splits;
  p.longest_first = (clusters * plan.splits > sm_count() && s.batch > 1 && s.batch <= 256) ? 1 : 0;
  const int pieces = pieces_of(max_ctx_len) + pieces_of(s.n_nodes);
  p.ask_ahead = plan.parts > 1 && !p.longest_first && pieces >= 2 * kAheadFrom * plan.splits ? 1 : 0;
  p.scale_log2 = scale * 1.4426950408889634f;
  p.wait_limit = wait_limit_cycles();
  p.tickets = tickets;
  p.blocks_per_seq = s.n_kv_heads * plan.groups * plan.splits;
  p.tile_nodes = BM / plan.parts / G;
  p.by_splits = Divisor::of((unsigned)plan.splits);
  p.by_groups = Divisor::of((unsigned)plan.groups);
  p.by_kv_heads = Divisor::of((unsigned)s.n_kv_heads);
  p.by_group_heads = Divisor::of((unsigned)G);

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * plan.splits), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;  // the blocks that share row tiles
  attr[0].val.clusterDim.x = (unsigned)plan.splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // set-up overlaps the previous kernel's tail
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel_of(plan.rows2, plan.parts, plan.splits), tm, p);
}

}  // namespace clv
