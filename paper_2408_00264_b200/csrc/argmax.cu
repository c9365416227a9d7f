// Per-node greedy choice: argmax over the vocabulary of each logits row (Sec. 4.2, T = 0).
//
// Pure HBM stream: every logit is read once with 16-byte loads that bypass L1.  With enough rows to cover the
// machine a block takes a whole row; with fewer a row is cut into `chunks` pieces, one per block of a cluster,
// whose (value, lowest index) pairs meet in the shared memory of the cluster's first block.  Long rows in small
// numbers are cut further, and the last block to arrive for a row takes the best of its pieces from global memory.
// The result is independent of the cut and of block scheduling.
#include <limits.h>

#include "clv_internal.cuh"

namespace clv {
namespace {

constexpr int kUnroll = 8;  // 16-byte loads of a batch (the results of about four at a time fit beside the maxima in 32 registers)
constexpr int kPieces = 6;                                   // of a row that a cluster shares
constexpr int kOnePerSm = 226 * 1024;                        // shared memory that only one block of an SM can have
constexpr int kPieceThreads = 256;                           // of blocks that meet through global memory
constexpr int kMaxPiece = 2 * kUnroll * kPieceThreads * 8;   // logits of such a block
constexpr int kMaxWholeRow = 1 << 26;                        // visits of a thread are numbered in 16 bits
enum Join { kWholeRow, kByCluster, kByTickets };

__device__ __forceinline__ uint4 ld_stream16(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t u) {
  return *reinterpret_cast<__nv_bfloat162*>(&u);
}

// Per-thread state: for each of the 8 positions inside a 16-byte vector, the running maximum (bf16)
// and the number of the visit at which it was first reached, both packed two per register.
// Updating is branch free (compare mask, max, bit select): a data-dependent branch would be taken
// by some lane of the warp at almost every step, because a thread only sees a few dozen vectors.
struct Track {
  __nv_bfloat162 m[4];
  uint32_t at[4];  // two 16-bit visit numbers; 0xFFFF = nothing above -inf seen yet
};
__device__ __forceinline__ void track_init(Track& t) {
#pragma unroll
  for (int j = 0; j < 4; ++j) { t.m[j] = as_bf162(0xFF80FF80u); t.at[j] = 0xFFFFFFFFu; }
}
__device__ __forceinline__ void take_vec(Track& t, const uint4& w, uint32_t visit2) {
  const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 x = as_bf162(u[j]);
    const uint32_t gt = __hgt2_mask(x, t.m[j]);  // strictly greater (false for NaN): first hit stays
    t.m[j] = __hmax2(t.m[j], x);                 // NaN operands are dropped
    t.at[j] = (t.at[j] & ~gt) | (visit2 & gt);
  }
}
struct Best {
  float v;
  int i;
};

// unsigned order = order of the values; -0 and +0 are the same value: one bit pattern
__device__ __forceinline__ uint32_t ordered(float v) {
  if (v == 0.0f) v = 0.0f;
  const uint32_t f = __float_as_uint(v);
  return (f & 0x80000000u) ? ~f : (f | 0x80000000u);
}
// of a warp: the highest value, and the lowest index that has it
__device__ __forceinline__ void first_of_highest(uint32_t& value, uint32_t& index) {
  const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, value);
  index = __reduce_min_sync(0xFFFFFFFFu, value == top ? index : 0xFFFFFFFFu);
  value = top;
}

struct Params {
  const uint16_t* logits;
  int64_t ld;
  int vocab;
  int chunks;
  int chunk_elems;
  int32_t* ids;
  unsigned* tickets;
  uint2* partial;   // (value in unsigned order, index) per piece of a row
};

__device__ __forceinline__ void cluster_started() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// a pair to the shared memory of the cluster's first block
__device__ __forceinline__ void st_first_block(const uint2* local, uint32_t x, uint32_t y) {
  uint32_t at;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(local)));
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(at), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void take_better(uint32_t& value, uint32_t& index, uint2 k) {
  if (k.x > value || (k.x == value && k.y < index)) { value = k.x; index = k.y; }
}

// 32 registers, so that as many blocks fit on an SM as its threads allow (with 34, 1024 rows of 128256: 39.0 -> 46.7 us)
template <int kThreads, Join kJoin>
__global__ void __launch_bounds__(kThreads, 2048 / kThreads) argmax_kernel(Params p) {
  const int row = blockIdx.x / p.chunks;
  const int chunk = blockIdx.x - row * p.chunks;
  const int begin = chunk * p.chunk_elems;
  const int end = min(p.vocab, begin + p.chunk_elems);
  const uint16_t* base = p.logits + (int64_t)row * p.ld;
  const int nvec = (end - begin) >> 3;
  const uint4* vp = reinterpret_cast<const uint4*>(base + begin);
  const int tid = threadIdx.x;
  // programmatic launch: the grid may be set up while the previous kernel of the stream drains;
  // nothing is read or written before that kernel's results are complete
  if (kJoin == kByCluster) cluster_started();
  cudaGridDependencySynchronize();

  Track trk;
  track_init(trk);
  int i = tid;
  uint32_t visit2 = 0;  // visit number in both halves
  for (; i + (kUnroll - 1) * kThreads < nvec; i += kUnroll * kThreads) {
    uint4 w[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) w[u] = ld_stream16(vp + i + u * kThreads);
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) { take_vec(trk, w[u], visit2); visit2 += 0x00010001u; }
  }
  // what is left, in one or two batches of four (vector by vector each of them cost a round trip: 64 rows of 32000 in
  // clusters of 4 3.14 -> 3.04 us, of 64000 5.8 -> 4.2)
  auto four = [&](bool guarded) {
    uint4 w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      w[u] = !guarded || i + u * kThreads < nvec ? ld_stream16(vp + i + u * kThreads) : make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
#pragma unroll
    for (int u = 0; u < 4; ++u) { take_vec(trk, w[u], visit2); visit2 += 0x00010001u; }
    i += 4 * kThreads;
  };
  if (i + 3 * kThreads < nvec) four(false);
  // (blocks through tickets take the same number of visits by all threads but in a row's last one: a single visit left
  // is not worth the three it would be filled up to, 8 x 262144 5.7 -> 5.1)
  if (kJoin == kByTickets && i + kThreads >= nvec) {
    if (i < nvec) take_vec(trk, ld_stream16(vp + i), visit2);
  } else if (i < nvec) {
    four(true);
  }
  // the thread's best of its 8 positions: visit k of this thread is vector tid + k * kThreads
  Best best = {-INFINITY, INT_MAX};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
#pragma unroll
    for (int hlf = 0; hlf < 2; ++hlf) {
      const uint32_t k = hlf ? (trk.at[j] >> 16) : (trk.at[j] & 0xFFFFu);
      if (k == 0xFFFFu) continue;
      const float v = hlf ? __high2float(trk.m[j]) : __low2float(trk.m[j]);
      const int idx = begin + 8 * (tid + (int)k * kThreads) + 2 * j + hlf;
      if ((v > best.v) || (v == best.v && idx < best.i)) { best.v = v; best.i = idx; }
    }
  }
  // ragged end of the row (vocab not a multiple of 8): at most 7 scalars, after all vectors
  {
    const int t0 = begin + 8 * nvec + tid;
    if (t0 < end) {
      float x = __uint_as_float((uint32_t)base[t0] << 16);
      if (x > best.v) { best.v = x; best.i = t0; }
    }
  }

  // Reduction in the order (value descending, index ascending), by whole warps: of a warp, of the row's or the
  // block's warps, of the row's pieces.  What a small call takes is this chain: through global memory (result, fence,
  // ticket, fence, results) it took 1.7 us of the 5 of 64 rows of 32000, which take 2.7 now.
  const int lane = tid & 31;
  constexpr int kWarps = kThreads / 32;
  uint32_t value = ordered(best.v), index = (uint32_t)best.i;
  first_of_highest(value, index);
  if constexpr (kJoin == kByCluster) {
    __shared__ uint2 s_pair[kPieces * kWarps];
    cluster_wait();   // every block of the row runs
    if (lane == 0) st_first_block(&s_pair[chunk * kWarps + (tid >> 5)], value, index);
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (chunk != 0 || tid >= 32) return;
    value = 0u;
    index = 0xFFFFFFFFu;
#pragma unroll
    for (int c = 0; c < kPieces * kWarps; c += 32)
      if (c + lane < p.chunks * kWarps) take_better(value, index, s_pair[c + lane]);
    first_of_highest(value, index);
  } else {
    __shared__ uint2 s_pair[kWarps];
    if (lane == 0) s_pair[tid >> 5] = make_uint2(value, index);
    __syncthreads();
    if (tid >= 32) return;
    const uint2 k = lane < kWarps ? s_pair[lane] : make_uint2(0u, 0xFFFFFFFFu);
    value = k.x;
    index = k.y;
    first_of_highest(value, index);
  }
  if constexpr (kJoin == kByTickets) {
    uint2* mine = p.partial + (size_t)row * p.chunks;
    unsigned arrived = 0;
    if (lane == 0) {
      __stcg(mine + chunk, make_uint2(value, index));
      __threadfence();
      arrived = atomicInc(p.tickets + row, (unsigned)p.chunks - 1);  // wraps to 0
    }
    if (__shfl_sync(0xFFFFFFFFu, arrived, 0) != (unsigned)p.chunks - 1) return;
    __threadfence();
    for (int c = lane; c < p.chunks; c += 32) take_better(value, index, __ldcg(mine + c));
    first_of_highest(value, index);
  }
  if (lane == 0) p.ids[row] = (index == (uint32_t)INT_MAX) ? 0 : (int)index;  // a row of only -inf / NaN: first index
}

}  // namespace

// How a call through tickets would cut its rows, which is also what a caller's workspace is sized for (whichever way
// the call takes): 32768 logits (64 KB) per block, less where there are too few rows to cover the machine.
ArgmaxPlan argmax_plan(int rows, int vocab) {
  ArgmaxPlan pl;
  pl.rows = rows;
  const int unit = kPieceThreads * 8;  // elements one pass of the block covers
  int chunk_elems = kMaxPiece;
  const int want_blocks = 4 * sm_count();
  while (chunk_elems > unit && (int64_t)rows * ((vocab + chunk_elems - 1) / chunk_elems) < want_blocks)
    chunk_elems >>= 1;
  pl.chunk_elems = chunk_elems;
  pl.chunks = (vocab + chunk_elems - 1) / chunk_elems;
  pl.scratch_bytes = pl.chunks > 1 ? sizeof(uint2) * (size_t)rows * pl.chunks : 0;
  return pl;
}

namespace {
// SMs that run a block each, of as much shared memory as there is, when all blocks are of clusters of kPieces
cudaError_t sms_of_clusters(void (*kernel)(Params), int threads, int* sms) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kPieces;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(kPieces * sm_count()), 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = kOnePerSm;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
  *sms = n > 0 ? n * kPieces : kPieces;
  return e;
}

template <int kThreads, Join kJoin>
cudaError_t launch(const Params& p, int rows, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((int64_t)rows * p.chunks), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  // Small blocks that are launched early would pile up on the SMs that attention leaves idle (step of 1 x 64 nodes x 2048
  // keys: with 32000 logits, clusters, 21.6 -> 21.0 us; with 200000, tickets, 25.2 -> 24.2).  Larger ones need the L1 that this
  // would take for their loads in flight.  A cluster's SMs are of one GPC, so its share is one of the SMs that clusters can
  // have (of all of them, 23-24, 47-49 and 72-74 rows had their last clusters wait for a wave: 24 x 128256 8.2 us, where 25
  // rows took 4.7).
  if (kJoin == kByCluster || (kJoin == kByTickets && p.chunk_elems < kMaxPiece)) {
    static OncePerDevice once;
    static int cluster_sms[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    const bool by_cluster = kJoin == kByCluster && dev < kMaxDevices;
    if (e == cudaSuccess)
      e = run_once_per_device(once, [&] {
        const cudaError_t set = cudaFuncSetAttribute(argmax_kernel<kThreads, kJoin>, cudaFuncAttributeMaxDynamicSharedMemorySize, kOnePerSm);
        return set == cudaSuccess && by_cluster ? sms_of_clusters(argmax_kernel<kThreads, kJoin>, kThreads, &cluster_sms[dev]) : set;
      });
    if (e != cudaSuccess) return e;
    cfg.dynamicSmemBytes = even_share_smem((int64_t)rows * p.chunks, 2048 / kThreads, by_cluster ? cluster_sms[dev] : sm_count());
  }
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)p.chunks;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = kJoin == kByCluster ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, argmax_kernel<kThreads, kJoin>, p);
}
}  // namespace

namespace {
// Logits up to which six blocks are enough for one of a few rows, and up to which rows that leave up to half of the SMs idle
// are not cut.  Back to back from a graph, cold, in us:
//    rows x vocabulary   cluster of 6   1024 threads   tickets
//       4 x 128256                4.4                      4.0   (a step of 1 x 4 nodes x 2048 keys: 17.7, 18.8)
//      50 x 152064                6.1                      6.5
//      74 x 153600                7.3                      7.5
//      74 x 163840                8.7                      7.5
//      32 x 200000                6.7                      6.1
//       4 x 262144                6.8                      4.3
//      75 x 180000                               8.1       9.7
//     100 x 196608                               9.3      10.0
//      80 x 200000                               9.3       8.7
//      75 x 400000                              15.4      12.5
//     111 x 400000                              17.4      18.9
constexpr int kLongForClusters = 153600, kLongForHalfAWave = 196608;
// Logits from which an SM's two rows are taken by 1024 threads each, rather than 512: 180 rows of 24000 4.4 us (512: 4.0), of
// 40000 6.0 (5.1), of 50257 6.2 (5.9), of 64000 6.2 (6.6), of 128256 9.4 (10.8); 149 and 296 rows likewise.
constexpr int kLongForTwo = 57344;

// Which way a call takes.
Join argmax_join(int rows, int vocab) {
  const int sms = sm_count();
  if (2 * rows <= sms) return vocab <= kLongForClusters ? kByCluster : kByTickets;
  return vocab <= (4 * rows < 3 * sms ? kLongForHalfAWave : kMaxWholeRow) ? kWholeRow : kByTickets;
}
}  // namespace

// Rows that cover the SMs at least half are not cut, and their blocks are as large as lets one wave take them all;
// fewer rows are shared by clusters of six blocks (of a row's best cut into 1, 2, 3, 4, 6, 8, six lost least); long rows that
// would leave much of the GPU idle are cut finely and go through tickets.  Back to back from a graph, cold, in us (before: all through tickets):
//   rows x vocabulary     before   1024 threads    512    256   cluster of 6   taken
//    16 x 32000              3.6            2.6    2.4    2.8            2.3   cluster
//    64 x 32000              5.5            2.7    3.1    4.2            2.7   cluster
//    64 x 128256             6.7            6.3    9.2   15.4            5.5   cluster
//   100 x 128256             8.7            7.0    9.7   15.6            6.8   1024
//   128 x 16000              5.7            3.2    3.3    4.9            4.0   1024
//   192 x 32000              5.9            5.0    4.6    5.8            5.4   512
//   256 x 128256            13.3           11.9   12.7   17.4           14.6   1024
//   512 x 64000             14.1           13.5   12.1   13.5           15.5   512
//   768 x 32000             10.1           11.7   11.0   10.1           14.9   256
//  1024 x 128256            41.4           42.2   39.8   39.0           44.8   256
cudaError_t launch_argmax(const ArgmaxPlan& plan, const void* logits, int64_t ld, int vocab,
                          int32_t* ids, unsigned* tickets, void* scratch, cudaStream_t stream) {
  Params p;
  p.logits = static_cast<const uint16_t*>(logits);
  p.ld = ld;
  p.vocab = vocab;
  p.chunks = 1;
  p.chunk_elems = vocab;
  p.ids = ids;
  p.tickets = tickets;
  p.partial = static_cast<uint2*>(scratch);
  switch (argmax_join(plan.rows, vocab)) {
    case kWholeRow: {
      const int sms = sm_count();
      if (plan.rows <= sms || (plan.rows <= 2 * sms && vocab > kLongForTwo)) return launch<1024, kWholeRow>(p, plan.rows, stream);
      if (plan.rows <= 4 * sms) return launch<512, kWholeRow>(p, plan.rows, stream);
      return launch<256, kWholeRow>(p, plan.rows, stream);
    }
    case kByTickets:
      p.chunks = plan.chunks;
      p.chunk_elems = plan.chunk_elems;
      return launch<kPieceThreads, kByTickets>(p, plan.rows, stream);
    case kByCluster: break;
  }
  p.chunk_elems = ((vocab + kPieces - 1) / kPieces + 7) & ~7;
  p.chunks = (vocab + p.chunk_elems - 1) / p.chunk_elems;
  return launch<256, kByCluster>(p, plan.rows, stream);
}

// ---- variant whose scratch lives in the library image ------------------------------------------
// For callers that cannot allocate device memory at all.  The scratch (arrival counters followed
// by the pieces' results) is a fixed array in this module's device image: every GPU that loads the
// library holds it until the process exits, and every call on that GPU shares it.
namespace {
constexpr int kStaticMaxRows = 4096;         // B * N
constexpr int kStaticMaxKeys = 131072;       // rows * chunks
constexpr size_t kStaticTicketBytes = sizeof(unsigned) * (size_t)kStaticMaxRows;
constexpr size_t kStaticBytes = kStaticTicketBytes + sizeof(uint2) * (size_t)kStaticMaxKeys;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

unsigned char* g_static_ptr[kMaxDevices] = {};   // device address of g_static_scratch, per device
}  // namespace

bool argmax_static_fits(int rows, int vocab) {
  if (rows > kStaticMaxRows) return false;
  const ArgmaxPlan plan = argmax_plan(rows, vocab);
  return (int64_t)rows * plan.chunks <= kStaticMaxKeys;
}

cudaError_t launch_argmax_static(const void* logits, int64_t ld, int rows, int vocab, int32_t* ids,
                                 cudaStream_t stream) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (g_static_ptr[dev] == nullptr) {
    // In host code the array's name is only a handle; the address the kernel can use has to be
    // asked for, with the device that will run the kernel current.
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_static_scratch);
    if (e != cudaSuccess) return e;
    g_static_ptr[dev] = static_cast<unsigned char*>(ptr);
  }
  unsigned char* base = g_static_ptr[dev];
  const ArgmaxPlan plan = argmax_plan(rows, vocab);
  if (argmax_join(rows, vocab) == kByTickets) {
    // the counters must start at zero whatever an earlier (possibly aborted) call left behind (without the fill
    // 64 rows of 128256 that stay in L2 take 3.5 us instead of 7.4)
    e = cudaMemsetAsync(base, 0, sizeof(unsigned) * (size_t)rows, stream);
    if (e != cudaSuccess) return e;
  }
  return launch_argmax(plan, logits, ld, vocab, ids, reinterpret_cast<unsigned*>(base),
                       base + kStaticTicketBytes, stream);
}

}  // namespace clv
