// What the whole step from host buffers needs besides the step's own kernels: a second stream for the
// copies that attention does not wait for, and one launch that writes the small results to the host.
// The step is bound by the link: 1 x 64 nodes, 32000 logits each, are 5.6 MB up (108 us at 52 GB/s) and
// 0.5 MB down.  Both copies up at once fill the gaps between them, attention and the copy down hide behind
// the logits: 202 -> 147 us.  (With the logits behind Q and the tree's rows instead of beside them: 156.)
#include <algorithm>
#include <mutex>

#include "clv_internal.cuh"

namespace clv {
namespace {

struct SideSlot {
  SideStream side = {};
  bool made = false, taken = false;
  unsigned long long user = 0;   // id of the caller's stream that it served last
};
constexpr int kSideSlots = 8;   // per device: callers' streams with a step under way; any further one does without
std::mutex g_side_mu;
SideSlot g_side[kMaxDevices][kSideSlots];

// What is done in here may not disturb a capture that a host thread has under way.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
};

cudaError_t make_side(SideStream* s) {
  cudaError_t e = cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s->fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s->join, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    if (s->fork) (void)cudaEventDestroy(s->fork);
    if (s->stream) (void)cudaStreamDestroy(s->stream);
    *s = SideStream{};
    (void)cudaGetLastError();
  }
  return e;
}

struct HostArrays {
  const int32_t* from[kHostArrays];
  int32_t* to[kHostArrays];
  int n[kHostArrays];
};

__global__ void __launch_bounds__(256) host_results_kernel(HostArrays a) {
  cudaGridDependencySynchronize();
  const int t = blockIdx.x * 256 + threadIdx.x, stride = gridDim.x * 256;
#pragma unroll
  for (int k = 0; k < kHostArrays; ++k)
    for (int i = t; i < a.n[k]; i += stride) a.to[k][i] = a.from[k][i];
}

}  // namespace

// The slot is the caller's until it is given back, which is when the call has enqueued its work: the
// next user's events then replace this one's, whose waits have taken note of them already.  What the
// call has put on the slot's stream waits for the caller's stream, so the next user may be a call on the
// same stream, or any once that work is done: two streams of a caller's are never ordered by a slot.
SideStream* take_side_stream(cudaStream_t s) {
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;   // never used again for another stream, as a handle may be
  int dev = 0;
  if (cudaStreamIsCapturing(s, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone ||
      cudaStreamGetId(s, &id) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return nullptr;   // a capture: a side stream would belong to it until it ends
  }
  if (dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_side_mu);
  RelaxedCapture relaxed;
  SideSlot* pick = nullptr;
  for (SideSlot& slot : g_side[dev])
    if (slot.made && !slot.taken && slot.user == id) pick = &slot;
  for (int i = 0; i < kSideSlots && !pick; ++i) {
    SideSlot& slot = g_side[dev][i];
    if (slot.taken) continue;
    if (!slot.made) {
      if (make_side(&slot.side) != cudaSuccess) return nullptr;
      slot.made = true;
      pick = &slot;
    } else if (cudaEventQuery(slot.side.join) == cudaSuccess) {
      pick = &slot;
    } else {
      (void)cudaGetLastError();   // not done
    }
  }
  if (!pick) return nullptr;
  pick->taken = true;
  pick->user = id;
  return &pick->side;
}

void give_side_stream(SideStream* s) {
  std::lock_guard<std::mutex> lock(g_side_mu);
  reinterpret_cast<SideSlot*>(s)->taken = false;   // the stream is the slot's first member
}

// Device addresses of pinned host arrays; false if one of them is not the kernel's to write: not pinned from end
// to end (asked page by page: what is pinned is whole pages), not aligned, or so long that a copy is
// as good.
bool host_arrays_on_device(int32_t* const* host, const size_t* n, int32_t** device) {
  constexpr size_t kPage = 4096, kMostPages = 64;
  for (int k = 0; k < kHostArrays; ++k) {
    const uintptr_t begin = reinterpret_cast<uintptr_t>(host[k]), end = begin + n[k] * sizeof(int32_t);
    if (begin % sizeof(int32_t) != 0 || end - begin > kMostPages * kPage) return false;
    const uintptr_t last = end - sizeof(int32_t);
    for (uintptr_t at = begin; at < end; at = at == last ? end : std::min((at / kPage + 1) * kPage, last)) {
      cudaPointerAttributes a;
      if (cudaPointerGetAttributes(&a, reinterpret_cast<const void*>(at)) != cudaSuccess || a.type != cudaMemoryTypeHost ||
          !a.devicePointer) {
        (void)cudaGetLastError();
        return false;
      }
      if (at == begin) device[k] = static_cast<int32_t*>(a.devicePointer);
      else if (reinterpret_cast<uintptr_t>(a.devicePointer) - reinterpret_cast<uintptr_t>(device[k]) != at - begin) return false;
    }
  }
  return true;
}

// One launch in place of a copy per array: each costs 2 to 3 us of the copy engine, for a few hundred bytes.
cudaError_t launch_host_results(const int32_t* const* from, int32_t* const* to, const size_t* n, cudaStream_t stream) {
  HostArrays a;
  size_t most = 1;
  for (int k = 0; k < kHostArrays; ++k) {
    a.from[k] = from[k];
    a.to[k] = to[k];
    a.n[k] = (int)n[k];
    if (n[k] > most) most = n[k];
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((most + 255) / 256 < 64 ? (most + 255) / 256 : 64), 1, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, host_results_kernel, a);
}

}  // namespace clv
