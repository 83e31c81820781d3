// Stream-K GEMM entry point for callers that cannot allocate device memory.
//
// Who needs it: code that runs where cudaMalloc is off limits -- inside a latency-critical serving loop that
// must not take the allocator's locks or trigger an implicit device synchronisation, in a plugin whose host
// gave it a fixed memory budget, or after the process has handed all free device memory to a pool it does not
// control.  hydra_gemm makes such a caller bring the partial-sum buffer itself; this variant keeps
// that buffer inside the library image instead.
#include "launch.h"

namespace {

// Partial sums of the stream-K GEMM: m n floats for every CTA that touches a tile; where those of the usual plan do not fit, fewer CTAs
// share the work, down to one a tile.  8 MiB per GPU that loads the library, held until the process exits.  Shared by every call (and
// every thread) on that GPU.
constexpr size_t NOALLOC_SCRATCH_BYTES = 8u << 20;
// behind them the counters of one-launch calls (see GemmArrivals)
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES + hydra::GEMM_ONE_LAUNCH_TILES * sizeof(unsigned long long)];

// device address of the array, per device; 0 until the first call on that device has looked it up (any thread may
// make that call: the slot is an atomic, and two threads racing on it store the same address)
std::atomic<uintptr_t> g_scratch_ptr[hydra::MAX_DEVICES];
std::atomic<unsigned long long> g_ticket[hydra::MAX_DEVICES];      // of the last one-launch call

hydra_status scratch_on_current_device(int* dev, uintptr_t* addr) {
  using namespace hydra;
  *dev = -1;
  HYDRA_CUDA(cudaGetDevice(dev));
  if (*dev < 0 || *dev >= MAX_DEVICES) return HYDRA_ERR_UNSUPPORTED;
  *addr = g_scratch_ptr[*dev].load(std::memory_order_acquire);
  if (!*addr) {
    // The array's name is only a host-side handle here; the kernels need its address on the current device.
    void* p = nullptr;
    HYDRA_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    *addr = reinterpret_cast<uintptr_t>(p);
    g_scratch_ptr[*dev].store(*addr, std::memory_order_release);
  }
  return HYDRA_OK;
}

}  // namespace

extern "C" hydra_status hydra_gemm_noalloc_scratch(void** dev_ptr, size_t* partial_bytes, size_t* counter_bytes) {
  if (!dev_ptr) return HYDRA_ERR_INVALID;
  int dev;
  uintptr_t addr;
  HYDRA_TRY(scratch_on_current_device(&dev, &addr));
  *dev_ptr = reinterpret_cast<void*>(addr);
  if (partial_bytes) *partial_bytes = NOALLOC_SCRATCH_BYTES;
  if (counter_bytes) *counter_bytes = sizeof(g_noalloc_scratch) - NOALLOC_SCRATCH_BYTES;
  return HYDRA_OK;
}

extern "C" hydra_status hydra_gemm_noalloc(const void* x, const void* w, float* out, int m, int n, int k, int32_t* status,
                                           void* stream) {
  using namespace hydra;
  if (!x || !w || !out || !status || m < 1 || n < 1 || k < 1) return HYDRA_ERR_INVALID;
  if (n % 128 || k % 64) return HYDRA_ERR_UNSUPPORTED;
  if ((size_t)m * (size_t)n * sizeof(float) > NOALLOC_SCRATCH_BYTES) {
    set_last_error("hydra_gemm_noalloc: the partial sums exceed the 8 MiB built-in scratch", cudaErrorInvalidValue);
    return HYDRA_ERR_CAPACITY;
  }
  int dev;
  uintptr_t addr;
  HYDRA_TRY(scratch_on_current_device(&dev, &addr));
  if (!gemm_tc_available()) { set_last_error("cuTensorMapEncodeTiled entry point", cudaErrorUnknown); return HYDRA_ERR_CUDA; }
  float* part = reinterpret_cast<float*>(addr);
  // A captured call would keep its ticket for every replay: it takes the two-launch form, which has no state.
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  const cudaError_t asked = cudaStreamIsCapturing((cudaStream_t)stream, &capturing);
  if (asked != cudaSuccess) cudaGetLastError();          // (the default stream while another one captures: the launch will say so)
  const bool eager = asked == cudaSuccess && capturing == cudaStreamCaptureStatusNone;
  GemmArrivals arr{reinterpret_cast<unsigned long long*>(addr + NOALLOC_SCRATCH_BYTES), 0};
  if (eager) arr.ticket = g_ticket[dev].fetch_add(1, std::memory_order_relaxed) + 1;
  // every partial element that is added is written first: nothing has to be cleared
  return gemm_tc((const bf16*)x, m, 1, (const bf16*)w, part, m, n, k, nullptr, false, status, nullptr, nullptr, (cudaStream_t)stream,
                 NOALLOC_SCRATCH_BYTES / sizeof(float), out, eager ? &arr : nullptr);
}
