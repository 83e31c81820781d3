// Shared device/host helpers of libhydra (internal).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <atomic>
#include "../../include/hydra.h"

namespace hydra {

typedef __nv_bfloat16 bf16;

// Device status word bits (sticky until polled).
enum : int { ST_BOUNDS = 1, ST_TIMEOUT = 2 };

// Launch bookkeeping: every launcher reports through this so the library can count its kernels.
extern thread_local long long* g_launch_counter;
void set_last_error(const char* what, cudaError_t e);
inline void count_launch() { if (g_launch_counter) ++*g_launch_counter; }

// Per-device one-time set-up (function attributes, SM counts) is keyed by the current device, so that one process
// may drive several GPUs; the flags are atomics because any thread may make the first call on a device.
constexpr int MAX_DEVICES = 64;
inline int current_device() { int d = 0; return cudaGetDevice(&d) == cudaSuccess && d >= 0 && d < MAX_DEVICES ? d : 0; }
struct PerDeviceFlag {
  std::atomic<bool> done[MAX_DEVICES];
  bool get() const { return done[current_device()].load(std::memory_order_acquire); }
  void set() { done[current_device()].store(true, std::memory_order_release); }
};
inline int sm_count() {
  static std::atomic<int> n[MAX_DEVICES];
  const int dev = current_device();
  int v = n[dev].load(std::memory_order_relaxed);
  if (v > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) v = 148;
  n[dev].store(v, std::memory_order_relaxed);
  return v;
}

#define HYDRA_CUDA(call)                                                        \
  do { cudaError_t e_ = (call);                                                 \
       if (e_ != cudaSuccess) { hydra::set_last_error(#call, e_); return HYDRA_ERR_CUDA; } } while (0)

#define HYDRA_LAUNCH_CHECK()                                                    \
  do { hydra::count_launch(); cudaError_t e_ = cudaGetLastError();              \
       if (e_ != cudaSuccess) { hydra::set_last_error("kernel launch", e_); return HYDRA_ERR_CUDA; } } while (0)

#define HYDRA_TRY(call) do { hydra_status s_ = (call); if (s_ != HYDRA_OK) return s_; } while (0)

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<bf16>(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f<bf16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// Sum of v[r] over the warp, for R values at once: lanes first trade halves of the values (R-1 shuffles for R values), then the
// remaining lane bits are folded.  Value warp_sum_owner(lane) ends up in lanes 0..R-1.
template <int R>
__device__ __forceinline__ float warp_sum_multi(float (&v)[R], int lane) {
#pragma unroll
  for (int n = R / 2, bit = 1; n >= 1; n /= 2, bit *= 2) {
    const bool up = lane & bit;
#pragma unroll
    for (int r = 0; r < n; ++r) {
      const float give = up ? v[r] : v[r + n], keep = up ? v[r + n] : v[r];
      v[r] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
    }
  }
  float s = v[0];
#pragma unroll
  for (int bit = R; bit < 32; bit *= 2) s += __shfl_xor_sync(0xffffffffu, s, bit);
  return s;
}
// which of the R values: the lowest lane bit chose the upper half, the next bit the upper quarter, ...
template <int R>
__device__ __forceinline__ int warp_sum_owner(int lane) {
  int r = 0;
#pragma unroll
  for (int n = R / 2, bit = 1; n >= 1; n /= 2, bit *= 2) r += (lane & bit) ? n : 0;
  return r;
}

// Programmatic dependent launch: every kernel of the library starts with pdl_trigger() (lets the next kernel
// in the stream get resident early) and pdl_wait() (blocks until the preceding kernel has completed and its
// writes are visible) before it touches what other kernels write, so dependencies stay transitive along the stream.  What an earlier
// kernel of the stream writes is never a `const ... __restrict__` parameter: the compiler may take such data as constant for the
// kernel's lifetime, which here begins before the writer has ended, and move its loads over the wait.  Weights and tables may be.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float silu_f(float x) { return x / (1.0f + __expf(-x)); }

// Where the partial sums of a GEMM output element live.  The tensor-core GEMM lays its (tile, k-block) pairs out in one line and cuts it
// into ranges of q units; tile t = (n >> bn_shift) * m_tiles + m / mt (weight tiles of 128 or 256 rows; mt: the rows of a group of row tiles that walk
// the line together) owns units [t*kb, (t+1)*kb), so its
// partial sums sit in slots 0 .. split_count-1 (slot s at part + s*stride + m*N + n), one per range that
// touches the tile, in their order.  A single-slot output is described by q = kb = 1.
struct SplitDesc {
  int q, kb, m_tiles, mt, bn_shift;
  unsigned long long q_inv, mt_inv;      // ceil(2^63 / q), ceil(2^32 / mt)
  size_t stride;
  void set_inverses() {
    q_inv = ((1ull << 63) + (unsigned)q - 1) / (unsigned)q;
    mt_inv = ((1ull << 32) + (unsigned)mt - 1) / (unsigned)mt;
  }
  // u / q, exact for all u, q < 2^31 (u * q_inv >> 63; the excess of q_inv, below 1, adds less than u / 2^63 < 1 / q); two multiplications
  __host__ __device__ unsigned div_q(unsigned u) const {
    return (unsigned)(((unsigned long long)u * (unsigned)(q_inv >> 32) + ((unsigned long long)u * (unsigned)q_inv >> 32)) >> 31);
  }
  // m / mt, exact while m mt < 2^32; other mt than 256 and 4096, which are exact for all m, come with at most 65536 rows
  __host__ __device__ int div_mt(int m) const { return (int)(((unsigned)m * mt_inv) >> 32); }
};
__host__ __device__ __forceinline__ int split_count(const SplitDesc& sd, int m, int n) {
  const int mi = sd.m_tiles == 1 ? 0 : sd.div_mt(m);
  const unsigned u0 = (unsigned)(((n >> sd.bn_shift) * sd.m_tiles + mi) * sd.kb);   // tiles * kb stays below 2^31
  return (int)(sd.div_q(u0 + sd.kb - 1) - sd.div_q(u0)) + 1;
}
// acc[u] = sum over the ns[u] slots of the four floats at element offset off[u] of a slot (all loads of a round in flight together)
template <int U, int PMAX = 6>
__device__ __forceinline__ void sum_slots_multi(const float* part, size_t stride, const size_t (&off)[U], const int (&ns)[U], float4 (&acc)[U]) {
  int mx = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) { acc[u] = make_float4(0.f, 0.f, 0.f, 0.f); mx = max(mx, ns[u]); }
#pragma unroll
  for (int p = 0; p < PMAX; ++p) {
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = p < ns[u] ? __ldcg(reinterpret_cast<const float4*>(part + p * stride + off[u])) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < U; ++u) { acc[u].x += v[u].x; acc[u].y += v[u].y; acc[u].z += v[u].z; acc[u].w += v[u].w; }
  }
  for (int p = PMAX; p < mx; ++p)
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (p < ns[u]) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(part + p * stride + off[u]));
        acc[u].x += v.x; acc[u].y += v.y; acc[u].z += v.z; acc[u].w += v.w;
      }
}
inline SplitDesc single_slot(size_t stride) {
  SplitDesc sd{1 << 30, 1, 1, 1 << 30, 30, 0, 0, stride};
  sd.set_inverses();
  return sd;
}

// Launch with programmatic stream serialisation allowed (see pdl_wait).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// A run of consecutive prompt rows of one sequence that an attention CTA takes as its query tile (packed row sets).
struct AttBlock {
  int seq, row0;           // sequence; the run's first row in the row set
  int pos0, n;             // cache slot of the first row; rows
  int call0;               // first cache slot that the forward call writes for this sequence
  int pad[3];
};

// Rows of one forward call: `batch` sequences with `tc` row slots each; sequence b uses its first
// n_rows[b] slots (all tc when n_rows is null).  Row i of b has KV slot pos0[b]+i, rotary position
// pos0[b]+depth[i] and may attend to cache slots < pos0[b] and to slot pos0[b]+j iff bit j of mask[i].
// With row_at the set is packed instead: n_packed causal rows back to back, row r = (sequence, cache slot = rotary position),
// cut into n_blocks attention blocks; the fields above are unused.
struct RowSet {
  int batch, tc;
  const int* n_rows;      // device [batch] or null
  const int* pos0;        // device [batch]
  const int* depth;       // device [tc]
  const uint64_t* mask;   // device [tc]; null: a causal chunk (row i sees new slots 0..i), bfloat16 model path only
  const int2* row_at = nullptr;          // device [n_packed]
  const AttBlock* blocks = nullptr;      // device [n_blocks]
  int n_packed = 0, n_blocks = 0;
  int n_tiles = 0;                       // 64-key tiles that the blocks of one head walk, all together
  __host__ __device__ int rows() const { return row_at ? n_packed : batch * tc; }
};

}  // namespace hydra
