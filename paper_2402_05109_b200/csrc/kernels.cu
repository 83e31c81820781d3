// Row-wise, element-wise, attention, draft-head and acceptance kernels of libhydra (everything that is
// not the tensor-core GEMM).  float or bfloat16 storage, float arithmetic.
#include "launch.h"
#include <math.h>
#include <algorithm>
#include <vector>

namespace hydra {

// ------------------------------------------------------------------------------------------------
// SIMT GEMM of bfloat16 operands (the debug mode): out[m][n] = sum_k x[m][k] w[n][k].  One warp per output feature, MR rows per pass.
// (Float operands: float_path.cu.)
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ void load_bf16x4(const bf16* p, float (&v)[4]) {
  uint2 t = *reinterpret_cast<const uint2*>(p);
  __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162*>(&t.x), b = *reinterpret_cast<__nv_bfloat162*>(&t.y);
  v[0] = __low2float(a); v[1] = __high2float(a); v[2] = __low2float(b); v[3] = __high2float(b);
}

// MR activation rows; KS warps share an output column (each every KS-th piece of 128 weights of its row), 8 / KS columns per
// block.  The first WPRE weight pieces of a lane are loaded before the wait for the preceding kernel (w_const: the weights of a context, which no
// kernel writes; a stand-alone call's w may be the preceding kernel's result), the MR sums share one transposing reduction, and the
// split keeps the activation loads of a lane to one or two rounds and fills the SMs.
template <int MR, int KS>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const bf16* x, const bf16* w,      // not __restrict__: such loads may be moved over the wait
                                                        float* __restrict__ out, int m, int n, int k, int w_const) {
  constexpr int WPRE = 2;
  pdl_trigger();
  __shared__ float s_part[8][MR];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int col = blockIdx.x * (8 / KS) + warp / KS, k0 = (warp % KS) * 128 + lane * 4;
  const int m0 = blockIdx.y * MR;
  const bf16* wr = w + (size_t)min(col, n - 1) * k;
  float wv[WPRE][4];
  if (!w_const) pdl_wait();
#pragma unroll
  for (int i = 0; i < WPRE; ++i)
    if (k0 + i * KS * 128 < k) load_bf16x4(wr + k0 + i * KS * 128, wv[i]);
  if (w_const) pdl_wait();
  float acc[MR];
#pragma unroll
  for (int r = 0; r < MR; ++r) acc[r] = 0.f;
  auto step = [&](int kk, const float (&wk)[4]) {
#pragma unroll
    for (int r = 0; r < MR; ++r) {
      const int row = m0 + r < m ? m0 + r : m - 1;
      float xv[4];
      load_bf16x4(x + (size_t)row * k + kk, xv);
      acc[r] += wk[0] * xv[0] + wk[1] * xv[1] + wk[2] * xv[2] + wk[3] * xv[3];
    }
  };
#pragma unroll
  for (int i = 0; i < WPRE; ++i)
    if (k0 + i * KS * 128 < k) step(k0 + i * KS * 128, wv[i]);
  for (int kk = k0 + WPRE * KS * 128; kk < k; kk += KS * 128) {
    float wk[4];
    load_bf16x4(wr + kk, wk);
    step(kk, wk);
  }
  float s = warp_sum_multi<MR>(acc, lane);
  const int r = warp_sum_owner<MR>(lane);
  if constexpr (KS > 1) {
    if (lane < MR) s_part[warp][r] = s;
    __syncthreads();
    if (warp % KS) return;
    if (lane < MR) {
#pragma unroll
      for (int q = 1; q < KS; ++q) s += s_part[warp + q][r];
    }
  }
  if (lane < MR && m0 + r < m && col < n) out[(size_t)(m0 + r) * n + col] = s;
}

template <int MR>
static void launch_gemm_simt(const void* x, const void* w, float* out, int m, int n, int k, bool w_const, cudaStream_t st) {
  const int groups = (m + MR - 1) / MR;
  auto go = [&](auto kernel, int ks) {
    launch_pdl(kernel, dim3((n * ks + 7) / 8, groups), dim3(256), 0, st, (const bf16*)x, (const bf16*)w, out, m, n, k, (int)w_const);
  };
  // warps per column: until there are two blocks per SM or a lane has one piece
  const int pieces = (k + 127) / 128, want = 2 * sm_count();
  if (pieces >= 4 && (long)n * groups / 4 <= want) go(gemm_simt_kernel<MR, 4>, 4);
  else if (pieces >= 2 && (long)n * groups / 8 <= want) go(gemm_simt_kernel<MR, 2>, 2);
  else go(gemm_simt_kernel<MR, 1>, 1);
}
hydra_status gemm_simt(const void* x, const void* w, float* out, int m, int n, int k, int dtype, bool w_const, cudaStream_t st) {
  if (m <= 0 || n <= 0 || k <= 0 || (k & 3)) return HYDRA_ERR_UNSUPPORTED;
  if (((uintptr_t)x | (uintptr_t)w) & (dtype == 0 ? 15 : 7)) return HYDRA_ERR_INVALID;      // both are read four elements at a time
  if (dtype == 0) return f32_gemm((const float*)x, (const float*)w, out, m, n, k, w_const, st);
  if (m == 1) launch_gemm_simt<1>(x, w, out, m, n, k, w_const, st);
  else if (m <= 4) launch_gemm_simt<4>(x, w, out, m, n, k, w_const, st);
  else if (m <= 8) launch_gemm_simt<8>(x, w, out, m, n, k, w_const, st);
  else launch_gemm_simt<16>(x, w, out, m, n, k, w_const, st);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

template <typename T> inline bool on_vec4(const T* p) { return ((uintptr_t)p & (4 * sizeof(T) - 1)) == 0; }
// Up to twelve slots: four columns of a row a thread, all slots in flight together, index work ahead of the wait.  VEC: the result lies on a 16-byte boundary.
constexpr int REDUCE_THREADS = 64, REDUCE_SLOTS = 12;
template <bool VEC>
__global__ void __launch_bounds__(REDUCE_THREADS) reduce_splits_kernel(const float* part, SplitDesc sd, float* __restrict__ out, int n) {
  pdl_trigger();
  const int c = (blockIdx.x * REDUCE_THREADS + threadIdx.x) * 4, r = blockIdx.y;
  if (c >= n) return;
  const size_t off[1] = {(size_t)r * n + c};
  const int ns[1] = {split_count(sd, r, c)};
  pdl_wait();
  float4 v[1];
  sum_slots_multi<1, REDUCE_SLOTS>(part, sd.stride, off, ns, v);
  float* dst = out + off[0];
  if constexpr (VEC) *reinterpret_cast<float4*>(dst) = v[0];
  else { dst[0] = v[0].x; dst[1] = v[0].y; dst[2] = v[0].z; dst[3] = v[0].w; }
}
// Any number of them: a column a thread.
__global__ void reduce_splits_any_kernel(const float* part, SplitDesc sd, float* __restrict__ out, int m, int n) {
  pdl_trigger();
  pdl_wait();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)m * n) return;
  const int ns = split_count(sd, (int)(i / n), (int)(i % n));
  float s = 0.f;
  for (int p = 0; p < ns; ++p) s += part[p * sd.stride + i];
  out[i] = s;
}
hydra_status reduce_splits(const float* part, SplitDesc sd, float* out, int m, int n, cudaStream_t st) {
  // Back to back with the GEMM, 11 rows, a column a thread against four: 4096 x 4096 (10 slots) 10.00 / 9.62 us, 8192 x 2048 9.98 / 9.31, 4096 x 2048 7.94 / 7.23, 6656 x 6656
  // 17.6 / 16.5; with more slots than are in flight together 2048 x 8192 10.45 / 10.94, 32 x 256 x 11008 8.28 / 9.62
  const int slots = (sd.kb + sd.q - 2) / sd.q + 1;
  if (slots <= REDUCE_SLOTS && on_vec4(part) && n % 4 == 0 && m <= 65535) {
    const dim3 grid((n / 4 + REDUCE_THREADS - 1) / REDUCE_THREADS, m);
    launch_pdl(on_vec4(out) ? reduce_splits_kernel<true> : reduce_splits_kernel<false>, grid, dim3(REDUCE_THREADS), 0, st, part, sd, out, n);
  } else {
    launch_pdl(reduce_splits_any_kernel, dim3((unsigned)(((size_t)m * n + 255) / 256)), dim3(256), 0, st, part, sd, out, m, n);
  }
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <> __device__ __forceinline__ float4 load4<bf16>(const bf16* p) {
  float v[4]; load_bf16x4(p, v); return make_float4(v[0], v[1], v[2], v[3]);
}
// Four elements at an element boundary (VEC: at a boundary of four).
template <bool VEC, typename T> __device__ __forceinline__ float4 load4_at(const T* p) {
  if constexpr (VEC) return load4<T>(p);
  else return make_float4(to_f<T>(p[0]), to_f<T>(p[1]), to_f<T>(p[2]), to_f<T>(p[3]));
}

// ------------------------------------------------------------------------------------------------
// Residual add of split-K partial sums + RMSNorm (Llama: x * gain / sqrt(mean(x^2) + eps))
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float block_sum(float v, float* sh) {
  v = warp_sum(v);
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  float t = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.f;
  if (warp == 0) { t = warp_sum(t); if (lane == 0) sh[0] = t; }
  __syncthreads();
  t = sh[0];
  __syncthreads();
  return t;
}

template <typename T> __device__ __forceinline__ void store4(T* p, float4 v);
template <> __device__ __forceinline__ void store4<float>(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
template <> __device__ __forceinline__ void store4<bf16>(bf16* p, float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  uint2 u; u.x = *reinterpret_cast<uint32_t*>(&a); u.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}
template <> __device__ __forceinline__ void store4<__half>(__half* p, float4 v) {
  __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
  uint2 u; u.x = *reinterpret_cast<uint32_t*>(&a); u.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}
// hi = f16(v) and, ps elements further on, lo = f16(v - hi) (ps = 0: hi only).
__device__ __forceinline__ void put4h(__half* p, size_t ps, float4 v) {
  const float4 h = make_float4(__half2float(__float2half_rn(v.x)), __half2float(__float2half_rn(v.y)),
                               __half2float(__float2half_rn(v.z)), __half2float(__float2half_rn(v.w)));
  store4<__half>(p, h);
  if (ps) store4<__half>(p + ps, make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w));
}

// Operand storage.  float buffers hold one plane.  bfloat16 operand buffers hold two planes `ps` elements apart:
// hi = bf16(v) and lo = bf16(v - hi), together about 16 mantissa bits (ps = 0 stores hi only).
template <typename T> __device__ __forceinline__ void put(T* p, size_t ps, float v);
template <> __device__ __forceinline__ void put<float>(float* p, size_t, float v) { *p = v; }
template <> __device__ __forceinline__ void put<bf16>(bf16* p, size_t ps, float v) {
  const bf16 h = __float2bfloat16_rn(v);
  *p = h;
  if (ps) p[ps] = __float2bfloat16_rn(v - __bfloat162float(h));
}
template <typename T> __device__ __forceinline__ void put4(T* p, size_t ps, float4 v);
template <> __device__ __forceinline__ void put4<float>(float* p, size_t, float4 v) { *reinterpret_cast<float4*>(p) = v; }
template <> __device__ __forceinline__ void put4<bf16>(bf16* p, size_t ps, float4 v) {
  const float4 h = make_float4(__bfloat162float(__float2bfloat16_rn(v.x)), __bfloat162float(__float2bfloat16_rn(v.y)),
                               __bfloat162float(__float2bfloat16_rn(v.z)), __bfloat162float(__float2bfloat16_rn(v.w)));
  store4<bf16>(p, h);
  if (ps) store4<bf16>(p + ps, make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w));
}

template <typename T> struct alignas(4 * sizeof(T)) Raw4 { T v[4]; };      // four elements as stored
constexpr int NORM_THREADS = 1024;
// x_out = res + sum of the partial-sum slots; with `gain`, also xn = rmsnorm(x_out) * gain (operand planes) and hn (float).
// A row is shared by the CS CTAs of a thread-block cluster (CTA `rank` owns d / CS consecutive columns), so that few rows
// still pull their partial sums through many SMs.  The kernel is a chain of latencies (a few hundred KB in all), so what does
// not depend on the preceding kernel - the slot counts, the gain - comes before the wait for it,
// and every warp leaves its sum of squares in the shared memory of all CTAs of the row, so that one barrier follows the sums.  A CTA's shared
// memory may be stored to once that CTA has started: a barrier, arrived at on entry and waited for behind the sums, says so (0.35 % of
// a 7B step without a tree; waited for ahead of the sums 0.6 %).
template <typename T, int CS>
__global__ void __launch_bounds__(NORM_THREADS) residual_rmsnorm_kernel(const float* res, const float* part,
                                                                        SplitDesc sd, float* x_out,
                                                                        const T* __restrict__ gain, T* __restrict__ xn, size_t xn_ps,
                                                                        float* __restrict__ hn, int d, float eps) {
  pdl_trigger();
  if constexpr (CS > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  __shared__ float s_ss[CS * 32];
  const int row = blockIdx.x / CS, rank = blockIdx.x % CS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int dc = d / CS, c0 = rank * dc, i0 = c0 + threadIdx.x * 4;
  const size_t base = (size_t)row * d;
  int ns0 = part && i0 < c0 + dc ? split_count(sd, row, i0) : 0;
  Raw4<T> g0{};
  if (gain && i0 < c0 + dc) g0 = *reinterpret_cast<const Raw4<T>*>(gain + i0);
  pdl_wait();
  float ss = 0.f;
  float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f);                          // this thread's first piece stays in registers
  for (int i = i0; i < c0 + dc; i += blockDim.x * 4) {                  // one 16-byte piece per thread and round, all its slot loads in flight together
    size_t off[1] = {base + i};
    int ns[1] = {i == i0 ? ns0 : part ? split_count(sd, row, i) : 0};
    float4 acc[1];
    float4 v = res ? *reinterpret_cast<const float4*>(res + base + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    sum_slots_multi<1, 12>(part, sd.stride, off, ns, acc);             // narrow outputs are cut into up to ~11 slots per tile
    v.x += acc[0].x; v.y += acc[0].y; v.z += acc[0].z; v.w += acc[0].w;
    *reinterpret_cast<float4*>(x_out + base + i) = v;
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    if (i == i0) v0 = v;
  }
  if constexpr (CS > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // all CTAs of the row have started
  if (!gain) return;
  ss = warp_sum(ss);
  if constexpr (CS > 1) {
    if (lane < CS) {                                                     // lane r leaves the warp's sum in CTA r's table
      uint32_t local = (uint32_t)__cvta_generic_to_shared(&s_ss[rank * 32 + warp]), remote;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"((uint32_t)lane));
      asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(ss) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    if (lane == 0) s_ss[warp] = ss;
    __syncthreads();
  }
  float tot = 0.f;
#pragma unroll
  for (int c = 0; c < CS; ++c) tot += lane < nw ? s_ss[c * 32 + lane] : 0.f;
  tot = warp_sum(tot);
  const float inv = rsqrtf(tot / (float)d + eps);
  for (int i = i0; i < c0 + dc; i += blockDim.x * 4) {
    float4 v = i == i0 ? v0 : *reinterpret_cast<const float4*>(x_out + base + i);
    const float4 gn = i == i0 ? load4<T>(reinterpret_cast<const T*>(&g0)) : load4<T>(gain + i);
    v.x *= inv * gn.x; v.y *= inv * gn.y; v.z *= inv * gn.z; v.w *= inv * gn.w;
    if (xn) put4<T>(xn + base + i, xn_ps, v);
    if (hn) *reinterpret_cast<float4*>(hn + base + i) = v;
  }
}
// Many rows: one CTA of at most 512 threads per row, P pieces per thread in registers, two CTAs per SM.  (With the kernel above,
// 1024 threads at 64 registers, one CTA fills an SM and 512 rows run as four latencies one after the other: 20 us at 512 x 4096, here 12.)
constexpr int NORM_ROW_THREADS = 512;
template <typename T, int P>
__global__ void __launch_bounds__(NORM_ROW_THREADS, 2) residual_rmsnorm_rows_kernel(const float* res, const float* part, SplitDesc sd,
                                                                                 float* x_out, const T* __restrict__ gain, T* __restrict__ xn, size_t xn_ps,
                                                                                 float* __restrict__ hn, int d, float eps) {
  pdl_trigger();
  __shared__ float s_ss[NORM_ROW_THREADS / 32];
  const int row = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5, i0 = threadIdx.x * 4, di = blockDim.x * 4;
  const size_t base = (size_t)row * d;
  int ns[P], mx = 0;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    ns[p] = part && i0 + p * di < d ? split_count(sd, row, i0 + p * di) : 0;
    mx = max(mx, ns[p]);
  }
  pdl_wait();
  float4 v[P];
#pragma unroll
  for (int p = 0; p < P; ++p)
    v[p] = res && i0 + p * di < d ? *reinterpret_cast<const float4*>(res + base + i0 + p * di) : make_float4(0.f, 0.f, 0.f, 0.f);
  const float* src = part + base + i0;
  float4 acc[P];
#pragma unroll
  for (int p = 0; p < P; ++p) acc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
  for (int s = 0; s < mx; ++s) {
    float4 u[P];
#pragma unroll
    for (int p = 0; p < P; ++p) u[p] = s < ns[p] ? __ldcg(reinterpret_cast<const float4*>(src + s * sd.stride + p * di)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int p = 0; p < P; ++p) { acc[p].x += u[p].x; acc[p].y += u[p].y; acc[p].z += u[p].z; acc[p].w += u[p].w; }
  }
  float ss = 0.f;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    if (i0 + p * di >= d) continue;
    v[p].x += acc[p].x; v[p].y += acc[p].y; v[p].z += acc[p].z; v[p].w += acc[p].w;
    *reinterpret_cast<float4*>(x_out + base + i0 + p * di) = v[p];
    ss += v[p].x * v[p].x + v[p].y * v[p].y + v[p].z * v[p].z + v[p].w * v[p].w;
  }
  if (!gain) return;
  ss = warp_sum(ss);
  if (lane == 0) s_ss[warp] = ss;
  __syncthreads();
  const float inv = rsqrtf(warp_sum(lane < nw ? s_ss[lane] : 0.f) / (float)d + eps);
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int i = i0 + p * di;
    if (i >= d) continue;
    const float4 gn = load4<T>(gain + i);
    const float4 y = make_float4(v[p].x * (inv * gn.x), v[p].y * (inv * gn.y), v[p].z * (inv * gn.z), v[p].w * (inv * gn.w));
    if (xn) put4<T>(xn + base + i, xn_ps, y);
    if (hn) *reinterpret_cast<float4*>(hn + base + i) = y;
  }
}
template <typename T, int CS>
static cudaError_t launch_norm(int rows, int d, cudaStream_t st, const float* res, const float* part, SplitDesc sd, float* x_out,
                               const void* gain, void* xn, size_t xn_ps, float* hn, float eps) {
  int threads = (d / CS / 4 + 31) / 32 * 32;
  if (threads > NORM_THREADS) threads = NORM_THREADS;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(rows * CS); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = 0; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = CS > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, residual_rmsnorm_kernel<T, CS>, res, part, sd, x_out, (const T*)gain, (T*)xn, xn_ps, hn, d, eps);
}
template <typename T>
static void norm_dispatch(const float* res, const float* part, SplitDesc sd, float* x_out, const void* gain, void* xn, size_t xn_ps, float* hn, int rows,
                          int d, float eps, cudaStream_t st) {
  // few rows: 8, 4 or 2 CTAs per row (the columns must split into whole 16-byte pieces); many: one CTA with everything in registers
  if (rows <= 16 && d % 32 == 0) { launch_norm<T, 8>(rows, d, st, res, part, sd, x_out, gain, xn, xn_ps, hn, eps); return; }
  if (rows <= 40 && d % 16 == 0) { launch_norm<T, 4>(rows, d, st, res, part, sd, x_out, gain, xn, xn_ps, hn, eps); return; }
  // (two where that is one CTA an SM; 80 rows with two / one, the norm behind the down projection: 7B shape 4.4 / 3.7 us, 13B 8.3 / 4.8, 33B 7.7 / 6.8)
  if (2 * rows <= sm_count() && d % 8 == 0) { launch_norm<T, 2>(rows, d, st, res, part, sd, x_out, gain, xn, xn_ps, hn, eps); return; }
  const int pieces = (d / 4 + NORM_ROW_THREADS - 1) / NORM_ROW_THREADS, threads = ((d / 4 + pieces - 1) / pieces + 31) / 32 * 32;
  auto go = [&](auto kernel) {
    launch_pdl(kernel, dim3(rows), dim3(threads), 0, st, res, part, sd, x_out, (const T*)gain, (T*)xn, xn_ps, hn, d, eps);
  };
  if (pieces == 1) go(residual_rmsnorm_rows_kernel<T, 1>);
  else if (pieces == 2) go(residual_rmsnorm_rows_kernel<T, 2>);
  else if (pieces == 3) go(residual_rmsnorm_rows_kernel<T, 3>);
  else if (pieces == 4) go(residual_rmsnorm_rows_kernel<T, 4>);
  else launch_norm<T, 1>(rows, d, st, res, part, sd, x_out, gain, xn, xn_ps, hn, eps);
}
hydra_status residual_rmsnorm(const float* res, const float* part, SplitDesc sd, float* x_out,
                              const void* gain, void* xn, size_t xn_ps, float* hn, int rows, int d, float eps, int dtype,
                              cudaStream_t st) {
  if (d & 3) return HYDRA_ERR_UNSUPPORTED;
  if (dtype == 0) norm_dispatch<float>(res, part, sd, x_out, gain, xn, xn_ps, hn, rows, d, eps, st);
  else norm_dispatch<bf16>(res, part, sd, x_out, gain, xn, xn_ps, hn, rows, d, eps, st);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// ------------------------------------------------------------------------------------------------
// Rotary table + QKV post-processing (sum partials, rotate q and k, append K,V to the cache)
// ------------------------------------------------------------------------------------------------
// The first kernel of every forward call: the rotary table of its rows and, where they come as tokens, their embeddings.  It lets its successors start only
// AFTER it has waited for everything before it (trigger after wait): no kernel of this call can be resident, however early the following launches are, while a
// kernel of an earlier call (the acceptance kernel that wrote the lengths, the kernels that filled the committed cache
// rows) is still running.  The early cache fetches of the attention kernel rely on that.
template <typename T>
__global__ void forward_start_kernel(RowSet rs, float2* __restrict__ table, int half, float theta, const T* __restrict__ embed, const int* tok, float* __restrict__ x, int d,
                                     int vocab, int* status) {
  pdl_wait();
  pdl_trigger();
  const int r = blockIdx.x;
  if (tok) {
    int t = tok[r];
    if (t < 0 || t >= vocab) { if (threadIdx.x == 0) atomicOr(status, ST_BOUNDS); t = 0; }
    const T* e = embed + (size_t)t * d;
    for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4) *reinterpret_cast<float4*>(x + (size_t)r * d + i) = load4<T>(e + i);   // d % 4 == 0
  }
  int pos;
  if (rs.row_at) pos = rs.row_at[r].y;
  else pos = rs.pos0[r / rs.tc] + rs.depth[r % rs.tc];
  for (int j = threadIdx.x; j < half; j += blockDim.x) {
    double inv = exp2(-((double)j / (double)half) * log2((double)theta));
    double s, c;
    sincos((double)pos * inv, &s, &c);
    table[(size_t)r * half + j] = make_float2((float)c, (float)s);
  }
}
hydra_status forward_start(RowSet rs, float2* table, int head_dim, float theta, const void* embed, const int* tok, float* x, int d, int vocab, int dtype, int* status,
                           cudaStream_t st) {
  const dim3 threads(tok ? 256 : 64);
  if (dtype == 0) launch_pdl(forward_start_kernel<float>, dim3(rs.rows()), threads, 0, st, rs, table, head_dim / 2, theta, (const float*)embed, tok, x, d, vocab, status);
  else launch_pdl(forward_start_kernel<bf16>, dim3(rs.rows()), threads, 0, st, rs, table, head_dim / 2, theta, (const bf16*)embed, tok, x, d, vocab, status);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// One thread takes four consecutive pairs (j..j+3, j+half..j+half+3) of one head of q, k or v (blockIdx.z): q and k are rotated,
// k and v appended to the cache; all loads and stores are 16 bytes wide.  Three short threads instead of one long one: the sums
// of two pieces leave registers for twice the warps (512 rows of 32 heads: 23 us with one thread for q, k and v, 17 so), and 64 rows spread over
// more SMs.  What the call's earlier kernels cannot change - slot counts, lengths, row table - is read before the wait (the
// lengths are stable within a forward call, see forward_start_kernel).
// (The float path does this in its product: float_path.cu.)
// first = 1: the projection has no q columns (a layer of which only the cache rows are wanted).
__global__ void __launch_bounds__(128) qkv_rope_store_kernel(const float* part, SplitDesc sd,
                                                             const float2* table, __half* __restrict__ q, size_t q_ps,
                                                             __half* __restrict__ kc, __half* __restrict__ vc, size_t kv_ps,
                                                             RowSet rs, int H, int hd, int max_seq, int first,
                                                             int* status) {
  pdl_trigger();
  const int r = blockIdx.x, which = blockIdx.z + first;
  const int d = H * hd, half = hd >> 1, cols = (3 - first) * d;
  const int tph = half >> 2;                                       // threads per head
  const int h = blockIdx.y * (blockDim.x / tph) + threadIdx.x / tph;
  const int j = (threadIdx.x % tph) * 4;
  const int c0 = blockIdx.z * d + h * hd + j;
  const size_t off[2] = {(size_t)r * cols + c0, (size_t)r * cols + c0 + half};
  const int ns[2] = {split_count(sd, r, c0), split_count(sd, r, c0 + half)};
  int b, slot;
  bool live = h < H;
  if (rs.row_at) {
    const int2 at = rs.row_at[r];
    b = at.x; slot = at.y;
  } else {
    const int i = r % rs.tc;
    b = r / rs.tc;
    live = live && i < (rs.n_rows ? rs.n_rows[b] : rs.tc);
    slot = rs.pos0[b] + i;
  }
  const bool in_range = slot >= 0 && slot < max_seq;
  pdl_wait();
  if (!live) return;
  if (!in_range) { if (threadIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) atomicOr(status, ST_BOUNDS); return; }
  const float4 t01 = *reinterpret_cast<const float4*>(table + (size_t)r * half + j);        // (cos, sin) of j, j+1
  const float4 t23 = *reinterpret_cast<const float4*>(table + (size_t)r * half + j + 2);    // (cos, sin) of j+2, j+3
  float4 v2[2];
  sum_slots_multi<2>(part, sd.stride, off, ns, v2);
  if (which < 2) {
    const float cs[4] = {t01.x, t01.z, t23.x, t23.z}, sn[4] = {t01.y, t01.w, t23.y, t23.w};
    const float av[4] = {v2[0].x, v2[0].y, v2[0].z, v2[0].w}, bv[4] = {v2[1].x, v2[1].y, v2[1].z, v2[1].w};
    float l[4], hh[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) { l[e] = av[e] * cs[e] - bv[e] * sn[e]; hh[e] = bv[e] * cs[e] + av[e] * sn[e]; }
    v2[0] = make_float4(l[0], l[1], l[2], l[3]); v2[1] = make_float4(hh[0], hh[1], hh[2], hh[3]);
  }
  __half* dst = which == 0 ? q + (size_t)r * d + h * hd : (which == 1 ? kc : vc) + (((size_t)b * H + h) * max_seq + slot) * hd;
  const size_t ps = which == 0 ? q_ps : kv_ps;
  put4h(dst + j, ps, v2[0]);
  put4h(dst + j + half, ps, v2[1]);
}
hydra_status qkv_rope_store(const float* part, SplitDesc sd, const float2* table, void* q, size_t q_ps, void* kcache, void* vcache,
                            size_t kv_ps, RowSet rs, int H, int hd, int max_seq, bool kv_only, int* status, cudaStream_t st) {
  const int first = kv_only ? 1 : 0;
  if (hd % 8 || 128 % (hd / 8)) return HYDRA_ERR_UNSUPPORTED;
  const int heads_per_block = 128 / (hd / 8);
  dim3 grid(rs.rows(), (H + heads_per_block - 1) / heads_per_block, 3 - first);
  launch_pdl(qkv_rope_store_kernel, grid, dim3(128), 0, st, part, sd, table, (__half*)q, q_ps, (__half*)kcache, (__half*)vcache, kv_ps, rs, H, hd, max_seq, first, status);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// ------------------------------------------------------------------------------------------------
// Tree attention of the float path, split over the KV length and the query rows.  One CTA per (head, sequence, KV chunk, row
// group of 8 RPW rows); a warp keeps an online softmax (running max, sum, weighted V) for RPW rows.  The small decoders this
// path serves have a handful of (head, sequence) pairs and one chunk, so the time is the serial chain inside a warp: few rows
// per warp spread it over the SMs (each row group reads the chunk's K,V again, out of L2), and with a single chunk the kernel
// writes the result itself instead of leaving it to the combine kernel.  Measured at 16 rows x 4 heads x 48..80 slots: 28 us with
// eight consecutive rows per warp and the combine kernel, 10 us with one row per warp; two keys per lane shorten the chain further.
// ------------------------------------------------------------------------------------------------
constexpr int ATT_CHUNK = ATT_CHUNK_ROWS;
constexpr int ATT_TILE = 64;      // KV rows staged per iteration: two keys per lane
constexpr int ATT_WARPS = 8;

// Rows and keys of sequence b: no more rows than the call has and no key past the cache, whatever the device-side lengths say.  (A row past the
// cache is not in it: qkv_rope_store skips it and raises the status bit; the row then attends to what there is.)
struct AttSpan { int nr, p0, total; };
__device__ __forceinline__ AttSpan att_span(const RowSet& rs, int b, int max_seq) {
  const int nr = min(rs.n_rows ? rs.n_rows[b] : rs.tc, rs.tc), p0 = rs.pos0[b];
  return AttSpan{nr, p0, min(min(p0, max_seq) + nr, max_seq)};
}

// (Three CTAs an SM for eight rows a warp at head_dim 64, and bounds that the compiler takes as plain numbers: left alone, the minima in att_span changed
// the loops' code, 8 x 8 pairs x 64 rows: 66 keys 23.8 -> 27.3 us, 128 keys 23.8 -> 26.9; so 24.4 and 24.5.)
template <typename T, int HD, int RPW, bool VEC>
__global__ void __launch_bounds__(ATT_WARPS * 32, HD == 64 && RPW == 8 ? 3 : 0) tree_attn_kernel(const T* q, const T* kc,
                                                                   const T* vc, RowSet rs,
                                                                   float* __restrict__ part_o, float* __restrict__ part_ml,
                                                                   T* __restrict__ out, int H, int max_seq, int nchunks) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ float smem[];
  constexpr int KPL = HD / 32;                            // output dims per lane
  constexpr int ROWS = ATT_WARPS * RPW;                   // query rows of this CTA
  float* qs = smem;                                       // [ROWS][HD]
  float* ks = qs + ROWS * HD;                             // [ATT_TILE][HD+1]
  float* vs = ks + ATT_TILE * (HD + 1);                   // [ATT_TILE][HD]
  const int h = blockIdx.x, b = blockIdx.y, c = blockIdx.z % nchunks, r0 = blockIdx.z / nchunks * ROWS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const AttSpan span = att_span(rs, b, max_seq);
  int nr = span.nr, p0 = span.p0, total = span.total;
  asm volatile("" : "+r"(nr), "+r"(p0), "+r"(total));
  const int s0 = c * ATT_CHUNK;
  const int s1 = min(s0 + ATT_CHUNK, total);
  const int d = H * HD;
  const float scale = rsqrtf((float)HD);

  for (int e = threadIdx.x * 4; e < min(ROWS, nr - r0) * HD; e += blockDim.x * 4) {
    const float4 v = load4_at<VEC>(q + ((size_t)(b * rs.tc + r0 + e / HD)) * d + h * HD + e % HD);
    *reinterpret_cast<float4*>(qs + e) = make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale);
  }
  float m[RPW], l[RPW], o[RPW][KPL];
  uint64_t msk[RPW];
#pragma unroll
  for (int j = 0; j < RPW; ++j) {                         // row j of this warp: r0 + 8 j + warp
    m[j] = -INFINITY; l[j] = 0.f;
    const int r = r0 + j * ATT_WARPS + warp;
    msk[j] = r < nr ? rs.mask[r] : 0ull;
#pragma unroll
    for (int kk = 0; kk < KPL; ++kk) o[j][kk] = 0.f;
  }
  const T* kbase = kc + ((size_t)b * H + h) * max_seq * HD;
  const T* vbase = vc + ((size_t)b * H + h) * max_seq * HD;

  for (int t0 = s0; t0 < s1 && r0 < nr; t0 += ATT_TILE) {
    __syncthreads();
#pragma unroll
    for (int e = threadIdx.x * 4; e < ATT_TILE * HD; e += ATT_WARPS * 32 * 4) {
      const int j = e / HD, k = e % HD, slot = t0 + j;
      float4 kv = make_float4(0.f, 0.f, 0.f, 0.f), vv = kv;
      if (slot < s1) { kv = load4_at<VEC>(kbase + (size_t)slot * HD + k); vv = load4_at<VEC>(vbase + (size_t)slot * HD + k); }
      float* kd = ks + j * (HD + 1) + k;
      kd[0] = kv.x; kd[1] = kv.y; kd[2] = kv.z; kd[3] = kv.w;
      *reinterpret_cast<float4*>(vs + e) = vv;
    }
    __syncthreads();
    const int sl0 = t0 + lane, sl1 = sl0 + 32;
#pragma unroll
    for (int j = 0; j < RPW; ++j) {
      const int r = r0 + j * ATT_WARPS + warp;
      if (r >= nr) continue;
      const bool ok0 = sl0 < s1 && (sl0 < p0 || ((msk[j] >> (sl0 - p0)) & 1ull)), ok1 = sl1 < s1 && (sl1 < p0 || ((msk[j] >> (sl1 - p0)) & 1ull));
      const float* qr = qs + (r - r0) * HD;
      const float *kr0 = ks + lane * (HD + 1), *kr1 = kr0 + 32 * (HD + 1);
      float a0[2] = {0.f, 0.f}, a1[2] = {0.f, 0.f};       // two chains per key
#pragma unroll 8
      for (int k = 0; k < HD; k += 2) {
        const float2 qv = *reinterpret_cast<const float2*>(qr + k);
        a0[0] += qv.x * kr0[k]; a0[1] += qv.y * kr0[k + 1];
        a1[0] += qv.x * kr1[k]; a1[1] += qv.y * kr1[k + 1];
      }
      const float sc0 = ok0 ? a0[0] + a0[1] : -INFINITY, sc1 = ok1 ? a1[0] + a1[1] : -INFINITY;
      const float mn = fmaxf(m[j], warp_max(fmaxf(sc0, sc1)));
      if (mn == -INFINITY) continue;
      const float alpha = expf(m[j] - mn);
      const float w0 = ok0 ? expf(sc0 - mn) : 0.f, w1 = ok1 ? expf(sc1 - mn) : 0.f;
      l[j] = l[j] * alpha + warp_sum(w0 + w1);
      float acc0[KPL], acc1[KPL];
#pragma unroll
      for (int kk = 0; kk < KPL; ++kk) { acc0[kk] = o[j][kk] * alpha; acc1[kk] = 0.f; }
#pragma unroll 8
      for (int jj = 0; jj < 32; ++jj) {
        const float p0j = __shfl_sync(0xffffffffu, w0, jj), p1j = __shfl_sync(0xffffffffu, w1, jj);
#pragma unroll
        for (int kk = 0; kk < KPL; ++kk) {
          acc0[kk] += p0j * vs[jj * HD + lane + 32 * kk];
          acc1[kk] += p1j * vs[(jj + 32) * HD + lane + 32 * kk];
        }
      }
#pragma unroll
      for (int kk = 0; kk < KPL; ++kk) o[j][kk] = acc0[kk] + acc1[kk];
      m[j] = mn;
    }
  }
#pragma unroll
  for (int j = 0; j < RPW; ++j) {
    const int r = r0 + j * ATT_WARPS + warp;
    if (r >= rs.tc) continue;
    if (out) {                                            // the only chunk: normalise; rows past nr come out as zeros
      T* dst = out + (size_t)(b * rs.tc + r) * d + h * HD;
#pragma unroll
      for (int kk = 0; kk < KPL; ++kk) dst[lane + 32 * kk] = from_f<T>(r < nr ? o[j][kk] / l[j] : 0.f);
      continue;
    }
    if (r >= nr) continue;
    size_t idx = ((size_t)(b * rs.tc + r) * H + h) * nchunks + c;
#pragma unroll
    for (int kk = 0; kk < KPL; ++kk) part_o[idx * HD + lane + 32 * kk] = o[j][kk];
    if (lane == 0) { part_ml[idx * 2] = m[j]; part_ml[idx * 2 + 1] = l[j]; }
  }
}

template <typename T, int HD>
__global__ void tree_attn_combine_kernel(const float* part_o, const float* part_ml, RowSet rs,
                                         T* __restrict__ out, int H, int max_seq, int nchunks) {
  pdl_trigger();
  pdl_wait();
  const int r = blockIdx.x, h = blockIdx.y, b = r / rs.tc, i = r % rs.tc;
  const auto [nr, p0, total] = att_span(rs, b, max_seq);
  const int k = threadIdx.x;
  T* dst = out + (size_t)r * H * HD + h * HD;
  if (i >= nr) { dst[k] = from_f<T>(0.f); return; }
  const int used = min(nchunks, (total + ATT_CHUNK - 1) / ATT_CHUNK);
  size_t idx = ((size_t)r * H + h) * nchunks;
  float M = -INFINITY;
  for (int c = 0; c < used; ++c) M = fmaxf(M, part_ml[(idx + c) * 2]);
  float L = 0.f, acc = 0.f;
  for (int c = 0; c < used; ++c) {
    float mc = part_ml[(idx + c) * 2];
    if (mc == -INFINITY) continue;
    float w = expf(mc - M);
    L += part_ml[(idx + c) * 2 + 1] * w;
    acc += part_o[(idx + c) * HD + k] * w;
  }
  dst[k] = from_f<T>(acc / L);
}

// The same for short caches and few rows: R query rows per CTA, its warps share the keys out (HD / 4 lanes a key, 16 bytes of it
// each, ATT_BATCH keys of a lane group in flight), every lane group keeps an online softmax of its keys, and they meet once, in shared memory.  A row's chain
// is then a handful of keys instead of all of them; each CTA reads the K, V of its pair again, out of L2.
// AHEAD: the next keys are fetched while these are worked on, which is most of the time of a round where many CTAs share the L2.  (A cache of a round or
// two has nothing to fetch ahead, and the longer code shows: tiny float model 814 -> 821 us; four rows leave no registers for it.)
// Full caches, back to back in a graph, head_dim 64, 4 heads; the kernel above / this one without / with AHEAD: 16 rows, 80 keys 6.6 / 3.3 us; 256 keys
// 9.0 / 5.6 / 5.1; 512 keys 9.4 / 9.2 / 8.2; 4 x 16 rows, 512 keys 13.0 / 15.4 / 9.2.  Tiny float model, 8 steps: 1013 -> 872 us.
constexpr int ATT_BATCH = 4;
constexpr int ATT_FEW_KEYS = 512;
template <int HD, int R, bool VEC, bool AHEAD>
__global__ void __launch_bounds__(ATT_WARPS * 32) tree_attn_few_kernel(const float* q, const float* kc, const float* vc, RowSet rs, float* __restrict__ out,
                                                                      int H, int max_seq) {
  pdl_trigger();
  constexpr int LPK = HD / 4, KPW = 32 / LPK;              // lanes a key; keys a warp takes at once
  const int h = blockIdx.x, b = blockIdx.y, r0 = blockIdx.z * R;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane / LPK, dim = lane % LPK * 4, d = H * HD;
  __shared__ float s_m[R][ATT_WARPS], s_l[R][ATT_WARPS];
  __shared__ __align__(16) float s_o[R][ATT_WARPS][HD];
  pdl_wait();
  const auto [nr, p0, end] = att_span(rs, b, max_seq);
  const int total = r0 < nr ? end : 0;
  const float scale = rsqrtf((float)HD);
  float4 qv[R], o[R];
  float m[R], l[R];
  uint64_t msk[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const bool live = r0 + r < nr;
    qv[r] = live ? load4_at<VEC>(q + (size_t)(b * rs.tc + r0 + r) * d + h * HD + dim) : make_float4(0.f, 0.f, 0.f, 0.f);
    qv[r].x *= scale; qv[r].y *= scale; qv[r].z *= scale; qv[r].w *= scale;
    msk[r] = live ? rs.mask[r0 + r] : 0ull;
    o[r] = make_float4(0.f, 0.f, 0.f, 0.f); m[r] = -INFINITY; l[r] = 0.f;
  }
  const size_t base = ((size_t)b * H + h) * max_seq * HD + dim;
  float4 kv[ATT_BATCH], vv[ATT_BATCH];
  auto fetch = [&](int at, float4 (&k)[ATT_BATCH], float4 (&v)[ATT_BATCH]) {
#pragma unroll
    for (int u = 0; u < ATT_BATCH; ++u) {
      const int slot = at + u * ATT_WARPS * KPW;
      k[u] = v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (slot < total) { k[u] = load4_at<VEC>(kc + base + (size_t)slot * HD); v[u] = load4_at<VEC>(vc + base + (size_t)slot * HD); }
    }
  };
  constexpr int STEP = ATT_WARPS * KPW * ATT_BATCH;
  if (AHEAD) fetch(warp * KPW + sub, kv, vv);
  for (int s0 = warp * KPW + sub; s0 - sub < total; s0 += STEP) {
    float4 kn[ATT_BATCH], vn[ATT_BATCH];
    if (AHEAD) fetch(s0 + STEP, kn, vn);
    else fetch(s0, kv, vv);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float s[ATT_BATCH], mn = m[r];
#pragma unroll
      for (int u = 0; u < ATT_BATCH; ++u) s[u] = (qv[r].x * kv[u].x + qv[r].y * kv[u].y) + (qv[r].z * kv[u].z + qv[r].w * kv[u].w);
#pragma unroll
      for (int bit = LPK / 2; bit > 0; bit >>= 1)
#pragma unroll
        for (int u = 0; u < ATT_BATCH; ++u) s[u] += __shfl_xor_sync(0xffffffffu, s[u], bit);
#pragma unroll
      for (int u = 0; u < ATT_BATCH; ++u) {
        const int slot = s0 + u * ATT_WARPS * KPW;
        if (!(slot < total && (slot < p0 || ((msk[r] >> (slot - p0)) & 1ull)))) s[u] = -INFINITY;
        mn = fmaxf(mn, s[u]);
      }
      if (mn == -INFINITY) continue;
      const float alpha = expf(m[r] - mn);
      m[r] = mn;
      l[r] *= alpha; o[r].x *= alpha; o[r].y *= alpha; o[r].z *= alpha; o[r].w *= alpha;
#pragma unroll
      for (int u = 0; u < ATT_BATCH; ++u) {
        if (s[u] == -INFINITY) continue;
        const float w = expf(s[u] - mn);
        l[r] += w; o[r].x += w * vv[u].x; o[r].y += w * vv[u].y; o[r].z += w * vv[u].z; o[r].w += w * vv[u].w;
      }
    }
    if (AHEAD) {
#pragma unroll
      for (int u = 0; u < ATT_BATCH; ++u) { kv[u] = kn[u]; vv[u] = vn[u]; }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (KPW == 2) {                                        // the two halves of the warp
      const float m2 = __shfl_xor_sync(0xffffffffu, m[r], 16), M = fmaxf(m[r], m2);
      const float f = m[r] == -INFINITY ? 0.f : expf(m[r] - M);
      l[r] *= f; o[r].x *= f; o[r].y *= f; o[r].z *= f; o[r].w *= f;
      l[r] += __shfl_xor_sync(0xffffffffu, l[r], 16);
      o[r].x += __shfl_xor_sync(0xffffffffu, o[r].x, 16); o[r].y += __shfl_xor_sync(0xffffffffu, o[r].y, 16);
      o[r].z += __shfl_xor_sync(0xffffffffu, o[r].z, 16); o[r].w += __shfl_xor_sync(0xffffffffu, o[r].w, 16);
      m[r] = M;
    }
    if (lane == 0) { s_m[r][warp] = m[r]; s_l[r][warp] = l[r]; }
    if (sub == 0) *reinterpret_cast<float4*>(&s_o[r][warp][dim]) = o[r];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < R * HD; e += ATT_WARPS * 32) {
    const int r = e / HD, k = e % HD;
    if (r0 + r >= rs.tc) continue;
    float M = -INFINITY, L = 0.f, acc = 0.f;
#pragma unroll
    for (int w = 0; w < ATT_WARPS; ++w) M = fmaxf(M, s_m[r][w]);
#pragma unroll
    for (int w = 0; w < ATT_WARPS; ++w) {
      const float f = s_m[r][w] == -INFINITY ? 0.f : expf(s_m[r][w] - M);
      L += s_l[r][w] * f; acc += s_o[r][w][k] * f;
    }
    out[(size_t)(b * rs.tc + r0 + r) * d + h * HD + k] = r0 + r < nr ? acc / L : 0.f;      // rows past nr come out as zeros
  }
}

size_t attention_scratch_bytes(int batch, int tc, int n_heads, int head_dim, int max_seq) {
  size_t nchunks = (size_t)(max_seq + ATT_CHUNK - 1) / ATT_CHUNK;
  return (size_t)batch * tc * n_heads * nchunks * (head_dim + 2) * sizeof(float);
}

template <typename T, int HD, int RPW, bool VEC = true>
static hydra_status launch_tree_attn(const T* q, const T* kc, const T* vc, RowSet rs, float* part_o, float* part_ml, T* out, int H, int max_seq,
                                     int nchunks, cudaStream_t st) {
  const size_t smem = (size_t)(ATT_WARPS * RPW * HD + ATT_TILE * (HD + 1) + ATT_TILE * HD) * sizeof(float);
  static PerDeviceFlag attr_done;
  if (!attr_done.get()) {
    HYDRA_CUDA(cudaFuncSetAttribute(tree_attn_kernel<T, HD, RPW, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    attr_done.set();
  }
  const int groups = (rs.tc + ATT_WARPS * RPW - 1) / (ATT_WARPS * RPW);
  launch_pdl(tree_attn_kernel<T, HD, RPW, VEC>, dim3(H, rs.batch, nchunks * groups), dim3(ATT_WARPS * 32), smem, st, q, kc, vc, rs, part_o, part_ml,
             nchunks == 1 ? out : (T*)nullptr, H, max_seq, nchunks);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

template <typename T, int HD>
static hydra_status tree_attention_t(const T* q, const T* kc, const T* vc, RowSet rs, T* out, float* scratch, int H,
                                     int max_seq, int len_upper, cudaStream_t st) {
  int nchunks_max = (max_seq + ATT_CHUNK - 1) / ATT_CHUNK;
  int nchunks = (len_upper + ATT_CHUNK - 1) / ATT_CHUNK;
  if (nchunks < 1) nchunks = 1;
  if (nchunks > nchunks_max) nchunks = nchunks_max;
  size_t rows = (size_t)rs.batch * rs.tc;
  float* part_o = scratch;
  float* part_ml = scratch + rows * H * nchunks_max * HD;
  // one row per warp while that leaves at most two CTAs per SM; more rows per warp share the staged K,V tile instead
  const long ctas1 = (long)H * rs.batch * nchunks * ((rs.tc + ATT_WARPS - 1) / ATT_WARPS), cap = 2L * sm_count();
  // Short caches: the keys of a row shared out over the warps of a CTA, with the fewest rows a CTA that leave two CTAs per SM, or four rows and up to four
  // CTAs, which pay from the second chunk on (head_dim 64, 2 x 64 rows x 4 heads: two rows a CTA, 80 keys 7.3 us with a chunk per CTA and the combine
  // kernel, 5.6 so, 256 keys 10.5 and 8.4; 4 x 64 rows, four a CTA, 256 keys 15.3 and 12.7).  len_upper bounds lengths that only the device knows, and a
  // CTA's chain follows the length.  Timed from 1 to 8 sequences, 2 to 8 heads, 1 to 64 rows and 66 to 512 keys, nothing at head_dim 64 is slower than with
  // chunks, at any length.  At head_dim 128 nothing is up to 384 keys; the full 512 take 1.04 to 1.31 as long (4 x 16 rows x 4 heads 13.3 -> 16.9 us), 256 and
  // 80 keys under the same bound a half and a third, so the line stays at 512 there too.
  // (The stand-alone call takes operands on any element boundary; loads of one element then, the same sums.)
  const bool vec = on_vec4(q) && on_vec4(kc) && on_vec4(vc);
  const long pairs = (long)H * rs.batch;
  const int R = pairs * rs.tc <= cap ? 1 : pairs * ((rs.tc + 1) / 2) <= cap ? 2 : len_upper > ATT_CHUNK && pairs * ((rs.tc + 3) / 4) <= 2 * cap ? 4 : 0;
  if (R && len_upper <= ATT_FEW_KEYS) {
    // (head_dim 128 and few CTAs: the L2 answers as fast as they ask; 16 rows x 4 heads, 256 keys 8.4 us without, 8.9 with)
    const bool ahead = len_upper > ATT_CHUNK && (HD == 64 || pairs * ((rs.tc + R - 1) / R) > sm_count() / 2);
    auto go = [&](auto kernel, auto scalar) {
      launch_pdl(vec ? kernel : scalar, dim3(H, rs.batch, (rs.tc + R - 1) / R), dim3(ATT_WARPS * 32), 0, st, q, kc, vc, rs, out, H, max_seq);
    };
    if (R == 1 && ahead) go(tree_attn_few_kernel<HD, 1, true, true>, tree_attn_few_kernel<HD, 1, false, true>);
    else if (R == 1) go(tree_attn_few_kernel<HD, 1, true, false>, tree_attn_few_kernel<HD, 1, false, false>);
    else if (R == 2 && ahead) go(tree_attn_few_kernel<HD, 2, true, true>, tree_attn_few_kernel<HD, 2, false, true>);
    else if (R == 2) go(tree_attn_few_kernel<HD, 2, true, false>, tree_attn_few_kernel<HD, 2, false, false>);
    else go(tree_attn_few_kernel<HD, 4, true, false>, tree_attn_few_kernel<HD, 4, false, false>);
    HYDRA_LAUNCH_CHECK();
    return HYDRA_OK;
  }
  if (!vec) HYDRA_TRY((launch_tree_attn<T, HD, 8, false>(q, kc, vc, rs, part_o, part_ml, out, H, max_seq, nchunks, st)));
  else if (ctas1 <= cap) HYDRA_TRY((launch_tree_attn<T, HD, 1>(q, kc, vc, rs, part_o, part_ml, out, H, max_seq, nchunks, st)));
  else if (ctas1 <= 2 * cap) HYDRA_TRY((launch_tree_attn<T, HD, 2>(q, kc, vc, rs, part_o, part_ml, out, H, max_seq, nchunks, st)));
  else HYDRA_TRY((launch_tree_attn<T, HD, 8>(q, kc, vc, rs, part_o, part_ml, out, H, max_seq, nchunks, st)));
  if (nchunks == 1) return HYDRA_OK;
  launch_pdl(tree_attn_combine_kernel<T, HD>, dim3(dim3((unsigned)rows, H)), dim3(HD), 0, st, part_o, part_ml, rs, out, H, max_seq, nchunks);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

hydra_status tree_attention_f32(const float* q, const float* kc, const float* vc, RowSet rs, float* out, void* scratch, int H, int hd,
                                int max_seq, int len_upper, cudaStream_t st) {
  if (rs.tc > 64 || !rs.mask) return HYDRA_ERR_UNSUPPORTED;
  if (hd == 64) return tree_attention_t<float, 64>(q, kc, vc, rs, out, (float*)scratch, H, max_seq, len_upper, st);
  if (hd == 128) return tree_attention_t<float, 128>(q, kc, vc, rs, out, (float*)scratch, H, max_seq, len_upper, st);
  return HYDRA_ERR_UNSUPPORTED;
}

// ------------------------------------------------------------------------------------------------
// SiLU(gate) * up from the gate/up partial sums: four columns a thread, rows on the grid's y, so that nothing but the slot counts is
// worked out and that before the wait (512 x 11008: 28 us with a flat index divided by the row length, 21 so; 64 rows: 6.0 and 3.5)
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) silu_mul_kernel(const float* part, SplitDesc sd, bf16* __restrict__ act, size_t act_ps, int f) {
  pdl_trigger();
  const int r = blockIdx.y, c = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
  const size_t off[2] = {(size_t)r * 2 * f + c, (size_t)r * 2 * f + f + c};
  const int ns[2] = {split_count(sd, r, c), split_count(sd, r, f + c)};
  pdl_wait();
  if (c >= f) return;
  float4 gu[2];
  sum_slots_multi<2, 4>(part, sd.stride, off, ns, gu);     // the widest output: few CTAs, hence few slots, per tile
  const float4 g = gu[0], u = gu[1];
  put4<bf16>(act + (size_t)r * f + c, act_ps, make_float4(silu_f(g.x) * u.x, silu_f(g.y) * u.y, silu_f(g.z) * u.z, silu_f(g.w) * u.w));
}
hydra_status silu_mul(const float* part, SplitDesc sd, void* act, size_t act_ps, int rows, int f, cudaStream_t st) {
  if (f & 3) return HYDRA_ERR_UNSUPPORTED;
  const dim3 grid((f / 4 + 255) / 256, rows);
  launch_pdl(silu_mul_kernel, grid, dim3(256), 0, st, part, sd, (bf16*)act, act_ps, f);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// ------------------------------------------------------------------------------------------------
// argmax / top-k with total order (value descending, token id ascending)
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ bool better(float v, int i, float bv, int bi) { return v > bv || (v == bv && i < bi); }

// The best (value, index) of a warp, in every lane.
__device__ __forceinline__ void warp_best(float& v, int& i) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float ov = __shfl_xor_sync(0xffffffffu, v, o);
    int oi = __shfl_xor_sync(0xffffffffu, i, o);
    if (better(ov, oi, v, i)) { v = ov; i = oi; }
  }
}

// Top-c of every logits row in two stages.  Stage 1: grid (rows, blocks of TOPK_SPAN columns); each block sums the
// partial slots of its columns (optionally storing the sums as the row's logits); every warp then picks the c best of
// its register-resident values in c rounds of a warp-wide reduction (no block barrier inside the rounds), and one warp
// merges the eight sorted lists.  Stage 2: one warp per winner list merges the sorted candidate lists of all column
// blocks out of shared memory and writes the winners (children of a tree node, or the argmax).
constexpr int TOPK_SPAN = 2048;           // columns per stage-1 block (8 per thread)
constexpr int TOPK_MAX = 64;              // a tree node has at most 63 children
constexpr int ARGMAX_CTAS_PER_SM = 8;
constexpr int TOPK_LISTS_PER_LANE = 4;    // stage 2: at most 128 column blocks (262144 tokens)

// out (a vocabulary of one column block): the block's list is the row's, and the winners go where stage 2 would have put them.
__global__ void __launch_bounds__(256) topk_stage1_kernel(const float* part, SplitDesc sd,
                                                          float* __restrict__ logits_out, float* __restrict__ cand_v,
                                                          int* __restrict__ cand_i, int vocab, int c, LevelDesc lv, const int* __restrict__ first_child,
                                                          const int* __restrict__ n_child, int* __restrict__ out, int T) {
  pdl_trigger();
  __shared__ float wv[8][TOPK_MAX];
  __shared__ int wi[8][TOPK_MAX];
  const int row = blockIdx.x, blk = blockIdx.y, nblk = gridDim.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float v[8]; int idx[8], ns[8], ns_max = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int col = blk * TOPK_SPAN + j * 256 + threadIdx.x;
    ns[j] = col < vocab ? split_count(sd, row, col) : 0;
    idx[j] = col < vocab ? col : 0x7fffffff;
    v[j] = col < vocab ? 0.f : -INFINITY;
    ns_max = max(ns_max, ns[j]);
  }
  const float* src = part + (size_t)row * vocab + blk * TOPK_SPAN + threadIdx.x;
  pdl_wait();
  for (int s = 0; s < ns_max; s += 4) {                    // four slots of the eight columns in flight together
    float u[4][8];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int j = 0; j < 8; ++j) u[q][j] = s + q < ns[j] ? __ldcg(src + (s + q) * sd.stride + j * 256) : 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] += u[q][j];
  }
  if (logits_out) {
    float* dst = logits_out + (size_t)row * vocab + blk * TOPK_SPAN + threadIdx.x;
#pragma unroll
    for (int j = 0; j < 8; ++j) if (ns[j]) dst[j * 256] = v[j];
  }
  for (int t = 0; t < c; ++t) {                            // this warp's c best, in order
    float bv = -INFINITY; int bi = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < 8; ++j) if (better(v[j], idx[j], bv, bi)) { bv = v[j]; bi = idx[j]; }
    warp_best(bv, bi);
    if (lane == 0) { wv[warp][t] = bv; wi[warp][t] = bi; }
#pragma unroll
    for (int j = 0; j < 8; ++j) if (idx[j] == bi) { v[j] = -INFINITY; idx[j] = 0x7fffffff; }    // taken
  }
  __syncthreads();
  if (warp == 0) {                                         // merge: lane w < 8 walks warp w's list
    int ptr = 0, count = c;
    int* dst = out + row;
    if (out && lv.parents) {
      const int p = lv.parents[row % lv.n_parents];
      dst = out + row / lv.n_parents * T + first_child[p];
      count = n_child[p];
    }
    for (int t = 0; t < count; ++t) {
      float hv = -INFINITY; int hi = 0x7fffffff;
      if (lane < 8 && ptr < c) { hv = wv[lane][ptr]; hi = wi[lane][ptr]; }
      float bv = hv; int bi = hi;
      warp_best(bv, bi);
      if (lane == 0) {
        if (out) dst[t] = bi;
        else { cand_v[((size_t)row * nblk + blk) * TOPK_MAX + t] = bv; cand_i[((size_t)row * nblk + blk) * TOPK_MAX + t] = bi; }
      }
      if (hi == bi && bi != 0x7fffffff) ++ptr;
    }
  }
}

// Stage 1 of an argmax: each CTA runs over every gridDim.y-th span of a row, 16 bytes of a slot at a time, and keeps its best in registers, so a
// CTA's end (the shuffles, a barrier, its candidate) is paid once a row part and not once 2048 columns.
// 512 rows of 32000: 69 -> 28 us; 128 rows 9.0 -> 7.7.
__global__ void __launch_bounds__(256) argmax_stage1_kernel(const float* part, SplitDesc sd, float* __restrict__ logits_out, float* __restrict__ cand_v,
                                                            int* __restrict__ cand_i, int vocab) {
  pdl_trigger();
  __shared__ float wv[8];
  __shared__ int wi[8];
  const int row = blockIdx.x, blk = blockIdx.y, nblk = gridDim.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t base = (size_t)row * vocab;
  float bv = -INFINITY; int bi = 0x7fffffff;
  pdl_wait();
  for (int span = blk * TOPK_SPAN; span < vocab; span += nblk * TOPK_SPAN) {
    size_t off[2]; int ns[2], col[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      col[j] = span + j * 1024 + threadIdx.x * 4;
      ns[j] = col[j] < vocab ? split_count(sd, row, col[j]) : 0;
      off[j] = base + col[j];
    }
    float4 v[2];
    sum_slots_multi<2, 4>(part, sd.stride, off, ns, v);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (!ns[j]) continue;
      if (logits_out) *reinterpret_cast<float4*>(logits_out + off[j]) = v[j];
      const float e[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) if (better(e[k], col[j] + k, bv, bi)) { bv = e[k]; bi = col[j] + k; }
    }
  }
  warp_best(bv, bi);
  if (lane == 0) { wv[warp] = bv; wi[warp] = bi; }
  __syncthreads();
  if (warp == 0) {
    bv = lane < 8 ? wv[lane] : -INFINITY; bi = lane < 8 ? wi[lane] : 0x7fffffff;
    warp_best(bv, bi);
    if (lane == 0) { cand_v[((size_t)row * nblk + blk) * TOPK_MAX] = bv; cand_i[((size_t)row * nblk + blk) * TOPK_MAX] = bi; }
  }
}

// out_of(row) and count_of(row): where the winners go.  lv.parents == null: argmax (one winner per row to amax[row]).
// One warp per winner list; dynamic shared memory: nblk * c (value, index) pairs.  depth (sequentially independent heads): the parents of all levels at once; those at
// depth t of sequence b share candidate row (top - t) * batch + b.
__global__ void __launch_bounds__(32) topk_stage2_kernel(const float* cand_v, const int* cand_i,
                                                         int nblk, int c, LevelDesc lv, const int* __restrict__ first_child,
                                                         const int* __restrict__ n_child, int* __restrict__ out, int T, const int* depth, int top, int batch) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ float s_cand[];
  float* sv = s_cand;
  int* si = reinterpret_cast<int*>(s_cand + nblk * c);
  const int row = blockIdx.x, lane = threadIdx.x;
  int* dst = out + row;
  int count = 1, crow = row;                               // crow: row of the candidate lists
  if (lv.parents) {
    const int b = row / lv.n_parents, p = lv.parents[row % lv.n_parents];
    dst = out + b * T + first_child[p];
    count = n_child[p];
    if (depth) crow = (top - depth[p]) * batch + b;
  }
  for (int e = lane; e < nblk * c; e += 32) {
    const size_t at = ((size_t)crow * nblk + e / c) * TOPK_MAX + e % c;
    sv[e] = cand_v[at]; si[e] = cand_i[at];
  }
  __syncwarp();
  int ptr[TOPK_LISTS_PER_LANE];                            // lane l walks the sorted lists l, l + 32, ...
#pragma unroll
  for (int q = 0; q < TOPK_LISTS_PER_LANE; ++q) ptr[q] = 0;
  for (int t = 0; t < count; ++t) {
    float bv = -INFINITY; int bi = 0x7fffffff;
#pragma unroll
    for (int q = 0; q < TOPK_LISTS_PER_LANE; ++q) {
      const int l = lane + 32 * q;
      if (l < nblk && ptr[q] < c && better(sv[l * c + ptr[q]], si[l * c + ptr[q]], bv, bi)) { bv = sv[l * c + ptr[q]]; bi = si[l * c + ptr[q]]; }
    }
    warp_best(bv, bi);
    if (lane == 0) dst[t] = bi;
#pragma unroll
    for (int q = 0; q < TOPK_LISTS_PER_LANE; ++q) {
      const int l = lane + 32 * q;
      if (l < nblk && ptr[q] < c && si[l * c + ptr[q]] == bi && bi != 0x7fffffff) ++ptr[q];
    }
  }
}

size_t topk_scratch_bytes(int rows, int vocab) {
  const size_t nblk = (size_t)(vocab + TOPK_SPAN - 1) / TOPK_SPAN;
  return (size_t)rows * nblk * TOPK_MAX * (sizeof(float) + sizeof(int));
}

struct TopkPlan { int nblk; float* cand_v; int* cand_i; };
static bool topk_plan(void* scratch, int rows_cap, int rows, int vocab, int c, TopkPlan* p) {
  if (c < 1 || c > TOPK_MAX || rows > rows_cap || rows < 1) return false;
  p->nblk = (vocab + TOPK_SPAN - 1) / TOPK_SPAN;
  if (p->nblk > 32 * TOPK_LISTS_PER_LANE || (size_t)p->nblk * c * 8 > 48 * 1024) return false;      // stage 2 keeps every candidate of a row in shared memory
  p->cand_v = (float*)scratch;
  p->cand_i = (int*)(p->cand_v + (size_t)rows_cap * p->nblk * TOPK_MAX);
  return true;
}

hydra_status argmax_rows(const float* part, SplitDesc sd, float* logits_out, int* amax, void* scratch, int rows_cap, int rows,
                         int vocab, cudaStream_t st) {
  TopkPlan p;
  if (!topk_plan(scratch, rows_cap, rows, vocab, 1, &p)) return HYDRA_ERR_UNSUPPORTED;
  int* direct = p.nblk == 1 ? amax : nullptr;
  // CTAs enough for eight per SM: rows that are that many have runs of several spans (75 rows and up at a vocabulary of 32000)
  const int runs = std::max(1, std::min(p.nblk, ARGMAX_CTAS_PER_SM * sm_count() / rows));
  if (vocab % 4 == 0 && runs < p.nblk && on_vec4(part) && on_vec4(logits_out) && sd.stride % 4 == 0) {
    p.nblk = runs;
    launch_pdl(argmax_stage1_kernel, dim3(rows, p.nblk), dim3(256), 0, st, part, sd, logits_out, p.cand_v, p.cand_i, vocab);
  } else {
    launch_pdl(topk_stage1_kernel, dim3(rows, p.nblk), dim3(256), 0, st, part, sd, logits_out, p.cand_v, p.cand_i, vocab, 1, LevelDesc{0, 0, nullptr},
               (const int*)nullptr, (const int*)nullptr, direct, 0);
  }
  HYDRA_LAUNCH_CHECK();
  if (direct) return HYDRA_OK;
  launch_pdl(topk_stage2_kernel, dim3(rows), dim3(32), (size_t)p.nblk * 8, st, (const float*)p.cand_v, (const int*)p.cand_i, p.nblk, 1, LevelDesc{0, 0, nullptr},
             (const int*)nullptr, (const int*)nullptr, amax, 0, (const int*)nullptr, 0, 0);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

hydra_status topk_candidates(const float* part, SplitDesc sd, float* logits, int max_children, void* scratch, int rows_cap, int rows, int vocab, cudaStream_t st) {
  TopkPlan p;
  if (!topk_plan(scratch, rows_cap, rows, vocab, max_children, &p)) return HYDRA_ERR_UNSUPPORTED;
  launch_pdl(topk_stage1_kernel, dim3(rows, p.nblk), dim3(256), 0, st, part, sd, logits, p.cand_v, p.cand_i, vocab, max_children, LevelDesc{0, 0, nullptr},
             (const int*)nullptr, (const int*)nullptr, (int*)nullptr, 0);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

hydra_status topk_children(const float* part, SplitDesc sd, float* logits, LevelDesc lv, int max_children, const int* first_child, const int* n_child,
                           int* tree_tok, void* scratch, int rows_cap, int batch, int T, int vocab, cudaStream_t st) {
  TopkPlan p;
  const int rows = batch * lv.n_parents;
  if (!topk_plan(scratch, rows_cap, rows, vocab, max_children, &p)) return HYDRA_ERR_UNSUPPORTED;
  // one column block: its list is the row's, and a launch of a chain of short ones goes (tiny float model, 8 steps: 872 -> 813 us)
  if (p.nblk == 1) {
    launch_pdl(topk_stage1_kernel, dim3(rows, 1), dim3(256), 0, st, part, sd, logits, p.cand_v, p.cand_i, vocab, max_children, lv, first_child, n_child, tree_tok, T);
    HYDRA_LAUNCH_CHECK();
    return HYDRA_OK;
  }
  HYDRA_TRY(topk_candidates(part, sd, logits, max_children, scratch, rows_cap, rows, vocab, st));
  return topk_merge(lv, max_children, first_child, n_child, tree_tok, scratch, rows_cap, rows, batch, T, vocab, nullptr, 0, st);
}

hydra_status topk_merge(LevelDesc lv, int max_children, const int* first_child, const int* n_child, int* tree_tok, void* scratch, int rows_cap, int cand_rows,
                        int batch, int T, int vocab, const int* depth, int top, cudaStream_t st) {
  TopkPlan p;
  if (!topk_plan(scratch, rows_cap, cand_rows, vocab, max_children, &p)) return HYDRA_ERR_UNSUPPORTED;
  launch_pdl(topk_stage2_kernel, dim3(batch * lv.n_parents), dim3(32), (size_t)p.nblk * max_children * 8, st, (const float*)p.cand_v, (const int*)p.cand_i, p.nblk,
             max_children, lv, first_child, n_child, tree_tok, T, depth, top, batch);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// ------------------------------------------------------------------------------------------------
// Draft heads (bfloat16 path): input gather and the residual SiLU layer epilogue
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) head_gather_kernel(const float* hprime, const bf16* __restrict__ embed,
                                                          const int* root_tok, int* tree_tok,
                                                          const int* __restrict__ path_tab, LevelDesc lv, int write_root, bf16* __restrict__ z,
                                                          size_t z_ps, int T_rows, int kp1, int d_model, int vocab, int* status) {
  pdl_trigger();
  pdl_wait();
  const int row = blockIdx.x, b = row / lv.n_parents, j = row % lv.n_parents;
  const int blk = blockIdx.y;                               // 0: hidden, 1..d: path tokens root..parent
  const int p = lv.parents[j];
  bf16* dst = z + ((size_t)row * (lv.d + 1) + blk) * d_model;
  if (blk == 0) {                                          // 16-byte pieces (d_model is a multiple of 4)
    for (int i = threadIdx.x * 4; i < d_model; i += blockDim.x * 4)
      put4<bf16>(dst + i, z_ps, *reinterpret_cast<const float4*>(hprime + (size_t)b * d_model + i));
    if (write_root && j == 0 && threadIdx.x == 0) tree_tok[b * T_rows] = root_tok[b];
    return;
  }
  int node = path_tab[p * kp1 + (blk - 1)];
  int t = node == 0 ? root_tok[b] : tree_tok[b * T_rows + node];
  if (t < 0 || t >= vocab) { if (threadIdx.x == 0) atomicOr(status, ST_BOUNDS); t = 0; }
  const bf16* e = embed + (size_t)t * d_model;
  for (int i = threadIdx.x * 4; i < d_model; i += blockDim.x * 4) put4<bf16>(dst + i, z_ps, load4<bf16>(e + i));      // embeddings are exact: lo = 0
}
hydra_status head_gather(const float* hprime, const void* embed, const int* root_tok, int* tree_tok, const int* path_tab,
                         LevelDesc lv, int write_root, void* z, size_t z_ps, int batch, int T, int kp1, int d_model, int vocab,
                         int* status, cudaStream_t st) {
  dim3 grid(batch * lv.n_parents, lv.d + 1);
  launch_pdl(head_gather_kernel, grid, dim3(256), 0, st, hprime, (const bf16*)embed, root_tok, tree_tok, path_tab, lv, write_root,
               (bf16*)z, z_ps, T, kp1, d_model, vocab, status);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// Four columns per thread in small CTAs (a level has 1 to a few dozen rows); the bias and the slot counts before the wait.
// VEC: the bias, a caller's vector, lies on a boundary of four elements.
constexpr int HEAD_ACT_THREADS = 64;
template <bool VEC>
__global__ void __launch_bounds__(HEAD_ACT_THREADS) head_act_kernel(const float* res, int res_is_hprime, int rows_per_b, const float* part,
                                SplitDesc sd, const bf16* __restrict__ bias, float* y_out, bf16* __restrict__ yb, size_t yb_ps,
                                int rows, int d) {
  pdl_trigger();
  const int d4 = d / 4, p = blockIdx.x * blockDim.x + threadIdx.x, r = p / d4, c = (p - r * d4) * 4;
  const size_t off[1] = {(size_t)r * d + c};
  const int ns[1] = {split_count(sd, r, c)};
  float4 v = bias ? load4_at<VEC>(bias + c) : make_float4(0.f, 0.f, 0.f, 0.f);
  const size_t at = res_is_hprime ? (size_t)(r / rows_per_b) * d + c : off[0];
  pdl_wait();
  if (r >= rows) return;
  const float4 base = *reinterpret_cast<const float4*>(res + at);
  float4 acc[1];
  sum_slots_multi<1, 12>(part, sd.stride, off, ns, acc);
  const float4 y = make_float4(base.x + silu_f(v.x + acc[0].x), base.y + silu_f(v.y + acc[0].y), base.z + silu_f(v.z + acc[0].z), base.w + silu_f(v.w + acc[0].w));
  *reinterpret_cast<float4*>(y_out + off[0]) = y;
  put4<bf16>(yb + off[0], yb_ps, y);
}
hydra_status head_act(const float* res, int res_is_hprime, int rows_per_b, const float* part, SplitDesc sd,
                      const void* bias, float* y_out, void* yb, size_t yb_ps, int rows, int d, cudaStream_t st) {
  if (d & 3) return HYDRA_ERR_UNSUPPORTED;
  const unsigned grid = (unsigned)(((size_t)rows * d / 4 + HEAD_ACT_THREADS - 1) / HEAD_ACT_THREADS);
  launch_pdl(on_vec4((const bf16*)bias) ? head_act_kernel<true> : head_act_kernel<false>, dim3(grid), dim3(HEAD_ACT_THREADS), 0, st, res, res_is_hprime, rows_per_b, part, sd,
             (const bf16*)bias, y_out, (bf16*)yb, yb_ps, rows, d);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// ------------------------------------------------------------------------------------------------
// Greedy acceptance + in-place KV compaction + state update, one kernel.
// grid (G, batch).  Every CTA recomputes the accepted path of its sequence (cheap), then moves its
// share of 16-byte KV pieces.  A thread moves its piece for k = 1..n in batches of 8 positions, reading a
// batch before writing it: the destination slot k can only be the source of a path position j <= k (a row
// at depth j has index >= j), which the same thread reads in the same or an earlier batch, before the
// write, so the in-place move is hazard-free.  The last CTA of a sequence to
// finish publishes the new length / root token; all CTAs read the old length before they signal.
// ------------------------------------------------------------------------------------------------
// Typical criterion for candidate row i of sequence b (Section "Typical acceptance sampling"): with p = softmax(l / tau) at
// the parent row and H its entropy, accept when p[token] > min(eps, alpha exp(-H)).  From the row statistics (max m,
// Z = sum exp((l - m)/tau), S = sum exp((l - m)/tau) (l - m)/tau): p[x] = exp((l_x - m)/tau) / Z, H = log Z - S / Z.
__device__ __forceinline__ bool typical_pass(const AcceptArgs& a, int b, int i) {
  const int prow = b * a.T + a.parent[i];
  const int tok = a.tree_tok[b * a.T + i];
  if (tok < 0 || tok >= a.vocab) return false;
  const float4 st = a.row_stats[prow];
  const float z = (a.logits[(size_t)prow * a.vocab + tok] - st.x) / a.tau;
  const float p = __expf(z) / st.y;
  const float H = __logf(st.y) - st.z / st.y;
  return p > fminf(a.eps, a.alpha * __expf(-H));
}

__global__ void __launch_bounds__(256) accept_compact_kernel(AcceptArgs a) {
  pdl_trigger();
  pdl_wait();
  __shared__ int s_path[72];
  __shared__ int s_n, s_best, s_bonus, s_owner, s_pick;
  __shared__ float s_scan[256], s_target, s_range[8][32][33];
  const int b = blockIdx.y;
  const int T = a.T;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    uint64_t bits = 0;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      int i = lane + 32 * half;
      bool mt = false;
      if (i >= 1 && i < T) mt = a.mode == 1 ? typical_pass(a, b, i) : a.tree_tok[b * T + i] == a.amax[b * T + a.parent[i]];
      bits |= (uint64_t)__ballot_sync(0xffffffffu, mt) << (32 * half);
    }
    if (lane == 0 && blockIdx.x == 0 && a.pass_bits) a.pass_bits[b] = bits;
    int key = -1;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      int i = lane + 32 * half;
      if (i < T) {
        bool acc = ((a.anc[i] & ~1ull) & ~bits) == 0ull;
        if (acc) key = max(key, a.depth[i] * 64 + (63 - i));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
    // walk from the best row to the root through the parents held in registers (lane i: rows i and i + 32)
    const int p_lo = lane < T ? a.parent[lane] : 0, p_hi = lane + 32 < T ? a.parent[lane + 32] : 0;
    const int best = 63 - (key & 63), n = key >> 6;
    int node = best;
    for (int k = n; k >= 0; --k) {
      if (lane == 0) s_path[k] = node;
      const int up_lo = __shfl_sync(0xffffffffu, p_lo, node & 31), up_hi = __shfl_sync(0xffffffffu, p_hi, node & 31);
      node = node < 32 ? up_lo : up_hi;
    }
    if (lane == 0) { s_n = n; s_best = best; }
  }
  __syncthreads();
  const int n = s_n, best = s_best;
  // the token after the accepted path: the best row's argmax, or (typical mode with uniform numbers) a draw from its
  // temperature distribution by inverse CDF in token-id order; only CTA 0 of the sequence works it out
  const bool sampled = a.mode == 1 && a.u != nullptr;
  if (blockIdx.x == 0) {
    if (!sampled) {
      if (threadIdx.x == 0) s_bonus = a.amax[b * T + best];
    } else {
      const float* lg = a.logits + (size_t)(b * T + best) * a.vocab;
      const float mx = a.row_stats[b * T + best].x, inv_tau = 1.f / a.tau;
      const int per = (a.vocab + 255) / 256, v0 = threadIdx.x * per, v1 = min(v0 + per, a.vocab);
      float part = 0.f;
      // A thread's range is summed in order; a warp fetches its 32 ranges 32 tokens at a time in whole lines and hands them on transposed (read
      // by their threads from memory, every load takes 32 lines).  With one thread's walk through the picked range the kernel took 35 us, now 20.
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
      for (int i0 = 0; i0 < per; i0 += 32) {
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
          const int v = (warp * 32 + j) * per + i0 + lane;
          s_range[warp][j][lane] = i0 + lane < per && v < a.vocab ? lg[v] : 0.f;
        }
        __syncwarp();
        const int cn = min(min(32, per - i0), v1 - v0 - i0);
#pragma unroll 8
        for (int i = 0; i < cn; ++i) part += __expf((s_range[warp][lane][i] - mx) * inv_tau);
        __syncwarp();
      }
      s_scan[threadIdx.x] = part;
      if (threadIdx.x == 0) { s_owner = -1; s_pick = 0x7fffffff; }
      __syncthreads();
      if (threadIdx.x == 0) {                                          // sequential scan of 256 partial sums: fixed order
        float run = 0.f;
#pragma unroll 16
        for (int t = 0; t < 256; ++t) { const float p = s_scan[t]; s_scan[t] = run; run += p; }
        s_target = a.u[b] * run;
      }
      __syncthreads();
      const float target = s_target;
      if (s_scan[threadIdx.x] <= target) atomicMax(&s_owner, (int)threadIdx.x);      // last thread whose range starts at or below the target
      __syncthreads();
      const int owner = s_owner < 0 ? 255 : s_owner, w0 = owner * per, w1 = min(w0 + per, a.vocab);
      float acc = s_scan[owner];
      int pick = -1;
      // the owner's range in the order of its sum, 256 weights at a time: worked out by all threads, added by one
      for (int c0 = w0; c0 < w1; c0 += 256) {
        const int cn = min(256, w1 - c0);
        __syncthreads();                                               // (the scan has been read)
        if (threadIdx.x < cn) s_scan[threadIdx.x] = __expf((lg[c0 + threadIdx.x] - mx) * inv_tau);
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll 8
          for (int v = 0; v < cn; ++v) { acc += s_scan[v]; if (pick < 0 && acc > target) pick = c0 + v; }
          if (pick >= 0) s_pick = pick;
        }
        __syncthreads();
        if (s_pick != 0x7fffffff) break;
      }
      const bool none = s_pick == 0x7fffffff;
      __syncthreads();
      if (none) {                                                      // rounding at a range boundary: the next token of non-zero weight
        for (int v = w1 + (int)threadIdx.x; v < a.vocab; v += 256) if (__expf((lg[v] - mx) * inv_tau) > 0.f) { atomicMin(&s_pick, v); break; }
        __syncthreads();
      }
      if (threadIdx.x == 0) s_bonus = s_pick == 0x7fffffff ? a.vocab - 1 : s_pick;
    }
    __syncthreads();
    if (threadIdx.x == 0 && a.bonus_tmp) a.bonus_tmp[b] = s_bonus;       // published with the fence before this CTA signs off below
  }
  const int L = a.len[b];
  const bool in_range = L >= 0 && L + T <= a.max_seq;
  if (!in_range) {
    if (threadIdx.x == 0) atomicOr(a.status, ST_BOUNDS);
  } else {
    const int row_bytes = a.head_dim * a.esize;
    const int ppr = row_bytes / 16;                                    // 16-byte pieces per row
    const long long units = (long long)a.n_layers * 2 * a.kv_planes * a.n_heads * ppr;
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < units; u += (long long)gridDim.x * blockDim.x) {
      int piece = (int)(u % ppr);
      long long t = u / ppr;
      int head = (int)(t % a.n_heads);
      long long lk = t / a.n_heads;                                    // (layer*2 + kv)*planes + plane
      char* base = (char*)a.kv_base + ((((size_t)lk * a.max_batch + b) * a.n_heads + head) * a.max_seq) * row_bytes;
      for (int k0 = 1; k0 <= n; k0 += 8) {                             // all reads of a batch in flight before its writes
        uint4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (k0 + j <= n) v[j] = *reinterpret_cast<const uint4*>(base + (size_t)(L + s_path[k0 + j]) * row_bytes + piece * 16);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (k0 + j <= n && s_path[k0 + j] != k0 + j) *reinterpret_cast<uint4*>(base + (size_t)(L + k0 + j) * row_bytes + piece * 16) = v[j];
      }
    }
    // hidden rows of the accepted path feed the next draft
    const int d4 = a.d_model / 4;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < (n + 1) * d4; u += gridDim.x * blockDim.x) {
      int k = u / d4, c = u % d4;
      reinterpret_cast<float4*>(a.h_new + ((size_t)b * (a.K + 1) + k) * a.d_model)[c] =
          reinterpret_cast<const float4*>(a.h_tree + ((size_t)b * a.h_tree_stride + s_path[k]) * a.d_model)[c];
    }
  }
  if (blockIdx.x == 0 && threadIdx.x <= a.K) {
    int k = threadIdx.x;
    if (a.path) a.path[b * (a.K + 1) + k] = k <= n ? s_path[k] : -1;
    if (a.out_tok) {
      int v = -1;
      if (k < n) v = a.tree_tok[b * T + s_path[k + 1]];
      else if (k == n) v = s_bonus;
      a.out_tok[b * (a.K + 1) + k] = v;
    }
    if (k == 0 && a.n_acc) a.n_acc[b] = n;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned prev = atomicAdd(&a.done_counter[b], 1u);
    if (prev == gridDim.x - 1) {
      a.done_counter[b] = 0;
      if (in_range) {
        a.len[b] = L + n + 1;
        __threadfence();
        a.root_tok[b] = a.bonus_tmp ? *((volatile int*)a.bonus_tmp + b) : a.amax[b * T + best];
        a.n_new[b] = n + 1;
      }
    }
  }
}
// (max, sum exp((l - max)/tau), sum exp((l - max)/tau) (l - max)/tau) of every logits row; one CTA per row, fixed reduction order
__global__ void __launch_bounds__(1024) softmax_row_stats_kernel(const float* logits, float4* __restrict__ stats, int vocab, float tau) {
  pdl_trigger();
  pdl_wait();
  __shared__ float sh[32];
  const float* lg = logits + (size_t)blockIdx.x * vocab;
  float mx = -INFINITY;
  for (int v = threadIdx.x; v < vocab; v += 1024) mx = fmaxf(mx, lg[v]);
  mx = warp_max(mx);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  mx = sh[0];
  for (int w = 1; w < 32; ++w) mx = fmaxf(mx, sh[w]);
  __syncthreads();
  float z_sum = 0.f, s_sum = 0.f;
  const float inv_tau = 1.f / tau;
  for (int v = threadIdx.x; v < vocab; v += 1024) {
    const float z = (lg[v] - mx) * inv_tau, e = __expf(z);
    z_sum += e; s_sum += e * z;
  }
  const float Z = block_sum(z_sum, sh), S = block_sum(s_sum, sh);
  if (threadIdx.x == 0) stats[blockIdx.x] = make_float4(mx, Z, S, 0.f);
}
hydra_status softmax_row_stats(const float* logits, float4* row_stats, int rows, int vocab, float tau, cudaStream_t st) {
  launch_pdl(softmax_row_stats_kernel, dim3(rows), dim3(1024), 0, st, logits, row_stats, vocab, tau);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

static dim3 accept_grid(const AcceptArgs& a) {
  long long units = (long long)a.n_layers * 2 * a.kv_planes * a.n_heads * (a.head_dim * a.esize / 16);
  int G = (int)((units + 255) / 256);
  int cap = (sm_count() * 4 + a.batch - 1) / a.batch;
  if (G > cap) G = cap;
  if (G < 1) G = 1;
  return dim3(G, a.batch);
}
hydra_status accept_compact(const AcceptArgs& a, cudaStream_t st) {
  launch_pdl(accept_compact_kernel, accept_grid(a), dim3(256), 0, st, a);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}
cudaError_t accept_graph_node(cudaGraph_t graph, cudaGraphNode_t* node) {
  size_t n = 0;
  cudaError_t e = cudaGraphGetNodes(graph, nullptr, &n);
  if (e != cudaSuccess) return e;
  std::vector<cudaGraphNode_t> nodes(n);
  if ((e = cudaGraphGetNodes(graph, nodes.data(), &n)) != cudaSuccess) return e;
  for (size_t i = n; i-- > 0;) {                           // the last launch of a step
    cudaGraphNodeType t;
    cudaKernelNodeParams p{};
    if ((e = cudaGraphNodeGetType(nodes[i], &t)) != cudaSuccess) return e;
    if (t != cudaGraphNodeTypeKernel) continue;
    if ((e = cudaGraphKernelNodeGetParams(nodes[i], &p)) != cudaSuccess) return e;
    if (p.func == (void*)accept_compact_kernel) { *node = nodes[i]; return cudaSuccess; }
  }
  return cudaErrorInvalidValue;
}
cudaError_t accept_graph_update(cudaGraphExec_t exec, cudaGraphNode_t node, const AcceptArgs& a) {
  AcceptArgs copy = a;
  void* args[] = {&copy};
  cudaKernelNodeParams p{};
  p.func = (void*)accept_compact_kernel; p.gridDim = accept_grid(a); p.blockDim = dim3(256); p.sharedMemBytes = 0; p.kernelParams = args;
  return cudaGraphExecKernelNodeSetParams(exec, node, &p);
}

// ------------------------------------------------------------------------------------------------
// Small state kernels
// ------------------------------------------------------------------------------------------------
__global__ void set_prompts_kernel(const PromptOffsets p, int batch, int* prompt_len, int* offsets) {
  pdl_trigger();
  pdl_wait();
  for (int i = threadIdx.x; i <= batch; i += blockDim.x) {
    offsets[i] = p.off[i];
    if (i < batch) prompt_len[i] = p.off[i + 1] - p.off[i];
  }
}
hydra_status set_prompts(const PromptOffsets& p, int batch, int* prompt_len, int* offsets, cudaStream_t st) {
  launch_pdl(set_prompts_kernel, dim3(1), dim3(MAX_BATCH + 1), 0, st, p, batch, prompt_len, offsets);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

__global__ void set_chunk_kernel(const int* prompt_len, int chunk, int tc, int* pos0, int* n_rows, int batch) {
  pdl_trigger();
  pdl_wait();
  int b = threadIdx.x;
  if (b >= batch) return;
  int rem = prompt_len[b] - chunk * tc;
  pos0[b] = rem > 0 ? chunk * tc : prompt_len[b];
  n_rows[b] = rem < 0 ? 0 : (rem > tc ? tc : rem);
}
hydra_status set_chunk(const int* prompt_len, int chunk, int tc, int* pos0, int* n_rows, int batch, cudaStream_t st) {
  launch_pdl(set_chunk_kernel, dim3(1), dim3(64), 0, st, prompt_len, chunk, tc, pos0, n_rows, batch);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

__global__ void gather_chunk_tokens_kernel(const int* tokens, const int* offsets, int chunk, int tc, int* tok_out) {
  pdl_trigger();
  pdl_wait();
  int b = blockIdx.x, i = threadIdx.x;
  if (i >= tc) return;
  int n = offsets[b + 1] - offsets[b];
  int idx = chunk * tc + i;
  tok_out[b * tc + i] = idx < n ? tokens[offsets[b] + idx] : 0;
}
hydra_status gather_chunk_tokens(const int* tokens, const int* offsets, int chunk, int tc, int* tok_out, int batch,
                                 cudaStream_t st) {
  launch_pdl(gather_chunk_tokens_kernel, dim3(batch), dim3((tc + 31) / 32 * 32), 0, st, tokens, offsets, chunk, tc, tok_out);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

__global__ void capture_last_kernel(const float* h, const int* prompt_len, int chunk, int tc, float* h_new, int kp1,
                                    int* n_new, int* len, int d) {
  pdl_trigger();
  pdl_wait();
  int b = blockIdx.x;
  int last = prompt_len[b] - 1;
  if (last < chunk * tc || last >= (chunk + 1) * tc) return;
  int i = last - chunk * tc;
  for (int c = threadIdx.x; c < d; c += blockDim.x) h_new[(size_t)b * kp1 * d + c] = h[((size_t)b * tc + i) * d + c];
  if (threadIdx.x == 0) { n_new[b] = 1; len[b] = prompt_len[b]; }
}
hydra_status capture_last(const float* h, const int* prompt_len, int chunk, int tc, float* h_new, int kp1, int* n_new,
                          int* len, int batch, int d, cudaStream_t st) {
  launch_pdl(capture_last_kernel, dim3(batch), dim3(256), 0, st, h, prompt_len, chunk, tc, h_new, kp1, n_new, len, d);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// Packed prompts: token g of the concatenated prompts (base = offsets[0]) is a slot of the sequence b whose range holds it.
__global__ void pack_rows_kernel(const int* offsets, int batch, int2* row_at, int base, int total) {
  pdl_trigger();
  pdl_wait();
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= total) return;
  int b = 0;
  while (b + 1 < batch && offsets[b + 1] - base <= g) ++b;
  row_at[g] = make_int2(b, g - (offsets[b] - base));
}
hydra_status pack_rows(const int* offsets, int batch, int2* row_at, int base, int total, cudaStream_t st) {
  launch_pdl(pack_rows_kernel, dim3((total + 255) / 256), dim3(256), 0, st, offsets, batch, row_at, base, total);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

// h holds the hidden rows of tokens g0 .. g0+rows-1 of the concatenated prompts
__global__ void capture_last_packed_kernel(const float* h, const int* offsets, int g0, int rows, float* h_new, int kp1, int* n_new,
                                           int* len, int d) {
  pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x, i = offsets[b + 1] - 1 - g0;
  if (i < 0 || i >= rows) return;
  for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4)                                  // d % 4 == 0
    *reinterpret_cast<float4*>(h_new + (size_t)b * kp1 * d + c) = *reinterpret_cast<const float4*>(h + (size_t)i * d + c);
  if (threadIdx.x == 0) { n_new[b] = 1; len[b] = offsets[b + 1] - offsets[b]; }
}
hydra_status capture_last_packed(const float* h, const int* offsets, int g0, int rows, float* h_new, int kp1, int* n_new, int* len,
                                 int batch, int d, cudaStream_t st) {
  launch_pdl(capture_last_packed_kernel, dim3(batch), dim3(256), 0, st, h, offsets, g0, rows, h_new, kp1, n_new, len, d);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

__global__ void prefix_rowset_kernel(const int* len, const int* n_new, int* pos0, int* n_rows, int batch) {
  pdl_trigger();
  pdl_wait();
  int b = threadIdx.x;
  if (b >= batch) return;
  pos0[b] = len[b] - n_new[b];
  n_rows[b] = n_new[b];
}
hydra_status prefix_rowset(const int* len, const int* n_new, int* pos0, int* n_rows, int batch, cudaStream_t st) {
  launch_pdl(prefix_rowset_kernel, dim3(1), dim3(64), 0, st, len, n_new, pos0, n_rows, batch);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

__global__ void pick_last_row_kernel(const float* x, const int* n_rows, int tc, float* hprime, int d) {
  pdl_trigger();
  pdl_wait();
  int b = blockIdx.x;
  int i = n_rows[b] - 1;
  if (i < 0) i = 0;
  for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4)                                  // d % 4 == 0
    *reinterpret_cast<float4*>(hprime + (size_t)b * d + c) = *reinterpret_cast<const float4*>(x + ((size_t)b * tc + i) * d + c);
}
hydra_status pick_last_row(const float* x, const int* n_rows, int tc, float* hprime, int batch, int d, cudaStream_t st) {
  launch_pdl(pick_last_row_kernel, dim3(batch), dim3(256), 0, st, x, n_rows, tc, hprime, d);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

__global__ void apply_plant_kernel(int* tree_tok, const int* plant, int count) {
  pdl_trigger();
  pdl_wait();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count && plant[i] >= 0) tree_tok[i] = plant[i];
}
hydra_status apply_plant(int* tree_tok, const int* plant, int count, cudaStream_t st) {
  launch_pdl(apply_plant_kernel, dim3((count + 255) / 256), dim3(256), 0, st, tree_tok, plant, count);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

template <typename T>
__global__ void cast_rows_kernel(const float* src, T* __restrict__ dst, size_t dst_ps, size_t count) {
  pdl_trigger();
  pdl_wait();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) put<T>(dst + i, dst_ps, src[i]);
}
hydra_status cast_rows(const float* src, void* dst, size_t dst_ps, size_t count, int dtype, cudaStream_t st) {
  unsigned grid = (unsigned)((count + 255) / 256);
  if (dtype == 0) launch_pdl(cast_rows_kernel<float>, dim3(grid), dim3(256), 0, st, src, (float*)dst, dst_ps, count);
  else launch_pdl(cast_rows_kernel<bf16>, dim3(grid), dim3(256), 0, st, src, (bf16*)dst, dst_ps, count);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

__global__ void copy_i32_kernel(int* dst, const int* src, int count) {
  pdl_trigger();
  pdl_wait();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) dst[i] = src[i];
}
hydra_status copy_i32(int* dst, const int* src, int count, cudaStream_t st) {
  launch_pdl(copy_i32_kernel, dim3((count + 255) / 256), dim3(256), 0, st, dst, src, count);
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

}  // namespace hydra
