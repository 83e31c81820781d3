// Attention of one or two query rows per sequence over the float16 caches of the bfloat16 model path: decoding without a tree, or with one candidate.
//
// A tensor-core tile has 128 rows whatever the call has, and its chain - tile into shared memory, scores into tensor memory, softmax, P back, product - is
// what a short cache then costs.  Here every key is a group of lanes (HD / 8, 16 bytes of each plane a lane): scores by shuffles, weights and sums in float, all of it
// in registers, straight from global memory.  16 warps a CTA share the keys of a chunk out, BATCH keys of a lane group in flight (128 KB an SM in all, which
// also keeps memory busy on long caches); the lane groups meet once in shared memory, and the chunks of a (head, sequence) pair, a cluster, in the first one's.
// Operands: hi + lo planes are added to one float (22 bits); the softmax weights stay float.  In a forward call committed keys are read ahead of the
// wait for the preceding kernel, as in attention_tc.cu.
// Alone, back to back over caches larger than the L2, two planes, 32 heads of 128, against the tensor-core kernel: one row, 1 sequence of 160 keys 7.8 -> 5.0 us, 500 9.8 ->
// 7.0, 2400 19.9 -> 17.4; 8 sequences of 160 keys 20.0 -> 15.5, 1000 51.7 -> 46.2; 40 heads, 2048 keys 26.9 -> 19.3.  A layer of 7B decoding without a tree 85.0 -> 80.5 us.
#include "launch.h"
#include <cuda_fp16.h>
#include <algorithm>
#include <type_traits>

namespace hydra {
namespace {

constexpr int WARPS = 16, THREADS = WARPS * 32, MAX_CHUNKS = 8;

struct RowsArgs {
  const __half *q, *kc, *vc; size_t q_ps, kv_ps;         // lo planes (NP = 2)
  RowSet rs;
  bf16* out; size_t out_ps;
  int H, max_seq, early;
};

__device__ __forceinline__ float ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
// eight float16 of each plane as floats
template <int NP> __device__ __forceinline__ void unpack8(const uint4 (&p)[NP], float (&v)[8]) {
  const uint32_t h[4] = {p[0].x, p[0].y, p[0].z, p[0].w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h[i])); v[2 * i] = f.x; v[2 * i + 1] = f.y; }
  if constexpr (NP == 2) {
    const uint32_t l[4] = {p[1].x, p[1].y, p[1].z, p[1].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&l[i])); v[2 * i] += f.x; v[2 * i + 1] += f.y; }
  }
}

template <int HD, int NP, int R>
__global__ void __launch_bounds__(THREADS, 1) tree_attn_rows_kernel(const RowsArgs a) {
  constexpr int LPK = HD / 8, KPW = 32 / LPK, GROUPS = WARPS * KPW, BATCH = 4;      // lanes a key; keys a warp takes at once; lane groups
  __shared__ float s_m[R][WARPS], s_l[R][WARPS];
  __shared__ __align__(16) float s_o[R][WARPS][HD];
  __shared__ float s_part[MAX_CHUNKS][R][HD + 2];         // the first CTA's: every chunk's rows, maximum and sum
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  pdl_trigger();
  const RowSet& rs = a.rs;
  const int h = blockIdx.x, b = blockIdx.y, c = blockIdx.z, nch = gridDim.z, H = a.H;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, sub = lane / LPK, dim = lane % LPK * 8;
  if (!a.early) pdl_wait();
  const int nr = min(rs.n_rows ? rs.n_rows[b] : rs.tc, rs.tc), p0 = rs.pos0[b], total = p0 + nr;
  const bool work = nr > 0 && p0 >= 0 && p0 <= a.max_seq - nr;
  const int k0 = work ? (int)((long long)total * c / nch) : 0, k1 = work ? (int)((long long)total * (c + 1) / nch) : 0;
  const size_t base = ((size_t)b * H + h) * a.max_seq * HD + dim;
  uint4 kv[BATCH][NP], vv[BATCH][NP];
  // keys at, at + GROUPS, ... of [from, to)
  auto fetch = [&](int at, int from, int to) {
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int slot = at + u * GROUPS;
      if (slot < from || slot >= to) continue;
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        kv[u][p] = __ldcs(reinterpret_cast<const uint4*>(a.kc + base + p * a.kv_ps + (size_t)slot * HD));
        vv[u][p] = __ldcs(reinterpret_cast<const uint4*>(a.vc + base + p * a.kv_ps + (size_t)slot * HD));
      }
    }
  };
  const int first = k0 + warp * KPW + sub;
#pragma unroll
  for (int u = 0; u < BATCH; ++u)
#pragma unroll
    for (int p = 0; p < NP; ++p) kv[u][p] = vv[u][p] = make_uint4(0u, 0u, 0u, 0u);
  if (a.early) { fetch(first, 0, min(k1, p0)); pdl_wait(); fetch(first, p0, k1); }      // committed keys are older than the preceding kernel
  else fetch(first, 0, k1);
  const float sc = rsqrtf((float)HD) * 1.4426950408889634f;   // 1/sqrt(hd) * log2(e)
  float q[R][8], o[R][8], m[R], l[R];
  uint64_t mask[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    uint4 p[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) p[i] = r < nr ? *reinterpret_cast<const uint4*>(a.q + i * a.q_ps + (size_t)(b * rs.tc + r) * H * HD + h * HD + dim) : make_uint4(0u, 0u, 0u, 0u);
    unpack8<NP>(p, q[r]);
    mask[r] = r < nr ? rs.mask ? rs.mask[r] : (2ull << r) - 1ull : 0ull;       // (no mask: a causal chunk)
    m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
    for (int d = 0; d < 8; ++d) { q[r][d] *= sc; o[r][d] = 0.f; }
  }
  for (int s0 = first; s0 - sub < k1; s0 += GROUPS * BATCH) {
    float s[R][BATCH];
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      float k[8];
      unpack8<NP>(kv[u], k);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float x = 0.f, y = 0.f;
#pragma unroll
        for (int d = 0; d < 8; d += 2) { x = fmaf(q[r][d], k[d], x); y = fmaf(q[r][d + 1], k[d + 1], y); }
        s[r][u] = x + y;
      }
    }
#pragma unroll
    for (int bit = LPK / 2; bit > 0; bit >>= 1)
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int u = 0; u < BATCH; ++u) s[r][u] += __shfl_xor_sync(0xffffffffu, s[r][u], bit);
    float w[R][BATCH];
    bool seen[R][BATCH];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float mn = m[r];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int slot = s0 + u * GROUPS;
        seen[r][u] = r < nr && slot < k1 && (slot < p0 || ((mask[r] >> (slot - p0)) & 1ull));
        if (!seen[r][u]) s[r][u] = -INFINITY;
        mn = fmaxf(mn, s[r][u]);
      }
      const float f = mn == -INFINITY ? 1.f : ex2(m[r] - mn), ref = mn == -INFINITY ? 0.f : mn;
      m[r] = mn;
      l[r] *= f;
#pragma unroll
      for (int d = 0; d < 8; ++d) o[r][d] *= f;
#pragma unroll
      for (int u = 0; u < BATCH; ++u) { w[r][u] = ex2(s[r][u] - ref); l[r] += w[r][u]; }
    }
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      if (s0 + u * GROUPS >= k1) continue;
      float v[8];
      unpack8<NP>(vv[u], v);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (seen[r][u]) {                                  // (a key that a row does not see adds nothing, whatever it holds)
#pragma unroll
          for (int d = 0; d < 8; ++d) o[r][d] = fmaf(w[r][u], v[d], o[r][d]);
        }
    }
    fetch(s0 + GROUPS * BATCH, 0, k1);
  }
  // lane groups of a warp, then warps
#pragma unroll
  for (int r = 0; r < R; ++r) {
#pragma unroll
    for (int bit = LPK; bit < 32; bit <<= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m[r], bit), M = fmaxf(m[r], m2), f = m[r] == -INFINITY ? 0.f : ex2(m[r] - M);
      l[r] *= f;
      l[r] += __shfl_xor_sync(0xffffffffu, l[r], bit);
#pragma unroll
      for (int d = 0; d < 8; ++d) { o[r][d] *= f; o[r][d] += __shfl_xor_sync(0xffffffffu, o[r][d], bit); }
      m[r] = M;
    }
    if (lane == 0) { s_m[r][warp] = m[r]; s_l[r][warp] = l[r]; }
    if (sub == 0) {
      *reinterpret_cast<float4*>(&s_o[r][warp][dim]) = make_float4(o[r][0], o[r][1], o[r][2], o[r][3]);
      *reinterpret_cast<float4*>(&s_o[r][warp][dim + 4]) = make_float4(o[r][4], o[r][5], o[r][6], o[r][7]);
    }
  }
  __syncthreads();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // the first CTA has started: its shared memory may be stored to
  const int r = tid / HD, k = tid % HD;                    // (512 threads: enough for two rows)
  if (r < R) {
    float M = -INFINITY, L = 0.f, acc = 0.f;
#pragma unroll
    for (int i = 0; i < WARPS; ++i) M = fmaxf(M, s_m[r][i]);
#pragma unroll
    for (int i = 0; i < WARPS; ++i) {
      const float f = s_m[r][i] == -INFINITY ? 0.f : ex2(s_m[r][i] - M);
      L += s_l[r][i] * f; acc += s_o[r][i][k] * f;
    }
    uint32_t to;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"((uint32_t)__cvta_generic_to_shared(&s_part[c][r][0])), "r"(0u));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to + 4u * k), "f"(acc) : "memory");
    if (k < 2) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to + 4u * (HD + k)), "f"(k ? L : M) : "memory");
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (c != 0 || r >= R || r >= rs.tc) return;
  float M = -INFINITY, L = 0.f, acc = 0.f;
  for (int i = 0; i < nch; ++i) M = fmaxf(M, s_part[i][r][HD]);
  for (int i = 0; i < nch; ++i) {
    const float mi = s_part[i][r][HD], f = mi == -INFINITY ? 0.f : ex2(mi - M);
    L += s_part[i][r][HD + 1] * f; acc += s_part[i][r][k] * f;
  }
  const float y = L == 0.f ? 0.f : acc / L;                // rows without keys get zeros; a sum that is no number stays none
  bf16* dst = a.out + (size_t)(b * rs.tc + r) * H * HD + h * HD + k;
  const bf16 hi = __float2bfloat16_rn(y);
  *dst = hi;
  if (a.out_ps) dst[a.out_ps] = __float2bfloat16_rn(y - __bfloat162float(hi));
}

}  // namespace

hydra_status tree_attention_rows(const __half* q, int q_rows, const __half* kc, const __half* vc, int cache_batch, int planes, RowSet rs, bf16* out, size_t out_ps, int H, int hd,
                                 int max_seq, int len_upper, bool stable_lengths, cudaStream_t st) {
  if (rs.blocks || rs.tc < 1 || rs.tc > 2 || (hd != 64 && hd != 128) || (planes != 1 && planes != 2)) return HYDRA_ERR_UNSUPPORTED;
  const RowsArgs a{q, kc, vc, (size_t)q_rows * H * hd, (size_t)cache_batch * H * max_seq * hd, rs, out, out_ps, H, max_seq, stable_lengths ? 1 : 0};
  // A chunk per 64 keys while the pairs leave SMs idle.  With more pairs, two where the last wave would fill at most half of the SMs with long CTAs, which
  // alone do not keep memory busy.  One chunk / two, us, two planes: 160 pairs of 500 keys 24.5 / 23.7, 1000 41.6 / 37.8, 4000 141 / 120; 208 of 1000 43.6 / 41.4, 8000 282 / 250; 352 of
  // 1000 68.1 / 69.4, 2000 123 / 118; 512 of 1000 91 / 94, 4000 321 / 311; but 256 (a last wave of 108) of 1000 47 / 53, 8000 307 / 322.
  const long long pairs = (long long)H * rs.batch, sms = sm_count(), last = pairs % sms;
  int n = (int)std::max(1ll, std::min({(long long)MAX_CHUNKS, sms / pairs, (len_upper + 63ll) / 64}));
  if (pairs > sms && last && 2 * last <= sms && len_upper >= 768 * (pairs / sms)) n = 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(H, rs.batch, n); cfg.blockDim = dim3(THREADS); cfg.dynamicSmemBytes = 0; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = (unsigned)n;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  auto rows = [&](auto hdc, auto np) -> cudaError_t {
    constexpr int HD = decltype(hdc)::value, NP = decltype(np)::value;
    return cudaLaunchKernelEx(&cfg, rs.tc == 1 ? tree_attn_rows_kernel<HD, NP, 1> : tree_attn_rows_kernel<HD, NP, 2>, a);
  };
  using std::integral_constant;
  if (hd == 128) HYDRA_CUDA(planes == 2 ? rows(integral_constant<int, 128>{}, integral_constant<int, 2>{}) : rows(integral_constant<int, 128>{}, integral_constant<int, 1>{}));
  else HYDRA_CUDA(planes == 2 ? rows(integral_constant<int, 64>{}, integral_constant<int, 2>{}) : rows(integral_constant<int, 64>{}, integral_constant<int, 1>{}));
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

}  // namespace hydra
