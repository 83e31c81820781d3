// The float path's matrix products, each with what follows it element by element, and with the RMSNorm ahead of it.
//
// The models of this path are small: a decode step is a chain of kernels of one to three microseconds each, most of it the way from one kernel's
// stores to the next one's loads, so what counts is how many there are.  Sums are whole here (no partial-sum slots), so the residual, SiLU and the
// rotary embedding with the cache rows happen where they are formed; and a norm needs the rows that are read for the product anyway: their squares
// are summed along, the gain goes to an operand and the row's factor to the sums.  A decoder layer is five launches (QKV with norm, rotation and cache rows; attention;
// O with the residual; gate and up with norm and SiLU; down with the residual; a sixth where the attention adds its chunks up) where it was nine, a draft head's layer one where it was two or
// three (gather, product, SiLU and residual).  Tiny float model (2 layers, d 256), a request of 32 tokens and 8 steps: 810 -> 577 us.
//
// Two forms.  Few rows or columns: a warp per output column (row_sums), so that a few hundred columns fill the SMs and the chain in a
// warp is short.  Many: 32 x 32 tiles out of shared memory, since a warp per column reads every row again for every column: 512 rows, d 256, f 688: QKV 21 -> 14 us, gate
// and up 38 -> 19, down 35 -> 16.  Requests of the tiny model's kind, before this file -> with it: 8 sequences, 64-row tree 5.09 -> 3.43 ms, a prompt of 1500
// tokens 3.90 -> 2.89, root-only decoding 0.52 -> 0.39; d 1024, 4 layers: 4.45 -> 3.43, 8 sequences 73.7 -> 33.1.
#include "launch.h"
#include <type_traits>

namespace hydra {
namespace {

constexpr int WARPS = 8, THREADS = WARPS * 32;

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float dot4(float4 a, float4 b, float s) { return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s)))); }
__device__ __forceinline__ float4 mul4(float4 a, float4 b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }

// Row n[b] - 1 of sequence b's tc rows (n null: its only one).
__device__ __forceinline__ const float* last_row(const LastRows& h, int b, int d) { return h.rows + ((size_t)b * h.tc + (h.n ? max(h.n[b] - 1, 0) : 0)) * d; }

// ---- where the rows of x come from.  prepare() waits for the preceding kernel and readies rows m0 .. m0 + R - 1; at(r, k): four elements of row m0 + r.
// tab: smem(R) bytes of shared memory.
struct Rows {
  const float* x; int m, k;
  size_t smem(int) const { return 0; }
  template <int R> __device__ __forceinline__ void prepare(int, void*) const { pdl_wait(); }
  __device__ __forceinline__ const float* at(int m0, int r, int kk, const void*) const { return x + (size_t)min(m0 + r, m - 1) * k + kk; }
};
// [h' ; E of the lv.d path tokens] of row (sequence, parent), read where they are; with write_root also tree_tok[b][0] = root_tok[b]
struct HeadRows {
  LastRows h; const float* embed;
  const int *root_tok, *path_tab; int* tree_tok;
  LevelDesc lv;
  int write_root, T, kp1, vocab, m, d;
  int* status;
  size_t smem(int r) const { return (size_t)r * (lv.d + 1) * sizeof(const float*); }
  template <int R> __device__ __forceinline__ void prepare(int m0, void* tab) const {      // tab [R][lv.d + 1]: where the blocks of the rows are
    const int blocks = lv.d + 1;
    for (int e = threadIdx.x; e < R * blocks; e += THREADS) {
      const int r = min(m0 + e / blocks, m - 1), blk = e % blocks, b = r / lv.n_parents, j = r - b * lv.n_parents;
      const int node = blk ? path_tab[lv.parents[j] * kp1 + blk - 1] : 0;       // (tables, older than any call)
      pdl_wait();
      const float* src = last_row(h, b, d);
      if (blk) {
        int t = node == 0 ? root_tok[b] : tree_tok[b * T + node];
        if (t < 0 || t >= vocab) { atomicOr(status, ST_BOUNDS); t = 0; }
        src = embed + (size_t)t * d;
      } else if (write_root && j == 0 && blockIdx.x == 0) {
        tree_tok[b * T] = root_tok[b];
      }
      static_cast<const float**>(tab)[e] = src;
    }
    pdl_wait();
    __syncthreads();
    if (h.copy && blockIdx.x == 0)                         // (one parent a sequence then: row r is sequence r)
      for (int e = threadIdx.x * 4; e < R * d; e += THREADS * 4) {
        const int r = e / d;
        if (m0 + r < m) *reinterpret_cast<float4*>(h.copy + (size_t)m0 * d + e) = ld4(static_cast<const float* const*>(tab)[r * blocks] + (e - r * d));
      }
  }
  __device__ __forceinline__ const float* at(int, int r, int kk, const void* tab) const {      // (d % 4 == 0: four elements lie in one block)
    const int blk = kk / d;
    return static_cast<const float* const*>(tab)[r * (lv.d + 1) + blk] + (kk - blk * d);
  }
};

// ---- what becomes of the sums.  An output unit is one column (NC = 1) or two that belong together (NC = 2): w_row(unit, c) are its weight rows.
// load(): what store() needs besides the sums, read behind the wait and ahead of the product.  NORM: the sums are those of rmsnorm(x) * gain.
struct Plain {
  static constexpr int NC = 1; static constexpr bool NORM = false;
  float* out; int n;
  struct Pre {};
  int units() const { return n; }
  __device__ __forceinline__ int w_row(int u, int) const { return u; }
  __device__ __forceinline__ Pre load(int, int) const { return Pre{}; }
  __device__ __forceinline__ void store(int row, int u, const Pre&, const float (&s)[1]) const { out[(size_t)row * n + u] = s[0]; }
};
// the product of rmsnorm(x) * gain, and those rows themselves
struct NormedOut {
  static constexpr int NC = 1; static constexpr bool NORM = true;
  float *out, *hn; int n;
  struct Pre {};
  int units() const { return n; }
  __device__ __forceinline__ int w_row(int u, int) const { return u; }
  __device__ __forceinline__ Pre load(int, int) const { return Pre{}; }
  __device__ __forceinline__ void store(int row, int u, const Pre&, const float (&s)[1]) const { out[(size_t)row * n + u] = s[0]; }
};
struct Add {
  static constexpr int NC = 1; static constexpr bool NORM = false;
  const float* res; float* out; int n;                     // out may be res
  struct Pre { float base; };
  int units() const { return n; }
  __device__ __forceinline__ int w_row(int u, int) const { return u; }
  __device__ __forceinline__ Pre load(int row, int u) const { return Pre{res[(size_t)row * n + u]}; }
  __device__ __forceinline__ void store(int row, int u, const Pre& p, const float (&s)[1]) const { out[(size_t)row * n + u] = p.base + s[0]; }
};
struct Glu {
  static constexpr int NC = 2; static constexpr bool NORM = true;
  float* act; int f;
  struct Pre {};
  int units() const { return f; }
  __device__ __forceinline__ int w_row(int u, int c) const { return c * f + u; }
  __device__ __forceinline__ Pre load(int, int) const { return Pre{}; }
  __device__ __forceinline__ void store(int row, int u, const Pre&, const float (&s)[2]) const { act[(size_t)row * f + u] = silu_f(s[0]) * s[1]; }
};
// Columns j and j + hd/2 of a head of q, k or v: q and k rotated, k and v into the cache.  first = 1: the projection has no q columns.
struct Qkv {
  static constexpr int NC = 2; static constexpr bool NORM = true;
  RowSet rs; const float2* table; float *q, *kc, *vc;
  int H, hd, max_seq, first; int* status;
  struct Pre { float2 cs; int b, slot; };                  // slot -2: a row that the call does not have
  int units() const { return (3 - first) * H * (hd >> 1); }
  __device__ __forceinline__ int w_row(int u, int c) const { const int half = hd >> 1, head = u / half; return head * hd + (u - head * half) + c * half; }
  __device__ __forceinline__ Pre load(int row, int u) const {
    const int half = hd >> 1, b = row / rs.tc, i = row - b * rs.tc;
    Pre p{make_float2(1.f, 0.f), b, -2};
    if (i < (rs.n_rows ? rs.n_rows[b] : rs.tc)) {
      const int slot = rs.pos0[b] + i;
      p.slot = slot >= 0 && slot < max_seq ? slot : -1;
    }
    if (u < (2 - first) * H * half) p.cs = table[(size_t)row * half + u % half];
    return p;
  }
  __device__ __forceinline__ void store(int row, int u, const Pre& p, const float (&s)[2]) const {
    if (p.slot < 0) { if (p.slot == -1 && u == 0) atomicOr(status, ST_BOUNDS); return; }
    const int half = hd >> 1, head = u / half, j = u - head * half, which = head / H + first, h = head % H;
    float* dst = which == 0 ? q + (size_t)row * (H * hd) + h * hd : (which == 1 ? kc : vc) + (((size_t)p.b * H + h) * max_seq + p.slot) * hd;
    dst[j] = which < 2 ? s[0] * p.cs.x - s[1] * p.cs.y : s[0];
    dst[j + half] = which < 2 ? s[1] * p.cs.x + s[0] * p.cs.y : s[1];
  }
};
// y = res + SiLU(s + bias), res: the last row of sequence row / rows_per_res
struct HeadAct {
  static constexpr int NC = 1; static constexpr bool NORM = false;
  LastRows res; const float* bias; float* y; int d, rows_per_res;
  struct Pre { float base, add; };
  int units() const { return d; }
  __device__ __forceinline__ int w_row(int u, int) const { return u; }
  __device__ __forceinline__ Pre load(int row, int u) const { return Pre{last_row(res, row / rows_per_res, d)[u], bias ? bias[u] : 0.f}; }
  __device__ __forceinline__ void store(int row, int u, const Pre& p, const float (&s)[1]) const { y[(size_t)row * d + u] = p.base + silu_f(s[0] + p.add); }
};

// The normed rows of a block's row group, dealt out over the blocks that share it: inv[r] of rows m0 .. m0 + R - 1 in shared memory.
template <int R, typename Src, typename Op>
__device__ __forceinline__ void normed_rows(const Src& src, const Op& op, const float* gain, const float* inv, int m0, int m, int k) {
  if constexpr (std::is_same<Op, NormedOut>::value) {
    __syncthreads();
    for (int e = (blockIdx.x * THREADS + threadIdx.x) * 4; e < R * k; e += gridDim.x * THREADS * 4) {
      const int r = e / k, c = e - r * k;
      if (m0 + r >= m) break;
      const float4 x = ld4(src.at(m0, r, c, nullptr)), g = ld4(gain + c);
      *reinterpret_cast<float4*>(op.hn + (size_t)(m0 + r) * k + c) = make_float4(x.x * (inv[r] * g.x), x.y * (inv[r] * g.y), x.z * (inv[r] * g.z), x.w * (inv[r] * g.w));
    }
  }
}

// ---- few rows: one warp per output column and MR rows
// What a warp makes of its share of the contraction: s[c] = sum_k w_c[k] x[r][k] for C weight rows, with NORM also s[C] = sum_k x[r][k]^2, of row
// r = warp_sum_owner(lane) in lanes 0..MR-1.  KS warps share an output: every KS-th 512-byte piece of its weight rows each, added in shared memory;
// the first of them ends up with the sums.  With NORM the weights come times the norm's gain.  w_const: no kernel in flight writes the weights, and
// their first pieces are loaded ahead of the wait.
template <int MR, int KS, int C, bool NORM, typename Src, typename AtWait>
__device__ __forceinline__ void row_sums(const Src& src, int m0, const float* const (&w)[C], const float* gain, int k, int w_const, AtWait at_wait, float (&s)[C + (NORM ? 1 : 0)]) {
  constexpr int NS = C + (NORM ? 1 : 0), PRE = 2;
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ float s_part[WARPS][NS][MR];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k0 = (warp % KS) * 128 + lane * 4;
  auto weights = [&](int kk, float4 (&v)[C]) {
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = ld4(w[c] + kk);
    if constexpr (NORM) {
      const float4 g = ld4(gain + kk);
#pragma unroll
      for (int c = 0; c < C; ++c) v[c] = mul4(v[c], g);
    }
  };
  float4 wp[PRE][C];
  if (!w_const) pdl_wait();
#pragma unroll
  for (int i = 0; i < PRE; ++i)
    if (k0 + i * KS * 128 < k) weights(k0 + i * KS * 128, wp[i]);
  src.template prepare<MR>(m0, s_dyn);
  at_wait();
  float acc[NS][MR];
#pragma unroll
  for (int c = 0; c < NS; ++c)
#pragma unroll
    for (int r = 0; r < MR; ++r) acc[c][r] = 0.f;
  auto step = [&](int kk, const float4 (&wk)[C]) {
#pragma unroll
    for (int r = 0; r < MR; ++r) {
      const float4 x = ld4(src.at(m0, r, kk, s_dyn));
#pragma unroll
      for (int c = 0; c < C; ++c) acc[c][r] = dot4(wk[c], x, acc[c][r]);
      if constexpr (NORM) acc[C][r] = dot4(x, x, acc[C][r]);
    }
  };
#pragma unroll
  for (int i = 0; i < PRE; ++i)
    if (k0 + i * KS * 128 < k) step(k0 + i * KS * 128, wp[i]);
  for (int kk = k0 + PRE * KS * 128; kk < k; kk += KS * 128) {
    float4 wk[C];
    weights(kk, wk);
    step(kk, wk);
  }
#pragma unroll
  for (int c = 0; c < NS; ++c) s[c] = warp_sum_multi<MR>(acc[c], lane);
  if constexpr (KS > 1) {
    const int r = warp_sum_owner<MR>(lane);
    if (lane < MR) {
#pragma unroll
      for (int c = 0; c < NS; ++c) s_part[warp][c][r] = s[c];
    }
    __syncthreads();
    if (lane < MR && warp % KS == 0) {
#pragma unroll
      for (int q = 1; q < KS; ++q)
#pragma unroll
        for (int c = 0; c < NS; ++c) s[c] += s_part[warp + q][c][r];
    }
  }
}

// SPLIT: the two columns of a unit are two neighbours' (of KS warps each) instead of one warp's.
template <int MR, int KS, bool SPLIT, typename Src, typename Op>
__global__ void __launch_bounds__(THREADS, 2) f32_rows_kernel(const Src src, const float* w, const float* gain, const Op op, int n_units, int m, int k, float eps, int w_const) {
  pdl_trigger();
  constexpr int NC = Op::NC, C = SPLIT ? 1 : NC, PER = WARPS / KS / (SPLIT ? NC : 1);      // units a block
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, mate = SPLIT ? warp / KS % NC : 0;
  const int unit = blockIdx.x * PER + warp / KS / (SPLIT ? NC : 1), m0 = blockIdx.y * MR, row = m0 + warp_sum_owner<MR>(lane), u = min(unit, n_units - 1);
  const bool mine = lane < MR && row < m && unit < n_units && warp % KS == 0 && mate == 0;
  const float* wr[C];
#pragma unroll
  for (int c = 0; c < C; ++c) wr[c] = w + (size_t)op.w_row(u, SPLIT ? mate : c) * k;
  float t[C + (Op::NORM ? 1 : 0)];
  typename Op::Pre pre;
  const float* const(&wc)[C] = wr;
  row_sums<MR, KS, C, Op::NORM>(src, m0, wc, gain, k, w_const, [&]() { if (mine) pre = op.load(row, unit); }, t);
  float s[NC];
#pragma unroll
  for (int c = 0; c < C; ++c) s[c] = t[c];
  if constexpr (SPLIT && NC == 2) {
    __shared__ float s_mate[WARPS][MR];
    if (mate && warp % KS == 0 && lane < MR) s_mate[warp][lane] = t[0];
    __syncthreads();
    if (mine) s[1] = s_mate[warp + KS][lane];
  }
  if constexpr (Op::NORM) {
    __shared__ float s_inv[MR];
    const float inv = rsqrtf(t[C] / (float)k + eps);
#pragma unroll
    for (int c = 0; c < NC; ++c) s[c] *= inv;
    if (std::is_same<Op, NormedOut>::value && warp == 0 && lane < MR) s_inv[warp_sum_owner<MR>(lane)] = inv;
    if (mine) op.store(row, unit, pre, s);
    normed_rows<MR>(src, op, gain, s_inv, m0, m, k);
  } else {
    if (mine) op.store(row, unit, pre, s);
  }
}

// ---- many rows: tiles of 32 rows x 32 weight rows (32 units, or 16 of two columns).  64 k a stage come by asynchronous copies, four stages, so that d = 256 is
// in flight as a whole: with few tiles an SM the time is that of the loads (one stage ahead through registers: gate and up of 512 rows 26 us, so 19).  A warp takes 8 of a
// stage's 64 k, 8 x 4 sums a thread: twelve 16-byte reads of shared memory for 128 multiply-adds (4 x 4: sixteen, and shared memory is what bounds the loop).  A row
// is 68 floats of shared memory, so the eight rows that a quarter warp reads lie in different banks.  The warps' sums meet in shared memory at the end.
constexpr int TM = 32, TN = 32, TK = 64, STAGES = 4, LDS_ROW = TK + 4, STAGE_FLOATS = (TM + TN) * LDS_ROW + TK;      // (the norm's gain at the end)
constexpr size_t TILE_SMEM = (size_t)STAGES * STAGE_FLOATS * sizeof(float);
__device__ __forceinline__ void copy16(float* dst, const float* src, bool there) {      // zeros where there is nothing
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(there ? 16 : 0) : "memory");
}
template <typename Src, typename Op>
__global__ void __launch_bounds__(THREADS, 2) f32_tile_kernel(const Src src, const float* w, const float* gain, const Op op, int n_units, int m, int k, float eps, int w_const) {
  pdl_trigger();
  constexpr int NC = Op::NC, UNITS = TN / NC, OUT = TM * UNITS / THREADS;
  extern __shared__ __align__(16) unsigned char s_dyn[];
  float* stage0 = reinterpret_cast<float*>(s_dyn);
  void* tab = s_dyn + TILE_SMEM;
  __shared__ float s_ss[WARPS][TM], s_inv[TM];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, m0 = blockIdx.y * TM, u0 = blockIdx.x * UNITS, n_stages = (k + TK - 1) / TK;
  // a thread copies 16 bytes of rows cr and cr + 16 of x and of w
  const int cr = tid >> 4, ck = (tid & 15) * 4;
  const float* wr[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) { const int n = cr + 16 * i; wr[i] = w + (size_t)op.w_row(min(u0 + n % UNITS, n_units - 1), n / UNITS) * k + ck; }
  auto copy_w = [&](int s) {
    float* dst = stage0 + (s % STAGES) * STAGE_FLOATS + (TM + cr) * LDS_ROW + ck;
    const bool there = s * TK + ck < k;
#pragma unroll
    for (int i = 0; i < 2; ++i) copy16(dst + 16 * i * LDS_ROW, there ? wr[i] + s * TK : w, there);
    if (Op::NORM && cr == 0) copy16(stage0 + (s % STAGES) * STAGE_FLOATS + (TM + TN) * LDS_ROW + ck, there ? gain + s * TK + ck : w, there);
  };
  auto copy_x = [&](int s) {
    float* dst = stage0 + (s % STAGES) * STAGE_FLOATS + cr * LDS_ROW + ck;
    const int kk = s * TK + ck;
#pragma unroll
    for (int i = 0; i < 2; ++i) copy16(dst + 16 * i * LDS_ROW, kk < k ? src.at(m0, cr + 16 * i, kk, tab) : w, kk < k);
  };
  auto commit = []() { asm volatile("cp.async.commit_group;" ::: "memory"); };
  if (!w_const) pdl_wait();
#pragma unroll
  for (int s = 0; s < STAGES; ++s) if (s < n_stages) copy_w(s);
  src.template prepare<TM>(m0, tab);
#pragma unroll
  for (int s = 0; s < STAGES; ++s) { if (s < n_stages) copy_x(s); commit(); }
  typename Op::Pre pre[OUT];
#pragma unroll
  for (int o = 0; o < OUT; ++o) {
    const int row = m0 + tid / UNITS + o * (THREADS / UNITS), unit = u0 + tid % UNITS;
    if (row < m && unit < n_units) pre[o] = op.load(row, unit);
  }
  const int ty = lane >> 3, tx = lane & 7;                 // rows ty + 4 i, columns tx + 8 j; the warp's 8 k of the stage's 64
  float acc[8][4] = {}, ss = 0.f;
  for (int s = 0; s < n_stages; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 1) : "memory");
    __syncthreads();
    const float* at = stage0 + (s % STAGES) * STAGE_FLOATS + warp * 8;
    const float *sx = at + ty * LDS_ROW, *sw = at + (TM + tx) * LDS_ROW, *sg = at + (TM + TN) * LDS_ROW;
#pragma unroll
    for (int q = 0; q < 8; q += 4) {
      float4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = ld4(sw + 8 * j * LDS_ROW + q);
      if constexpr (Op::NORM) {
        const float4 g = ld4(sg + q), mine = ld4(at + lane * LDS_ROW + q);
        ss = dot4(mine, mine, ss);                         // row `lane`
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = mul4(v[j], g);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 x = ld4(sx + 4 * i * LDS_ROW + q);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = dot4(x, v[j], acc[i][j]);
      }
    }
    if (s + STAGES < n_stages) {
      __syncthreads();                                     // everyone is past the stage
      copy_w(s + STAGES);
      copy_x(s + STAGES);
    }
    commit();
  }
  __syncthreads();
  float* red = stage0;                                     // [8 warps][TM][TN + 1]
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) red[(warp * TM + ty + 4 * i) * (TN + 1) + tx + 8 * j] = acc[i][j];
  if constexpr (Op::NORM) s_ss[warp][lane] = ss;
  __syncthreads();
#pragma unroll
  for (int o = 0; o < OUT; ++o) {
    const int r = tid / UNITS + o * (THREADS / UNITS), c0 = tid % UNITS, row = m0 + r, unit = u0 + c0;
    if (std::is_same<Op, NormedOut>::value && c0 == 0) {
      float t = 0.f;
#pragma unroll
      for (int v = 0; v < WARPS; ++v) t += s_ss[v][r];
      s_inv[r] = rsqrtf(t / (float)k + eps);
    }
    if (row >= m || unit >= n_units) continue;
    float s[NC] = {}, t = 0.f;
#pragma unroll
    for (int v = 0; v < WARPS; ++v) {
#pragma unroll
      for (int c = 0; c < NC; ++c) s[c] += red[(v * TM + r) * (TN + 1) + c * UNITS + c0];
      if constexpr (Op::NORM) t += s_ss[v][r];
    }
    if constexpr (Op::NORM) {
      const float inv = rsqrtf(t / (float)k + eps);
#pragma unroll
      for (int c = 0; c < NC; ++c) s[c] *= inv;
    }
    op.store(row, unit, pre[o], s);
  }
  normed_rows<TM>(src, op, gain, s_inv, m0, m, k);
}
static_assert(WARPS * TM * (TN + 1) <= STAGES * STAGE_FLOATS, "the warps' sums take the place of the stages");

constexpr int TILE_ROWS = 16, PAIR_K = 256;

template <typename Src, typename Op>
hydra_status product(const Src& src, const float* w, const float* gain, const Op& op, int m, int k, float eps, bool w_const, cudaStream_t st) {
  if (m <= 0 || k <= 0 || (k & 3) || op.units() <= 0) return HYDRA_ERR_UNSUPPORTED;
  if (((uintptr_t)w | (uintptr_t)gain) & 15) return HYDRA_ERR_INVALID;      // read four elements at a time, like the rows
  const int units = op.units();
  constexpr int U = TN / Op::NC;
  const long tiles = (long)((units + U - 1) / U) * ((m + TM - 1) / TM);
  // Tiles where they come to four fifths of the SMs (whole requests, us, with the line at 40 / 70 / 118 tiles: d 256, 64 rows 1009 / 990 / 956, 3 x 64 rows
  // 1801 / 1672 / 1674, 8 x 64 rows 3460 / 3442 / 3426, d 512, 3 x 64 rows 2984 / 2925 / 2863, d 1024, 16 rows behind a prompt 3396 / 3422 / 3428).
  if (m > TILE_ROWS && 5 * tiles >= 4 * sm_count()) {
    static PerDeviceFlag attr_done;
    const size_t most = TILE_SMEM + TM * 65 * sizeof(const float*);      // (a tree is at most 64 levels deep)
    if (!attr_done.get()) {
      HYDRA_CUDA(cudaFuncSetAttribute(f32_tile_kernel<Src, Op>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
      attr_done.set();
    }
    if (TILE_SMEM + src.smem(TM) > most) return HYDRA_ERR_UNSUPPORTED;
    launch_pdl(f32_tile_kernel<Src, Op>, dim3((units + U - 1) / U, (m + TM - 1) / TM), dim3(THREADS), TILE_SMEM + src.smem(TM), st, src, w, gain, op, units, m, k, eps, (int)w_const);
    HYDRA_LAUNCH_CHECK();
    return HYDRA_OK;
  }
  auto rows = [&](auto mr, auto split) {
    constexpr int MR = decltype(mr)::value;
    constexpr bool SPLIT = decltype(split)::value;
    const long cols = (long)units * (SPLIT ? Op::NC : 1), groups = (m + MR - 1) / MR, pieces = (k + 127) / 128, want = 2 * sm_count();
    auto launch = [&](auto ks) {
      constexpr int KS = decltype(ks)::value, PER = WARPS / KS / (SPLIT ? Op::NC : 1);
      launch_pdl(f32_rows_kernel<MR, KS, SPLIT, Src, Op>, dim3((units + PER - 1) / PER, (unsigned)groups), dim3(THREADS), src.smem(MR), st, src, w, gain, op, units, m, k, eps, (int)w_const);
    };
    // warps per column: until there are two to four blocks per SM or a lane has one piece
    if (pieces >= 4 && cols * groups / 4 <= want) launch(std::integral_constant<int, 4>{});
    else if (pieces >= 2 && cols * groups / 8 <= want) launch(std::integral_constant<int, 2>{});
    else launch(std::integral_constant<int, 1>{});
  };
  auto split = [&](auto mr) {
    // A warp that takes both columns of a unit reads the rows once for the two, but has half the loads in flight: the better form where its weights are
    // a piece or two (16 rows, d 256: a request of the tiny model 661 us, 691 with two warps; d 1024: 4.81 and 3.85 ms)
    if constexpr (Op::NC == 2) { if (k > PAIR_K) { rows(mr, std::true_type{}); return; } }
    rows(mr, std::false_type{});
  };
  if (m == 1) split(std::integral_constant<int, 1>{});
  else if (m <= 4) split(std::integral_constant<int, 4>{});
  else if (m <= 8) split(std::integral_constant<int, 8>{});
  else split(std::integral_constant<int, 16>{});
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}
inline bool off16(const void* p) { return ((uintptr_t)p & 15) != 0; }

}  // namespace

hydra_status f32_gemm(const float* x, const float* w, float* out, int m, int n, int k, bool w_const, cudaStream_t st) {
  if (off16(x)) return HYDRA_ERR_INVALID;
  return product(Rows{x, m, k}, w, nullptr, Plain{out, n}, m, k, 0.f, w_const, st);
}
hydra_status f32_normed_gemm(const float* x, const float* gain, const float* w, float* out, float* hn, int m, int n, int k, float eps, cudaStream_t st) {
  if (off16(x) || off16(hn)) return HYDRA_ERR_INVALID;
  return product(Rows{x, m, k}, w, gain, NormedOut{out, hn, n}, m, k, eps, true, st);
}
hydra_status f32_add(const float* x, const float* w, const float* res, float* out, int m, int n, int k, cudaStream_t st) {
  if (off16(x)) return HYDRA_ERR_INVALID;
  return product(Rows{x, m, k}, w, nullptr, Add{res, out, n}, m, k, 0.f, true, st);
}
hydra_status f32_glu(const float* x, const float* gain, const float* w, float* act, int m, int f, int d, float eps, cudaStream_t st) {
  if (off16(x)) return HYDRA_ERR_INVALID;
  return product(Rows{x, m, d}, w, gain, Glu{act, f}, m, d, eps, true, st);
}
hydra_status f32_qkv(const float* x, const float* gain, const float* w, const float2* table, float* q, float* kc, float* vc, RowSet rs, int H, int hd, int max_seq,
                     bool kv_only, float eps, int* status, cudaStream_t st) {
  if ((hd & 7) || rs.row_at) return HYDRA_ERR_UNSUPPORTED;
  if (off16(x)) return HYDRA_ERR_INVALID;
  const int m = rs.rows(), d = H * hd;
  return product(Rows{x, m, d}, w, gain, Qkv{rs, table, q, kc, vc, H, hd, max_seq, kv_only ? 1 : 0, status}, m, d, eps, true, st);
}
hydra_status f32_head_first(const LastRows& h, const float* embed, const int* root_tok, int* tree_tok, const int* path_tab, LevelDesc lv, int write_root,
                            const float* w, const float* bias, float* y, int batch, int T, int kp1, int d, int vocab, int* status, cudaStream_t st) {
  if (d & 3) return HYDRA_ERR_UNSUPPORTED;
  if (off16(h.rows) || off16(embed)) return HYDRA_ERR_INVALID;
  if (h.copy && lv.n_parents != 1) return HYDRA_ERR_INVALID;
  const int m = batch * lv.n_parents;
  return product(HeadRows{h, embed, root_tok, path_tab, tree_tok, lv, write_root, T, kp1, vocab, m, d, status}, w, nullptr, HeadAct{h, bias, y, d, lv.n_parents}, m,
                 (lv.d + 1) * d, 0.f, true, st);
}
hydra_status f32_head_next(const float* y_in, const float* w, const float* bias, float* y, int m, int d, cudaStream_t st) {
  if (off16(y_in)) return HYDRA_ERR_INVALID;
  return product(Rows{y_in, m, d}, w, nullptr, HeadAct{LastRows{y_in, nullptr, 1, nullptr}, bias, y, d, 1}, m, d, 0.f, true, st);
}

}  // namespace hydra
