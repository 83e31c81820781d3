// Tree attention for the bfloat16 model path on the sm_100a tensor cores: TMA tile loads, tcgen05.mma with the
// score and output accumulators in tensor memory, softmax out of tensor memory.
//
// Operand format: q, the K cache (post-RoPE), the V cache and the softmax weights are float16 (the values are O(1),
// far inside the float16 range) in NP planes.  NP = 2: hi = f16(v), lo = f16(v - hi), about 22 significant bits;
// a product x y is taken as x_hi y_hi + x_hi y_lo + x_lo y_hi.  For the scores, stacking the planes of K along the N
// dimension gives the first two terms in ONE instruction sequence (accumulator columns [0, n) and [n, 2n), added
// when the accumulator is read); the third is a second sequence into columns [0, n).  For P V, all three go into the
// same head_dim columns.  NP = 1: hi only, 11 bits
// (half the cache bytes; hidden states then drift to a few 1e-3 of a float reference over 32 layers).
// Scores, running maxima, sums and the output accumulate in float.  The result leaves as two bfloat16 planes
// (hi = bf16(v), lo = bf16(v - hi)), the operand format of the GEMM that consumes it.
//
// One CTA per (head, sequence, KV chunk).  A sequence's KV rows are cut into 64-row tiles and the tiles are dealt
// to the launch's chunks in equal contiguous runs, computed on the device from the real length (a captured graph
// keeps balanced chunks as the sequence grows).  Roles (256 threads for 64 query rows, 320 for 128):
//   one producer lane  TMA: Q once, then K tiles and V tiles through rings of their own (a K stage is free
//                      as soon as the scores of its tile are done, a V stage after the tile's P V product), each stage
//                      with its own "full" barrier, so the scores of a tile start before its V has landed;
//   one MMA lane       S_i = Q K_i^T (M = 128 query lanes, N = 64 keys) into one of two score buffers in
//                      tensor memory; O += P_i V_i (N = head_dim, V read as an MN-major operand
//                      straight from its [key][dim] tile) into one accumulator that lives across the chunk; whichever of
//                      the next S and the next P V has its operands is issued;
//   softmax warps      thread = query row (a tensor-memory lane), all 64 keys of a tile.  Two groups of warps take the tiles in
//                      turn, even and odd, so that one group's exponentials run while the other waits for scores, loads
//                      them or stores its P.  A thread reads its scores from tensor memory, applies
//                      the mask (committed slots are visible to every row; tree slot j to row i iff bit j of the
//                      row's ancestor bitmask, or j <= i for a causal chunk), takes the row's running reference
//                      maximum (exp2 domain) over from the other group, hands it on, and writes P_i as float16 into tensor
//                      memory, the A operand of the P V product.  The reference maximum only moves when a tile's maximum exceeds it by
//                      more than 8 (a factor 256, harmless in float16 and float); only then is the row's output
//                      accumulator rescaled in tensor memory (load, scale, store), so the common tile needs no
//                      round trip through registers for O.  Each group keeps its own row sum.
// What bounds a tile of the loop (two planes, head_dim 128): 64 KB from memory (1.1 us with 120 CTAs at 7 TB/s), about 1800
// cycles of shared memory and 1540 of the tensor pipe (see S_COLS), 512 of exponentials per 32 rows; a softmax step is a chain of
// about 1600 cycles, of which two run at a time.  With one group of softmax warps (a tile of 64 rows shared by two warps), P in
// shared memory and the rows of one chunk merged like those of several, a stand-alone call of 64 rows took, against now (back to back
// over caches larger than the L2, graph replay): 8 sequences of 250 to 1100 tokens x 32 heads 56.1 -> 49.2 us, 4 of 1050 x 52 heads
// 61.4 -> 58.1, 1 of 2000 x 40 heads 23.4 -> 22.7, 1 of 600 x 32 heads 12.6 -> 11.9.
// Query rows beyond the row count of the call ride along as unused lanes of the M = 128 tile.
// One chunk: the softmax warps normalise their rows out of tensor memory and write them, through a warp's own piece of the
// idle ring for whole 128-byte stores; no cluster, no merge.
// Several chunks of a (head, sequence) pair (at most 8) form a thread-block cluster: every CTA leaves its partial rows
// (un-normalised output, reference maximum, sum) in its own shared memory, and each CTA merges a share of the rows
// out of its peers' shared memory, in chunk order (deterministic; no scratch traffic, no atomics).
// (Sending the rows to the CTA that merges them, instead of reading them from there, took longer: 1.5 us for 64 rows of a chunk.)
// Every barrier wait is bounded; when one runs out the CTA raises the time-out bit of the status word, skips its
// stores, still takes part in the cluster barriers, frees its tensor memory and returns.
#include "tc.cuh"
#include <cuda_fp16.h>
#include <math.h>
#include <algorithm>

namespace hydra {

namespace {

using namespace tc;

constexpr int TILE = 64;           // KV rows per tile
constexpr int MAX_CHUNKS = 8;      // chunks of a (head, sequence) pair = cluster size
constexpr float RESCALE_STEP = 8.f;

__device__ __forceinline__ int chunk_first_tile(int c, int nt, int nch) { return (int)(((unsigned)c * (unsigned)nt) / (unsigned)nch); }

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_smem(uint32_t saddr, uint32_t rank) {     // the same offset in CTA `rank`'s shared memory
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_peer4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ float4 ld_smem4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
// two floats in one register pair: one instruction for both
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
  f32x2 v;
  asm("mov.b64 %0, {%1,%2};" : "=l"(v) : "f"(x), "f"(y));
  return v;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0,%1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 v;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 v;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
  return v;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float v;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(v) : "f"(a), "f"(b), "f"(c));
  return v;
}

struct AttArgs {
  RowSet rs;
  int q_plane_rows, kv_plane_rows;     // rows between the hi and lo planes in the q and cache tensor maps
  bf16* out; size_t out_ps;
  int H, max_seq, nchunks;
  int* status;
  uint32_t wait_limit;
  int early;                           // the lengths (rs.pos0, rs.n_rows) and the committed cache rows were written by kernels that
                                       // completed before the preceding kernel started (see tree_attention_tc)
};

template <int HD, int QROWS, int NP> struct AttCfg {
  static constexpr int NHALF = HD / 64;                       // 64-column (128-byte) halves of a head row
  static constexpr int QP_BYTES = NHALF * QROWS * 128;        // one plane of Q: [half][query row][128 bytes]
  static constexpr int Q_BYTES = NP * QP_BYTES;
  static constexpr int KH_BYTES = NP * TILE * 128;            // one half of a K tile: [plane][key][128 bytes] (the planes stacked along N)
  static constexpr int K_BYTES = NHALF * KH_BYTES;
  static constexpr int V_BYTES = NP * NHALF * TILE * 128;     // a V tile: [plane][half][key][128 bytes] (N blocks of 64 output columns)
  // K and V tiles travel through rings of their own: a K stage is free again as soon as the scores of its tile are done,
  // long before the tile's P V product frees the V stage, so K runs further ahead inside the same shared memory.
  // Two planes at head_dim 128: 64 KB a tile, 32 KB (64 query rows) or 64 KB (128) of Q.
  static constexpr int NSK = K_BYTES >= 32768 ? 3 : 4;           // K ring stages
  static constexpr int NSV = V_BYTES >= 32768 ? (Q_BYTES > 32768 ? 2 : 3) : 4;      // V ring stages
  // MMA M is 128 whatever QROWS is: with 64 query rows the upper 64 accumulator lanes are unused (M = 64 instructions
  // measured slower per instruction), and the operand reads of a 64-row Q tile run 8 KB past the tile, into the next
  // piece of Q or the ring (never read back).
  static constexpr int MROWS = 128;
  static constexpr int KRING_BYTES = NSK * K_BYTES;
  static constexpr int RING_BYTES = KRING_BYTES + NSV * V_BYTES;
  static constexpr int MERGE_BYTES = QROWS * HD * 4 + QROWS * 16;    // a chunk's partial rows + (max, sum) of either group; aliases the ring
  // softmax warps: group g (even / odd tiles), quadrant q of tensor memory -> warp 4 g + q; 64 query rows only fill quadrants
  // 0 and 1, which leaves warps 2 and 3 for the producer and the MMA lane
  static constexpr int NQUAD = QROWS / 32;
  static constexpr int NTHREADS = QROWS == 64 ? 256 : 320;
  static constexpr int W_PRODUCER = QROWS == 64 ? 2 : 8, W_MMA = W_PRODUCER + 1;
  static constexpr int XM_BYTES = 2 * QROWS * 4;                     // [group][row] reference maximum
  static constexpr int BUF_BYTES = NHALF * NQUAD * 2 * 32 * 128;     // one-chunk result on its way out: 32 rows x 64 columns x 2 planes per warp; aliases the ring
  static constexpr int NBAR = 1 + 2 * NSK + 2 * NSV + 9 + 2 * NQUAD;
  static constexpr int SMEM_BYTES = 1024 + Q_BYTES + RING_BYTES + XM_BYTES + NBAR * 8 + 16;
  // tensor memory: two score buffers [Q_hi K_hi + Q_lo K_hi | Q_hi K_lo], the output accumulator, two P buffers (32 columns a
  // plane, two keys a column): P is the A operand of P V, so neither its stores nor its reads pass through shared memory,
  // whose 128 bytes a cycle bound a tile (64 KB in from memory, 112 KB of operands for the scores, 48 KB of V: 1800 cycles; with P
  // in shared memory 2300)
  static constexpr int S_COLS = NP * TILE;
  static constexpr int O_COL0 = 2 * S_COLS, O_COLS = HD;
  static constexpr int P_COL0 = O_COL0 + O_COLS, P_COLS = NP * TILE / 2;
  static constexpr int TMEM_COLS = P_COL0 + 2 * P_COLS <= 256 ? 256 : 512;
  static_assert(RING_BYTES >= MERGE_BYTES && RING_BYTES >= BUF_BYTES + QROWS * 16, "what follows the last tile must fit in the ring");
  static_assert(P_COL0 + 2 * P_COLS <= 512, "tensor memory");
  static_assert(SMEM_BYTES <= 232448, "shared memory of one SM");
};

template <int HD, int QROWS, int NP>
__global__ void __launch_bounds__(AttCfg<HD, QROWS, NP>::NTHREADS, 1)
tree_attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const AttArgs a) {
  using C = AttCfg<HD, QROWS, NP>;
  constexpr int NSK = C::NSK, NSV = C::NSV;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t q_s = base, ring_s = q_s + C::Q_BYTES, vring_s = ring_s + C::KRING_BYTES;
  const uint32_t xm_s = ring_s + C::RING_BYTES;
  const uint32_t bars = xm_s + C::XM_BYTES;
  const uint32_t q_full = bars;
  auto k_full = [&](int s) { return bars + 8u * (1 + s); };
  auto k_empty = [&](int s) { return bars + 8u * (1 + NSK + s); };
  auto v_full = [&](int s) { return bars + 8u * (1 + 2 * NSK + s); };
  auto v_empty = [&](int s) { return bars + 8u * (1 + 2 * NSK + NSV + s); };
  constexpr int B0 = 1 + 2 * NSK + 2 * NSV;
  auto s_full = [&](int i) { return bars + 8u * (B0 + i); };
  auto s_empty = [&](int i) { return bars + 8u * (B0 + 2 + i); };
  auto p_full = [&](int i) { return bars + 8u * (B0 + 4 + i); };
  auto pv_done = [&](int i) { return bars + 8u * (B0 + 6 + i); };
  const uint32_t o_done = bars + 8u * (B0 + 8);          // every P V product of the chunk
  auto xm_bar = [&](int g, int quad) { return bars + 8u * (B0 + 9 + C::NQUAD * g + quad); };   // group g has left the quadrant's reference maxima
  const uint32_t tmem_slot = bars + 8u * C::NBAR;
  __shared__ int s_abort;

  const RowSet& rs = a.rs;
  const int h = blockIdx.x, b = blockIdx.y, c = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nchunks = a.nchunks, H = a.H;

  if (tid == 0) {
    s_abort = 0;
    mbar_init(q_full, 1); mbar_init(o_done, 1);
    for (int s = 0; s < NSK; ++s) { mbar_init(k_full(s), 1); mbar_init(k_empty(s), 1); }
    for (int s = 0; s < NSV; ++s) { mbar_init(v_full(s), 1); mbar_init(v_empty(s), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(s_full(i), 1); mbar_init(s_empty(i), C::NQUAD); mbar_init(p_full(i), C::NQUAD); mbar_init(pv_done(i), 1); }
    for (int i = 0; i < 2 * C::NQUAD; ++i) mbar_init(xm_bar(0, i), 1);
    mbar_init_fence();
    prefetch_tensormap(&tmQ); prefetch_tensormap(&tmK); prefetch_tensormap(&tmV);
  }
  if (warp == C::W_MMA) tmem_alloc(tmem_slot, C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  // q and the new cache rows are the preceding kernel's output.  With a.early the lengths and the committed cache rows
  // are known to be older than anything still in flight, so the producer requests committed tiles before it waits.
  if (!a.early) pdl_wait();
  uint32_t tmem_base;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));

  int nr, p_call, p0, seq, q_row0;                       // p_call: first cache slot written by this forward call; p0: first slot of this CTA's rows
  if (rs.blocks) {
    const AttBlock blk = rs.blocks[b];
    seq = blk.seq; q_row0 = blk.row0; nr = min(blk.n, QROWS); p0 = blk.pos0; p_call = blk.call0;
  } else {
    seq = b; q_row0 = b * rs.tc;
    nr = min(rs.n_rows ? rs.n_rows[b] : rs.tc, QROWS);
    p0 = p_call = rs.pos0[b];
  }
  const int total = p0 + nr;
  const int nt = (total + TILE - 1) / TILE;
  const int tile0 = chunk_first_tile(c, nt, nchunks), tile1 = chunk_first_tile(c + 1, nt, nchunks);
  const bool has_work = tile0 < tile1 && nr > 0 && p0 >= 0 && total <= a.max_seq;
  const int ntiles = has_work ? tile1 - tile0 : 0;
  const uint32_t limit = a.wait_limit;
  const int rows_cap = rs.blocks ? nr : min(rs.tc, QROWS);     // output rows of this pair; those past nr get zeros

  if (warp == C::W_PRODUCER) {
    if (lane == 0 && has_work) {
      const uint64_t pol = policy_evict_first(), pol_q = policy_evict_last();
      const int row0 = (seq * H + h) * a.max_seq;
      auto request_k = [&](int i) {
        const int s = i % NSK;
        const uint32_t k_dst = ring_s + s * C::K_BYTES;
        const int r = row0 + (tile0 + i) * TILE;
        mbar_arrive_expect_tx(k_full(s), C::K_BYTES);
#pragma unroll
        for (int pl = 0; pl < NP; ++pl)
#pragma unroll
          for (int hf = 0; hf < C::NHALF; ++hf)
            tma_load_2d(k_dst + hf * C::KH_BYTES + pl * TILE * 128, &tmK, hf * 64, pl * a.kv_plane_rows + r, k_full(s), pol);
      };
      auto request_v = [&](int i) {
        const int s = i % NSV;
        const uint32_t v_dst = vring_s + s * C::V_BYTES;
        const int r = row0 + (tile0 + i) * TILE;
        mbar_arrive_expect_tx(v_full(s), C::V_BYTES);
#pragma unroll
        for (int pl = 0; pl < NP; ++pl)
#pragma unroll
          for (int hf = 0; hf < C::NHALF; ++hf)
            tma_load_2d(v_dst + (pl * C::NHALF + hf) * TILE * 128, &tmV, hf * 64, pl * a.kv_plane_rows + r, v_full(s), pol);
      };
      int nk = 0, nv = 0;                                  // next K and V tile to request
      if (a.early) {                                       // committed rows only
        for (; nk < ntiles && nk < NSK && (tile0 + nk + 1) * TILE <= p_call; ++nk) {
          request_k(nk);
          if (nv == nk && nv < NSV) request_v(nv++);
        }
        pdl_wait();
      }
      mbar_arrive_expect_tx(q_full, C::Q_BYTES);
#pragma unroll
      for (int pl = 0; pl < NP; ++pl)
#pragma unroll
        for (int hf = 0; hf < C::NHALF; ++hf)
          tma_load_2d(q_s + pl * C::QP_BYTES + hf * QROWS * 128, &tmQ, h * HD + hf * 64, pl * a.q_plane_rows + q_row0, q_full, pol_q);
      // K stage i % NSK was last read by the scores of tile i - NSK (completion i / NSK - 1 of its empty barrier), V stage
      // i % NSV by the P V product of tile i - NSV; whichever ring has room is served first, K ahead of V
      uint32_t idle = 0;
      while (nk < ntiles || nv < ntiles) {
        bool did = false;
        if (nk < ntiles && (nk < NSK || mbar_test(k_empty(nk % NSK), (uint32_t)((nk / NSK - 1) & 1)))) { request_k(nk++); did = true; }
        if (nv < nk && (nv < NSV || mbar_test(v_empty(nv % NSV), (uint32_t)((nv / NSV - 1) & 1)))) { request_v(nv++); did = true; }
        if (did) idle = 0;
        else if (++idle > limit) { atomicOr(a.status, ST_TIMEOUT); s_abort = 1; break; }
      }
    }
  } else if (warp == C::W_MMA) {
    if (lane == 0 && has_work) {
      constexpr uint32_t idesc_s = instr_desc_f16(0, C::MROWS, NP * TILE, 0);      // Q_hi x [K_hi ; K_lo]
      constexpr uint32_t idesc_s2 = instr_desc_f16(0, C::MROWS, TILE, 0);          // Q_lo x K_hi
      constexpr uint32_t idesc_pv = instr_desc_f16(0, C::MROWS, HD, 1);            // P x V
      // operand descriptors: built once; a byte offset inside shared memory adds offset / 16 to the start-address field
      const uint64_t q_desc = smem_desc_sw128(q_s), k_desc = smem_desc_sw128(ring_s),
                     v_desc = smem_desc_sw128_mn(vring_s, TILE * 128);
      bool ok = mbar_wait(q_full, 0, limit);
      auto issue_s = [&](int i) {                        // S_i = Q K_i^T into score buffer i & 1
        const int s = i % NSK;
        tc_fence_after();
        const uint64_t kd = k_desc + (uint64_t)((s * C::K_BYTES) >> 4);
        const uint32_t d_s = tmem_base + (uint32_t)((i & 1) * C::S_COLS);
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk)
          umma_f16(d_s, q_desc + (uint64_t)(((kk >> 2) * QROWS * 128 + (kk & 3) * 32) >> 4),
                   kd + (uint64_t)(((kk >> 2) * C::KH_BYTES + (kk & 3) * 32) >> 4), idesc_s, (uint32_t)(kk != 0));
        if (NP == 2) {
#pragma unroll
          for (int kk = 0; kk < HD / 16; ++kk)
            umma_f16(d_s, q_desc + (uint64_t)((C::QP_BYTES + (kk >> 2) * QROWS * 128 + (kk & 3) * 32) >> 4),
                     kd + (uint64_t)(((kk >> 2) * C::KH_BYTES + (kk & 3) * 32) >> 4), idesc_s2, 1u);
        }
        umma_commit(k_empty(s));                        // frees the K stage once these MMAs have read it
        umma_commit(s_full(i & 1));
      };
      auto issue_pv = [&](int i) {
        const int s = i % NSV;
        tc_fence_after();
        const uint64_t vd = v_desc + (uint64_t)((s * C::V_BYTES) >> 4);
        const uint32_t d_o = tmem_base + (uint32_t)C::O_COL0, p_t = tmem_base + (uint32_t)(C::P_COL0 + (i & 1) * C::P_COLS);
#pragma unroll
        for (int kk = 0; kk < TILE / 16; ++kk)             // P_hi V_hi
          umma_f16_ts(d_o, p_t + (uint32_t)(kk * 8), vd + (uint64_t)((kk * 2048) >> 4), idesc_pv, (uint32_t)((i | kk) != 0));
        if (NP == 2) {
#pragma unroll
          for (int kk = 0; kk < TILE / 16; ++kk) {         // + P_hi V_lo + P_lo V_hi
            umma_f16_ts(d_o, p_t + (uint32_t)(kk * 8), vd + (uint64_t)((C::V_BYTES / 2 + kk * 2048) >> 4), idesc_pv, 1u);
            umma_f16_ts(d_o, p_t + (uint32_t)(TILE / 2 + kk * 8), vd + (uint64_t)((kk * 2048) >> 4), idesc_pv, 1u);
          }
        }
        umma_commit(v_empty(s));
        umma_commit(pv_done(i & 1));
      };
      // S_i waits for its K tile and for the softmax group to have read S_(i-2); P_i V_i for P_i and its V tile
      int is = 0, ip = 0;
      uint32_t idle = 0;
      while (ok && ip < ntiles) {
        bool did = false;
        if (is < ntiles && (is < 2 || mbar_test(s_empty(is & 1), (uint32_t)(((is >> 1) - 1) & 1))) && mbar_test(k_full(is % NSK), (uint32_t)((is / NSK) & 1))) {
          issue_s(is++); did = true;
        }
        if (ip < is && mbar_test(p_full(ip & 1), (uint32_t)((ip >> 1) & 1)) && mbar_test(v_full(ip % NSV), (uint32_t)((ip / NSV) & 1))) {
          issue_pv(ip++); did = true;
        }
        if (did) idle = 0;
        else if (++idle > limit) ok = false;
      }
      if (ok) umma_commit(o_done);
      if (!ok) { atomicOr(a.status, ST_TIMEOUT); s_abort = 1; }
    }
  } else if ((warp & 3) < C::NQUAD) {
    // ---- softmax warps: thread = accumulator row = a tensor-memory lane of the warp's quadrant
    const int quad = warp & 3, grp = warp >> 2, row = quad * 32 + lane;
    const bool warp_rows = quad * 32 < nr;            // any row of this warp in use
    const bool row_live = row < nr;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
    const uint64_t mask = (row_live && rs.mask) ? rs.mask[row] : 0ull;
    const bool causal = rs.mask == nullptr;
    const float sc = rsqrtf((float)HD) * 1.4426950408889634f;   // 1/sqrt(hd) * log2(e)
    float m_ref = -INFINITY, l = 0.f;                     // after this group's last tile; l: the sum over its tiles
    bool ok = true;
    const int gt = quad * 32 + lane;                      // thread of the group
    for (int i = grp; i < ntiles; i += 2) {
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }     // a wait that ran out in one lane ends the walk for the whole warp
      const int t0 = (tile0 + i) * TILE;
      if (!mbar_wait(s_full(grp), (uint32_t)((i >> 1) & 1), limit)) { ok = false; break; }
      tc_fence_after();
      f32x2 s2[TILE / 2];                                  // raw scores, two keys each
      if (warp_rows) {
        const uint32_t s_addr = lane_addr + (uint32_t)(grp * C::S_COLS);
#pragma unroll
        for (int c0 = 0; c0 < TILE; c0 += 32) {            // NP = 2: the two column halves of the score buffer, added
          uint32_t x[32], y[32];
          if constexpr (NP == 1) tmem_ld32(s_addr + (uint32_t)c0, x); else tmem_ld32x2(s_addr + (uint32_t)c0, s_addr + (uint32_t)(TILE + c0), x, y);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const f32x2 v = pack2(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1]));
            if constexpr (NP == 1) s2[c0 / 2 + j] = v;
            else s2[c0 / 2 + j] = add2(v, pack2(__uint_as_float(y[2 * j]), __uint_as_float(y[2 * j + 1])));
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(s_empty(grp));
      if (warp_rows) {
        if (t0 + TILE > p0) {                              // the tile reaches into the new rows (or past the end): hide keys
          // visibility word of this row for the tile's 64 keys (bit j: key t0 + j)
          uint64_t vis = 0ull;
          if (row_live) {
            const int shift = t0 - p0;                     // new-slot index of the tile's first key; negative: it is a committed row
            if (causal) {                                  // new slots 0..row: keys j <= row - shift
              const int n = row - shift + 1;
              vis = n >= 64 ? ~0ull : (n <= 0 ? 0ull : ((1ull << n) - 1ull));
            } else if (shift >= 0) {
              vis = shift < 64 ? mask >> shift : 0ull;
            } else {
              vis = (mask << (-shift)) | ((1ull << (-shift)) - 1ull);
            }
            const int nv = total - t0;                     // keys of the tile that exist
            if (nv < 64) vis &= (1ull << nv) - 1ull;
          }
#pragma unroll
          for (int j = 0; j < TILE / 2; ++j) {
            const float2 v = unpack2(s2[j]);
            s2[j] = pack2((vis >> (2 * j)) & 1ull ? v.x : -INFINITY, (vis >> (2 * j + 1)) & 1ull ? v.y : -INFINITY);
          }
        }
        float mx = -INFINITY, mx1 = -INFINITY;             // scores of dead rows are whatever Q holds there; nothing of theirs is used
#pragma unroll
        for (int j = 0; j < TILE / 2; j += 2) {
          const float2 v = unpack2(s2[j]), v1 = unpack2(s2[j + 1]);
          mx = max3(mx, v.x, v.y); mx1 = max3(mx1, v1.x, v1.y);
        }
        mx = fmaxf(mx, mx1) * sc;
        // the reference maximum after tile i - 1 from the other group's warp of the quadrant, the one after this tile back to it
        float m_in = -INFINITY;
        const uint32_t xm = xm_s + (uint32_t)(row * 4);
        if (i > 0) {
          if (!mbar_wait(xm_bar(grp ^ 1, quad), (uint32_t)(((i - 1) >> 1) & 1), limit)) { ok = false; break; }
          asm volatile("ld.shared.f32 %0, [%1];" : "=f"(m_in) : "r"(xm + (uint32_t)((grp ^ 1) * QROWS * 4)) : "memory");
        }
        const float m_new = mx > m_in + RESCALE_STEP ? mx : m_in;      // also the first finite maximum (m_in = -inf)
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(xm + (uint32_t)(grp * QROWS * 4)), "f"(m_new) : "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(xm_bar(grp, quad));
        const bool rescale = row_live && m_in != -INFINITY && m_new != m_in;
        if (m_ref != m_new) l *= ex2(m_ref - m_new);
        m_ref = m_new;
        const float bse = m_new == -INFINITY ? 0.f : -m_new;
        const f32x2 sc2 = pack2(sc, sc), bse2 = pack2(bse, bse);
        f32x2 sum2 = 0ull;
        uint32_t ph[TILE / 2], pl[NP == 2 ? TILE / 2 : 1];
#pragma unroll
        for (int j = 0; j < TILE / 2; ++j) {
          const float2 e = unpack2(fma2(s2[j], sc2, bse2));
          const f32x2 p = pack2(ex2(e.x), ex2(e.y));
          const float2 pv = unpack2(p);
          ph[j] = pack_half2(pv.x, pv.y);
          const __half2 hv = *reinterpret_cast<const __half2*>(&ph[j]);
          const f32x2 hi = pack2(__low2float(hv), __high2float(hv));
          if constexpr (NP == 1) {
            sum2 = add2(sum2, hi);                         // the sum of what the MMA will really weigh V with
          } else {
            sum2 = add2(sum2, p);
            const float2 lo = unpack2(fma2(hi, pack2(-1.f, -1.f), p));       // lo = f16(p - f16(p))
            pl[j] = pack_half2(lo.x, lo.y);
          }
        }
        const float2 sum = unpack2(sum2);
        l += sum.x + sum.y;
        if (i >= 2 && !mbar_wait(pv_done(grp), (uint32_t)(((i - 2) >> 1) & 1), limit)) { ok = false; break; }      // the P buffer is free
        if (__any_sync(0xffffffffu, rescale)) {
          const float alpha = rescale ? ex2(m_in - m_new) : 1.f;
          // P V of tile i - 2 is done, so the other buffer's barrier is at tile i - 1; it cannot pass it before this tile's P
          if (i >= 1 && !mbar_wait(pv_done((i - 1) & 1), (uint32_t)(((i - 1) >> 1) & 1), limit)) { ok = false; break; }
          tc_fence_after();
#pragma unroll 1
          for (int c0 = 0; c0 < C::O_COLS; c0 += 32) {
            uint32_t o[32];
            tmem_ld32(lane_addr + (uint32_t)(C::O_COL0 + c0), o);
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * alpha);
            tmem_st32(lane_addr + (uint32_t)(C::O_COL0 + c0), o);
          }
        }
        tc_fence_after();                                  // the product that read this buffer is over
        const uint32_t p_addr = lane_addr + (uint32_t)(C::P_COL0 + grp * C::P_COLS);
        tmem_st32(p_addr, ph);
        if constexpr (NP == 2) tmem_st32(p_addr + (uint32_t)(TILE / 2), pl);
      } else {
        if (i >= 2 && !mbar_wait(pv_done(grp), (uint32_t)(((i - 2) >> 1) & 1), limit)) { ok = false; break; }
      }
      if (t0 + TILE > total) {
        // rows of the V tile past the end of the sequence hold whatever the cache holds: zero them, so that a
        // zero weight times a non-finite stale value cannot reach the accumulator
        const int s = i % NSV;
        if (!mbar_wait(v_full(s), (uint32_t)((i / NSV) & 1), limit)) { ok = false; break; }
        const uint32_t v_src = vring_s + s * C::V_BYTES;
        const int first = total - t0;                       // first row to clear (>= 1)
        constexpr int BLK = NP * C::NHALF;                  // 64-column blocks of a V tile
        for (int e = gt; e < (TILE - first) * BLK * 8; e += QROWS) {
          const int rr = first + e / (BLK * 8), rem = e % (BLK * 8);
          const uint32_t dst = v_src + (uint32_t)((rem >> 3) * TILE * 128 + rr * 128 + (rem & 7) * 16);
          asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(dst), "r"(0u) : "memory");
        }
        fence_proxy_async();                               // the cleared rows become visible to the tensor core
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full(grp));
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) { atomicOr(a.status, ST_TIMEOUT); s_abort = 1; }
    // (not pv_done of the last tile: a group does not follow the other's phases, and a parity only tells neighbouring ones apart)
    if (ok && ntiles > 0 && !mbar_wait(o_done, 0, limit)) {
      ok = false; atomicOr(a.status, ST_TIMEOUT); s_abort = 1;
    }
    ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    // 32 output columns of this thread's row in one tensor-memory round trip
    auto read_o = [&](int c0, uint32_t (&o)[32]) { tmem_ld32(lane_addr + (uint32_t)(C::O_COL0 + c0), o); };
    if (nchunks == 1) {
      // the other group's maximum and sum; the output is relative to the larger maximum (the one after the last tile)
      const uint32_t xl = ring_s + (uint32_t)(C::BUF_BYTES + row * 16);
      asm volatile("st.shared.v2.f32 [%0], {%1,%2};" ::"r"(xl + (uint32_t)grp * 8u), "f"(m_ref), "f"(l) : "memory");
      asm volatile("bar.sync 1, %0;" ::"n"(2 * QROWS) : "memory");       // the softmax warps
      const float4 ml = ld_smem4(xl);
      const float M = fmaxf(ml.x, ml.z);
      const bool have = ok && row_live && M != -INFINITY;
      const float L = have ? ml.y * ex2(ml.x - M) + ml.w * ex2(ml.z - M) : 0.f;
      const float inv = L > 0.f ? 1.f / L : 0.f;
      if (a.early) pdl_wait();                             // (the producer lane has waited already) before the first global store
      const int w_rows = min(32, rows_cap - quad * 32);    // rows of this warp that exist
      const uint32_t buf = ring_s + (uint32_t)(grp * C::NQUAD + quad) * (2 * 32 * 128);
      if (ok && w_rows > 0) {
#pragma unroll 1
        for (int c0 = grp * 64; c0 < HD; c0 += 128) {        // the two warps of a quadrant take every other block of 64 columns
#pragma unroll 1
          for (int c1 = 0; c1 < 64; c1 += 32) {
            uint32_t o[32];
            if (ntiles > 0) read_o(c0 + c1, o);
#pragma unroll
            for (int j = 0; j < 4; ++j) {                  // 8 columns: 16 bytes of either plane; piece p of row `lane` sits at position p ^ (lane & 7)
              uint32_t hi[4], lo[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const float x = have ? __uint_as_float(o[8 * j + 2 * k]) * inv : 0.f, y = have ? __uint_as_float(o[8 * j + 2 * k + 1]) * inv : 0.f;
                const __nv_bfloat162 hv = __floats2bfloat162_rn(x, y);
                const __nv_bfloat162 lv = __floats2bfloat162_rn(x - __low2float(hv), y - __high2float(hv));
                hi[k] = *reinterpret_cast<const uint32_t*>(&hv); lo[k] = *reinterpret_cast<const uint32_t*>(&lv);
              }
              const uint32_t dst = buf + (uint32_t)(lane * 128 + (((c1 / 8 + j) ^ (lane & 7)) * 16));
              asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(hi[0]), "r"(hi[1]), "r"(hi[2]), "r"(hi[3]) : "memory");
              asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst + 32u * 128u), "r"(lo[0]), "r"(lo[1]), "r"(lo[2]), "r"(lo[3]) : "memory");
            }
          }
          __syncwarp();
          const int piece = lane & 7;
#pragma unroll 4
          for (int it = 0; it < 8; ++it) {
            const int i = it * 4 + (lane >> 3);
            if (i < w_rows) {
              const uint32_t src = buf + (uint32_t)(i * 128 + ((piece ^ (i & 7)) * 16));
              bf16* dst = a.out + (size_t)(q_row0 + quad * 32 + i) * (H * HD) + h * HD + c0 + piece * 8;
              *reinterpret_cast<float4*>(dst) = ld_smem4(src);
              if (a.out_ps) *reinterpret_cast<float4*>(dst + a.out_ps) = ld_smem4(src + 32u * 128u);
            }
          }
          __syncwarp();
        }
      }
    } else {
      if (ok && ntiles > 0 && warp_rows) {
        const uint32_t xo = ring_s + (uint32_t)row * (HD * 4);
#pragma unroll 1
        for (int c0 = grp * (HD / 2); c0 < (grp + 1) * (HD / 2); c0 += 32) {       // the two warps of a quadrant take half of the columns each
          uint32_t o[32];
          read_o(c0, o);
#pragma unroll
          for (int j = 0; j < 8; ++j)                      // float4 piece k4 of row i sits at position k4 ^ (i & (HD/4 - 1))
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(xo + (uint32_t)(((c0 / 4 + j) ^ (row & (HD / 4 - 1))) * 16)),
                         "r"(o[4 * j]), "r"(o[4 * j + 1]), "r"(o[4 * j + 2]), "r"(o[4 * j + 3]) : "memory");
        }
      }
      const bool have = ok && row_live;
      asm volatile("st.shared.v2.f32 [%0], {%1,%2};" ::"r"(ring_s + (uint32_t)(QROWS * HD * 4 + row * 16 + grp * 8)),
                   "f"(have ? m_ref : -INFINITY), "f"(have ? l : 0.f) : "memory");
    }
  }
  __syncwarp();                                           // the one-lane roles rejoin their warps before the block-wide barrier
  tc_fence_before();
  if (nchunks == 1) {
    __syncthreads();
  } else {
    cluster_sync_all();                                   // every chunk's rows are in its shared memory
    if (a.early) pdl_wait();                              // (the producer lane has waited already) before the first global store
    // out[r][h][:] = sum_c o_c 2^(m_c - M) / sum_c l_c 2^(m_c - M), chunks in order, M the maximum so far; this CTA takes
    // rows c, c + nchunks, ...; the loads of up to four chunks are in flight together
    constexpr int V4 = HD / 4;
    const int d = H * HD;
    const int my_rows = rows_cap > c ? (rows_cap - c + nchunks - 1) / nchunks : 0;
#pragma unroll 1
    for (int e = tid; e < my_rows * V4 && !s_abort; e += C::NTHREADS) {
      const int k4 = e % V4, i = c + (e / V4) * nchunks;
      const uint32_t xo = ring_s + (uint32_t)(i * (HD * 4) + ((k4 ^ (i & (V4 - 1))) * 16)), xml = ring_s + (uint32_t)(QROWS * HD * 4 + i * 16);
      float M = -INFINITY, L = 0.f;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
      for (int c0 = 0; c0 < nchunks; c0 += 4) {
        float4 ml[4], v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          ml[u] = make_float4(-INFINITY, 0.f, -INFINITY, 0.f); v[u] = acc;
          if (c0 + u < nchunks) { ml[u] = ld_peer4(peer_smem(xml, (uint32_t)(c0 + u))); v[u] = ld_peer4(peer_smem(xo, (uint32_t)(c0 + u))); }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float mu = fmaxf(ml[u].x, ml[u].z);        // the output is relative to the larger maximum of the two groups
          if (mu != -INFINITY) {                           // a chunk that saw no key of this row holds anything at all in its place
            const float m1 = fmaxf(M, mu), f = ex2(M - m1), w = ex2(mu - m1);
            M = m1;
            L = L * f + ml[u].y * ex2(ml[u].x - m1) + ml[u].w * ex2(ml[u].z - m1);
            acc.x = acc.x * f + v[u].x * w; acc.y = acc.y * f + v[u].y * w; acc.z = acc.z * f + v[u].z * w; acc.w = acc.w * f + v[u].w * w;
          }
        }
      }
      const float inv = L > 0.f ? 1.f / L : 0.f;
      acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
      bf16* dst = a.out + (size_t)(q_row0 + i) * d + h * HD + k4 * 4;      // rows past nr get zeros
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(acc.x, acc.y), h1 = __floats2bfloat162_rn(acc.z, acc.w);
      *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
      if (a.out_ps) {
        const __nv_bfloat162 l0 = __floats2bfloat162_rn(acc.x - __low2float(h0), acc.y - __high2float(h0));
        const __nv_bfloat162 l1 = __floats2bfloat162_rn(acc.z - __low2float(h1), acc.w - __high2float(h1));
        *reinterpret_cast<uint2*>(dst + a.out_ps) = make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
      }
    }
    cluster_sync_all();                                   // peers may still be reading this CTA's rows
  }
  if (s_abort) {                                          // let copies in flight land before the CTA retires
    for (int i = 0; i < 2000; ++i) __nanosleep(100);
  }
  if (warp == C::W_MMA) { tc_fence_after(); tmem_dealloc(tmem_base, C::TMEM_COLS); }
}

// Number of KV chunks per (head, sequence) or (head, block): the count (at most 8) with the least estimated time, in tiles; ties go
// to fewer chunks.  One CTA per SM (the rings take nearly all of its shared memory), nt tiles in the longest pair, `tiles` in
// all of a head's.  Besides its tiles a CTA pays about 3 tiles' time for set-up and its result, with a merge 4 and one more per 32
// rows (measured: 3.9 us, 7.3 with 64 rows, 10.5 with 128 at 1.35 us a tile).  Packed prompt blocks come longest first, so the SMs
// even out: the longest CTA or the mean load counts.  Otherwise all pairs may have nt tiles: whole waves count.
// 32 pairs of 10 tiles, 64 rows: 1, 2, 3, 4, 5 chunks take 18.1, 15.1, 13.6, 12.0, 21.8 us; 256 pairs of up to 18: 46.7 and 74 us.
// Blocks of prompts (192 of up to 10 tiles): 1, 2, 3 chunks take 27.7, 41.5, 55.6 us.
int pick_chunks(int pairs, int nt, long tiles, bool packed, int rows, int sms) {
  int hi = nt < MAX_CHUNKS ? nt : MAX_CHUNKS;
  if (hi < 1) hi = 1;
  auto cost = [&](int n) -> double {
    const double own = n == 1 ? 3 : 4 + rows / 32, longest = (double)nt / n + own;
    return packed ? std::max(longest, (tiles + pairs * n * own) / sms) : (pairs * n + sms - 1) / sms * longest;
  };
  int best = 1; double best_cost = cost(1);
  for (int n = 2; n <= hi; ++n)
    if (cost(n) < best_cost) { best = n; best_cost = cost(n); }
  return best;
}

template <int HD, int QROWS, int NP>
hydra_status run(const __half* q, int q_rows, const __half* kc, const __half* vc, int cache_batch, RowSet rs, bf16* out, size_t out_ps,
                 int H, int max_seq, int len_upper, int* status, bool stable_lengths, cudaStream_t st) {
  using C = AttCfg<HD, QROWS, NP>;
  CUtensorMap tq, tk, tv;
  const uint64_t cache_rows = (uint64_t)cache_batch * H * max_seq;
  if (cache_rows * NP > 0x7fffffffull) return HYDRA_ERR_UNSUPPORTED;          // tensor-map row coordinates are 32-bit
  if (!get_tensor_map(q, (uint64_t)NP * q_rows, (uint64_t)H * HD, QROWS, true, &tq) ||
      !get_tensor_map(kc, NP * cache_rows, HD, TILE, true, &tk) || !get_tensor_map(vc, NP * cache_rows, HD, TILE, true, &tv)) {
    set_last_error("cuTensorMapEncodeTiled", cudaErrorUnknown);
    return HYDRA_ERR_CUDA;
  }
  static PerDeviceFlag attr_done;
  if (!attr_done.get()) {
    HYDRA_CUDA(cudaFuncSetAttribute(tree_attn_tc_kernel<HD, QROWS, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES));
    attr_done.set();
  }
  AttArgs a{};
  a.rs = rs; a.out = out; a.out_ps = out_ps; a.H = H; a.max_seq = max_seq; a.status = status; a.wait_limit = WAIT_LIMIT;
  a.q_plane_rows = q_rows; a.kv_plane_rows = (int)cache_rows; a.early = stable_lengths ? 1 : 0;
  const int groups = rs.blocks ? rs.n_blocks : rs.batch;
  a.nchunks = pick_chunks(H * groups, (len_upper + TILE - 1) / TILE, (long)H * rs.n_tiles, rs.blocks != nullptr, rs.blocks ? QROWS : rs.tc, sm_count());
  if (a.nchunks == 1 && ((uintptr_t)out & 15)) a.nchunks = 2;      // one chunk writes 16 bytes at a time, the merge 8
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(H, groups, a.nchunks); cfg.blockDim = dim3(C::NTHREADS); cfg.dynamicSmemBytes = C::SMEM_BYTES; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = (unsigned)a.nchunks;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  HYDRA_CUDA(cudaLaunchKernelEx(&cfg, tree_attn_tc_kernel<HD, QROWS, NP>, tq, tk, tv, a));
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

template <int NP>
hydra_status dispatch(const __half* q, int q_rows, const __half* kc, const __half* vc, int cache_batch, RowSet rs, bf16* out, size_t out_ps,
                      int H, int hd, int max_seq, int len_upper, int* status, bool stable_lengths, cudaStream_t st) {
  const bool wide = rs.blocks || rs.tc > 64;
  if (hd == 128) return wide ? run<128, 128, NP>(q, q_rows, kc, vc, cache_batch, rs, out, out_ps, H, max_seq, len_upper, status, stable_lengths, st)
                             : run<128, 64, NP>(q, q_rows, kc, vc, cache_batch, rs, out, out_ps, H, max_seq, len_upper, status, stable_lengths, st);
  if (hd == 64) return wide ? run<64, 128, NP>(q, q_rows, kc, vc, cache_batch, rs, out, out_ps, H, max_seq, len_upper, status, stable_lengths, st)
                            : run<64, 64, NP>(q, q_rows, kc, vc, cache_batch, rs, out, out_ps, H, max_seq, len_upper, status, stable_lengths, st);
  return HYDRA_ERR_UNSUPPORTED;
}

}  // namespace


hydra_status tree_attention_tc(const __half* q, int q_rows, const __half* kc, const __half* vc, int cache_batch, int planes, RowSet rs,
                               bf16* out, size_t out_ps, int H, int hd, int max_seq, int len_upper, int* status, bool stable_lengths,
                               cudaStream_t st) {
  if ((!rs.blocks && (rs.tc > 128 || (rs.mask && rs.tc > 64))) || (planes != 1 && planes != 2)) return HYDRA_ERR_UNSUPPORTED;
  if (!tensor_map_encoder_available()) { set_last_error("cuTensorMapEncodeTiled entry point", cudaErrorUnknown); return HYDRA_ERR_CUDA; }
  if (((uintptr_t)q | (uintptr_t)kc | (uintptr_t)vc) & 15) return HYDRA_ERR_INVALID;
  // One row always: 3 to 48 % faster, 40 to 32000 keys, 1 to 64 sequences of 8 to 52 heads; two sequences of 32 heads with one plane from 8000 keys on 1 to 2 % slower.
  // Two rows up to 1024 keys: 0.53 to 0.95 of the time at 40 to 160 keys; at 1000 1 sequence of 32 heads 12.8 / 11.8 us, 8 52.7 / 51.4, 16 107 / 99, but 2 17.2 / 17.4, 4 26.2 / 27.5, 5 45.4 /
  // 48.1 (kept: with one plane the weights of these rows are float, not float16), 2 of 2400 31.1 / 32.2.  Four rows took as long at 160 keys and 10 to 40 % longer above.
  if (!rs.blocks && (rs.tc == 1 || (rs.tc == 2 && len_upper <= 1024)))
    return tree_attention_rows(q, q_rows, kc, vc, cache_batch, planes, rs, out, out_ps, H, hd, max_seq, len_upper, stable_lengths, st);
  return planes == 2 ? dispatch<2>(q, q_rows, kc, vc, cache_batch, rs, out, out_ps, H, hd, max_seq, len_upper, status, stable_lengths, st)
                     : dispatch<1>(q, q_rows, kc, vc, cache_batch, rs, out, out_ps, H, hd, max_seq, len_upper, status, stable_lengths, st);
}

}  // namespace hydra
