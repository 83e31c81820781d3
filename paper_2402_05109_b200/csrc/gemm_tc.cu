// Weight-streaming bfloat16 GEMM on the sm_100a tensor cores: persistent, stream-K, TMA + tcgen05 + TMEM.
//
//   part[slot][m][n] = sum over one K range of x[m][k] * w[n][k]        (float accumulate, float out)
//
// The weight matrix is the large operand (read once from HBM); the activation slab is small (tree rows x
// batch) and L2 resident.  So the roles are swapped with respect to the usual GEMM: weight rows [n][64 k] are the MMA "A"
// operand (M: TMEM lanes), activation rows [64 k] the "B" operand (N: TMEM columns).  Both are K-major and land in shared
// memory through TMA with the 128-byte swizzle; accumulators live in tensor memory.
//
// Work decomposition (stream-K): the (tile, k-block) pairs of the whole GEMM are laid out in one line,
// tile-major, and cut into equal contiguous ranges, one per CTA, so that every SM
// streams the same number of weight bytes without interruption.  A CTA's range covers the tail of one tile,
// possibly whole tiles, and the head of another; each such run is a "segment" whose partial sum goes to
// slot (CTA - first CTA of the tile) of the partial buffer.  The consumer kernel adds the slots of a tile in
// fixed order (SplitDesc), so results are deterministic.
// Several row tiles: the line is that of the weight tiles alone, and a group of neighbouring CTAs, one for each row tile, walks a range of it together, so
// that they read the same weights at the same time and those come from memory once.  (One line of all tiles, row tiles next to each other, had them read the same
// weights a third of the kernel's time apart: 768 x 22016 x 4096 read 505 MB, 203 so, for 180 MB of weights; 768 x 4096 x 11008 147 and 124.  The tensor cores
// run at the clock that power leaves them, so it shows in time: layers of a 7B prompt pass of 768 / 675 / 512 / 300 rows 544 / 523 / 382 / 274 -> 522 / 488 / 371 / 250 us,
// of the 13B shape 768 rows 901 -> 876, of the 33B shape 512 rows 884 -> 849.  Weights marked to go first: 6 us less a 7B layer than left to the L2.)
// (Ranges that end with the tiles where that makes them at most 5 % longer - 144 whole tiles of 768 x 12288 on 147 CTAs - leave fewer partial sums, 522 -> 500 us,
// but longer ones, and with those the error below: 6.6e-6 -> 9.3e-6.  Not done.)
//
// A unit is 64 k of NH = 1 or 2 weight tiles of 128 rows (one TMA box, one accumulator each) that share the activation tile.
//
// Warp roles (192 threads): warp 0 = TMA producer (one lane), warp 1 = TMEM allocation + MMA issue (one
// lane), warps 2..5 = epilogue (TMEM -> registers -> global, coalesced along n).  Two accumulator sets in
// TMEM (where 512 columns allow) let the epilogue of one segment overlap the main loop of the next.  The kernel is launched with
// programmatic stream serialisation: the weight tiles of a context's call (no kernel writes those) are requested
// before griddepcontrol.wait, activations and all global writes after it.  A stand-alone call takes any matrix as w, the preceding
// kernel's result included, so it only fetches the first tiles into the L2 (which changes nothing that is read) and requests them after the wait.
// Precision: weights are bfloat16 (exact: the reference model's weights are the same bfloat16 values).  The
// activation operand comes as TWO bfloat16 planes, hi = bf16(v) and lo = bf16(v - hi), i.e. about 16 mantissa
// bits; each weight tile is multiplied with both planes.  This doubles the MMA work
// (irrelevant while the kernel is HBM-bound) and the L2-resident activation traffic, not the HBM traffic, and
// keeps the hidden states within 1e-2 of a float reference over 32+ layers (plain bfloat16 operands drift to
// 4e-2).  x_lo_rows = 0 selects a single plane.
// The tensor unit cuts its float accumulator off after every addition instead of rounding it, so the error of a result grows with the
// MMAs of its longest slot (both planes count where they share columns, above 128 rows).  Against float64, 12288 x 4096: 64 rows 1.2e-6,
// 128 rows 2.3e-6, 256 rows 2.7e-6, 512 rows 4.9e-6, relative; one rounding of an operand to its two planes is 2.4e-6.
// Every mbarrier wait is bounded: when one runs out the CTA raises ST_TIMEOUT in the status word, stops
// storing, lets its copies settle, frees its tensor memory and returns.
#include "tc.cuh"
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

namespace hydra {

// ---- tensor maps -------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return (EncodeTiledFn)p;
  }();
  return fn;
}

bool tensor_map_encoder_available() { return encode_fn() != nullptr; }

bool get_tensor_map(const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows, bool half, CUtensorMap* out) {
  typedef std::tuple<const void*, uint64_t, uint64_t, uint32_t, bool> Key;
  static std::map<Key, CUtensorMap> cache;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  Key key(ptr, rows, cols, box_rows, half);
  auto it = cache.find(key);
  if (it != cache.end()) { *out = it->second; return true; }
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUtensorMap tm;
  CUresult r = fn(&tm, half ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  if (cache.size() > 4096) cache.clear();
  cache[key] = tm;
  *out = tm;
  return true;
}

namespace {

using namespace tc;

constexpr int BLOCK_N = 128;             // weight rows per tile (MMA M)
constexpr int BLOCK_K = 64;              // 64 bf16 = 128 bytes = one swizzle row
constexpr int A_BYTES = BLOCK_N * BLOCK_K * 2;

// Instruction descriptor: D = f32, A = B = bf16, both K-major, M = 128, N = MT.
__host__ __device__ constexpr uint32_t instr_desc(int mt) { return instr_desc_f16(1, BLOCK_N, mt, 0); }

// Accumulator columns of this thread's lane -> rows (distance n) of the partial buffer; with `cat` the W*lo columns, mt further
// on, are added.  Batches of 32 in a rolled loop: code unrolled for every shape does not
// stay in the instruction cache, and fetching it is what the epilogue then waits for (64 rows: 5.5 us with 64-column batches
// and a 16-column remainder unrolled, 1.5 us rolled).  Reads whole batches, so accumulators are spaced accordingly.
__device__ __forceinline__ void store_accumulator(uint32_t taddr, bool cat, int mt, float* dst, int rows, int n) {
#pragma unroll 1
  for (; rows > 0; rows -= 32, taddr += 32u, dst += (size_t)32 * n) {
    uint32_t r[32];
    if (cat) {
      uint32_t r2[32];
      tmem_ld32x2(taddr, taddr + (uint32_t)mt, r, r2);
#pragma unroll
      for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(r2[j]));
    } else {
      tmem_ld32(taddr, r);
    }
    float* p = dst;
#pragma unroll
    for (int j = 0; j < 32; ++j, p += n)
      if (j < rows) __stcg(p, __uint_as_float(r[j]));
  }
}
// Up to 16 rows (decoding without a tree, draft levels); one row: all tiles and planes in one tensor-memory round trip.
template <int NH>
__device__ __forceinline__ void store_few(uint32_t taddr, int acc_cols, bool cat, int mt, float* dst, int rows, int n, int tiles_in) {
  const uint32_t lo = cat ? (uint32_t)mt : 0u, t1 = taddr + (uint32_t)(NH == 2 ? acc_cols : 0);
  if (rows == 1) {
    uint32_t h0, l0, h1, l1;
    tmem_ld1x4(taddr, taddr + lo, t1, t1 + lo, h0, l0, h1, l1);
    __stcg(dst, cat ? __uint_as_float(h0) + __uint_as_float(l0) : __uint_as_float(h0));
    if (NH == 2 && tiles_in == 2) __stcg(dst + BLOCK_N, cat ? __uint_as_float(h1) + __uint_as_float(l1) : __uint_as_float(h1));
    return;
  }
#pragma unroll 1
  for (int hh = 0; hh < tiles_in; ++hh, taddr += acc_cols, dst += BLOCK_N) {
    uint32_t r[16], q[16];
    tmem_ld16x2(taddr, taddr + lo, r, q);
    if (!cat) {
#pragma unroll
      for (int j = 0; j < 16; ++j) q[j] = 0u;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (j < rows) __stcg(dst + (size_t)j * n, __uint_as_float(r[j]) + __uint_as_float(q[j]));
  }
}

// The slots of one tile (128 columns) added in slot order into the output by the 128 epilogue threads: a warp per row, 16 bytes
// per lane, two rows with all their slots in flight.
__device__ __forceinline__ void sum_tile(const float* part, size_t stride, int slots, float* out, int rows, int n, int e) {
  const int c = (e & 31) * 4;
#pragma unroll 1
  for (int r = e >> 5; r < rows; r += 8) {
    const size_t off[2] = {(size_t)r * n + c, (size_t)(r + 4) * n + c};
    const int ns[2] = {slots, r + 4 < rows ? slots : 0};
    float4 v[2];
    sum_slots_multi<2, 12>(part, stride, off, ns, v);
    *reinterpret_cast<float4*>(out + off[0]) = v[0];
    if (ns[1]) *reinterpret_cast<float4*>(out + off[1]) = v[1];
  }
}

struct GemmArgs {
  float* part; size_t slot_stride;
  float* out; GemmArrivals arr;            // REDUCE only: the output, and per tile how many of its CTAs have stored
  int m, n, kb, group, m_blocks, total_units, q;      // group: CTAs (row tiles) that walk a range together; m_blocks: groups of row tiles
  int x_lo_rows;                 // row offset of the lo plane inside the activation tensor map (0: single plane)
  // activation rows per tile, boxes (planes) of a stage, MMA passes over a weight tile and columns of one, ring stages,
  // accumulator columns and buffers, tensor-memory columns
  int mt, x_boxes, passes, mma_n, stages, acc_cols, acc_bufs, tmem_cols;
  int cat;                       // hi and lo planes are the halves of one MMA operand: columns [mt, 2 mt) hold W*lo
  int* status;
  int* diag;                     // optional int[8]: where the first bounded wait gave up (site, cta, unit, units, grid, m, n, kb)
  uint32_t wait_limit;           // polls before a barrier wait gives up
  int w_const;                   // no kernel in flight writes w
  int skip_unit;                 // >= 0: CTA 0 leaves out the weight-tile request of this unit (a test of the bounded waits), else -1
};

// Records the first wait that ran out (site: 1 producer/empty, 2 mma/acc-empty, 3 mma/full, 5 epilogue/acc-full).
#define GIVE_UP(site, unit) do { atomicOr(a.status, ST_TIMEOUT); \
    if (a.diag && atomicCAS(a.diag, 0, (site)) == 0) { a.diag[1] = blockIdx.x; a.diag[2] = (unit); a.diag[3] = n_units; \
      a.diag[4] = gridDim.x; a.diag[5] = a.m; a.diag[6] = a.n; a.diag[7] = a.kb; } } while (0)

__device__ __forceinline__ void epilogue_barrier() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
__device__ __forceinline__ bool epilogue_all(bool v) {       // v of all 128 epilogue threads
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}

constexpr int MAX_STAGES = 10;
constexpr int EPI_WARPS = 4;                             // one per quadrant of tensor memory (two measured no faster: the L2 takes the stores no sooner)
constexpr int THREADS = 64 + 32 * EPI_WARPS;
// Shared memory of the ring: 200 KB, above 64 rows up to 220 KB where that is another stage.  There a stage is 36 to 96 KB and two or three of them do
// not hide a load: 22016 x 4096, two planes, 144 rows 44.5 us with three stages / 40.1 with four, 288 rows 88 / 76, 320 rows 92 / 84 (two / three); 4096 x
// 4096, 400 and 432 rows 31.3 / 25.8, 33.3 / 27.6 (two / three).  Up to 64 rows the kernels around a GEMM want the rest: with 216 KB 1 and 16 rows took
// 27.7 and 28.2 instead of 26.8 and 27.2, and with 160 KB as long.
constexpr int RING_BYTES = 200 * 1024, RING_BYTES_MAX = 220 * 1024, RING_EXTRA_BYTES = 1024 /*alignment slack*/ + 512 /*barriers*/;

// Shapes are run-time arguments (one copy of the code for all row counts); NH: 128-row weight tiles per CTA and unit.
// REDUCE (stand-alone calls): the last CTA to store a tile's partial sums adds them, so the call is one launch.  (Inside a
// forward call the consumer kernels add them: there the extra round trip through the counters is on the critical path.)
template <int NH, bool REDUCE>
__global__ void __launch_bounds__(THREADS, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const GemmArgs a) {
  static_assert(!REDUCE || NH == 1, "sum_tile takes one weight tile");
  constexpr int W_BYTES = NH * A_BYTES, BN = NH * BLOCK_N;        // weight rows of a unit
  extern __shared__ uint8_t smem_raw[];
  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int stages = a.stages;
  const uint32_t x_box_bytes = (uint32_t)a.mt * (BLOCK_K * 2), x_bytes = a.x_boxes * x_box_bytes, stage_bytes = W_BYTES + x_bytes;
  const uint32_t bars = tiles + stages * stage_bytes;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (MAX_STAGES + s); };
  auto accfull_bar = [&](int i) { return bars + 8u * (2 * MAX_STAGES + i); };
  auto accempty_bar = [&](int i) { return bars + 8u * (2 * MAX_STAGES + 2 + i); };
  const uint32_t tmem_slot = bars + 8u * (2 * MAX_STAGES + 4);
  __shared__ int s_abort, s_last;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // this CTA's range of the line, and which of its group's row tiles is its own
  const int range = blockIdx.x / a.group, member = blockIdx.x - range * a.group, u_begin = range * a.q;
  const int u_end = min(u_begin + a.q, a.total_units);
  const int n_units = u_end - u_begin, ring = n_units < stages ? n_units : stages, pre = a.w_const ? (ring + 1) / 2 : 0;     // pre: weight tiles requested up front

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < stages; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(accfull_bar(i), 1); mbar_init(accempty_bar(i), EPI_WARPS); }
    mbar_init_fence();
    prefetch_tensormap(&tmW);
    prefetch_tensormap(&tmX);
    // weights do not depend on the preceding kernel: request half a ring of weight tiles right away, before the
    // CTA-wide set-up (TMEM allocation, barrier hand-over) and before griddepcontrol.wait; where they may, bring them nearer.
    // (The weight tiles of a whole ring are 128 KB an SM at 64 rows and 160 KB at one, 19 and 24 MB over the SMs; the preceding row-wise kernel's
    // loads queue behind them.  7B shape, 32 steps with a 64-row tree 145.2 -> 144.0 ms with half a ring, runs of one side 0.3 % apart; without a
    // tree, and 47 supplied rows, the same either way.  All stages but one gained as much as half, one stage alone nothing.)
    const uint64_t pol = a.m_blocks == 1 ? policy_evict_first() : policy_evict_normal();
    int tile = u_begin / a.kb, kb = u_begin - tile * a.kb, nrow = tile / a.m_blocks * BN;
    for (int i = 0; i < (a.w_const ? pre : ring); ++i) {
      if (!a.w_const) {
        tma_prefetch_2d(&tmW, kb * BLOCK_K, nrow);
      } else if (u_begin + i != a.skip_unit) {
        mbar_arrive_expect_tx(full_bar(i), W_BYTES);
        tma_load_2d(tiles + i * stage_bytes, &tmW, kb * BLOCK_K, nrow, full_bar(i), pol);
      }
      if (++kb == a.kb) { kb = 0; nrow = ++tile / a.m_blocks * BN; }
    }
  }
  if (warp == 1) tmem_alloc(tmem_slot, a.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_launch();                       // all CTAs of this grid are resident: let the next kernel get ready
  uint32_t tmem_base;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));

  if (warp == 0) {
    if (lane == 0) {
      // (several groups of row tiles: the next one reads the weights again)
      const uint64_t pol_w = a.m_blocks == 1 ? policy_evict_first() : policy_evict_normal(), pol_x = policy_evict_last();
      int kcol = 0, nrow = 0, mrow = 0;                  // (k column, weight row, activation row) of the unit being issued, advanced without divisions
      if (n_units > 0) {
        const int tile = u_begin / a.kb;
        kcol = (u_begin - tile * a.kb) * BLOCK_K; nrow = tile / a.m_blocks * BN; mrow = (tile % a.m_blocks * a.group + member) * a.mt;
      }
      const int kend = a.kb * BLOCK_K, mstep = a.group * a.mt, mend = a.m_blocks * mstep;
      int s = 0; uint32_t eph = 1;                       // ring stage, parity of its empty barrier
      grid_dep_wait();                                   // activations are the preceding kernel's output
      for (int i = 0; i < n_units; ++i) {
        const uint32_t dst = tiles + s * stage_bytes;
        if (i >= pre) {
          if (!mbar_wait(empty_bar(s), eph, a.wait_limit)) { GIVE_UP(1, i); s_abort = 1; break; }      // (passes at once the first time round)
          if (u_begin + i != a.skip_unit) {
            mbar_arrive_expect_tx(full_bar(s), W_BYTES);
            tma_load_2d(dst, &tmW, kcol, nrow, full_bar(s), pol_w);
          }
        }
        mbar_arrive_expect_tx(full_bar(s), x_bytes);
        tma_load_2d(dst + W_BYTES, &tmX, kcol, mrow, full_bar(s), pol_x);
        if (a.x_boxes == 2) tma_load_2d(dst + W_BYTES + x_box_bytes, &tmX, kcol, mrow + a.x_lo_rows, full_bar(s), pol_x);
        if (++s == stages) { s = 0; eph ^= 1u; }
        if ((kcol += BLOCK_K) == kend) { kcol = 0; if ((mrow += mstep) >= mend) { mrow -= mend; nrow += BN; } }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = instr_desc_f16(1, BLOCK_N, a.mma_n, 0);
      const uint64_t ring_desc = smem_desc_sw128(tiles);                       // + offset / 16 inside the ring
      int s = 0, acc = 0;
      uint32_t ph = 0, acc_ph = 0;                       // parities of the stage's full barrier and of the accumulator's barriers
      bool ok = true;
      int seg_len = n_units > 0 ? min((u_begin / a.kb + 1) * a.kb, u_end) - u_begin : 0;      // first segment: the tail of a tile
      for (int i = 0; i < n_units && ok;) {
        if (!mbar_wait(accempty_bar(acc), acc_ph ^ 1u, a.wait_limit)) { GIVE_UP(2, i); ok = false; break; }      // epilogue has drained this buffer
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)(acc * NH * a.acc_cols);
        for (int j = 0; j < seg_len; ++j, ++i) {
          if (!mbar_wait(full_bar(s), ph, a.wait_limit)) { GIVE_UP(3, i); ok = false; break; }
          tc_fence_after();
          const uint64_t wdesc = ring_desc + (uint64_t)((s * stage_bytes) >> 4), xdesc = wdesc + (uint64_t)(W_BYTES >> 4);
#pragma unroll
          for (int hh = 0; hh < NH; ++hh)                // the unit's weight tiles, one accumulator each, same activation tile
#pragma unroll
            for (int k = 0; k < BLOCK_K / 16; ++k)       // 16 bf16 = 32 bytes per MMA: +2 in 16-byte units
              umma_f16(tmem_d + (uint32_t)(hh * a.acc_cols), wdesc + (uint64_t)(hh * (A_BYTES >> 4) + 2 * k), xdesc + 2u * k, idesc, (uint32_t)((j | k) != 0));
          if (a.passes == 2) {                           // the low-order plane of the activations, same weights
            const uint64_t ldesc = xdesc + (uint64_t)(x_box_bytes >> 4);
#pragma unroll
            for (int hh = 0; hh < NH; ++hh)
#pragma unroll
              for (int k = 0; k < BLOCK_K / 16; ++k)
                umma_f16(tmem_d + (uint32_t)(hh * a.acc_cols), wdesc + (uint64_t)(hh * (A_BYTES >> 4) + 2 * k), ldesc + 2u * k, idesc, 1u);
          }
          umma_commit(empty_bar(s));                       // frees the stage once these MMAs have read it
          if (++s == stages) { s = 0; ph ^= 1u; }
        }
        if (!ok) break;
        umma_commit(accfull_bar(acc));                   // segment complete: hand the accumulators to the epilogue
        if (++acc == a.acc_bufs) { acc = 0; acc_ph ^= 1u; }
        seg_len = min(a.kb, n_units - i);                // every later segment starts a tile
      }
      if (!ok) { atomicOr(a.status, ST_TIMEOUT); s_abort = 1; }
    }
  } else {
    const int quarter = warp & 3;                        // TMEM lanes this warp may read
    grid_dep_wait();                                     // the partial buffer may still be read by the preceding kernel
    int acc = 0;
    uint32_t acc_ph = 0;
    for (int i = 0, tile = u_begin / a.kb; i < n_units; ++tile) {
      // where the segment goes, worked out while its accumulator fills
      const int seg_len = min((tile + 1) * a.kb, u_end) - (u_begin + i), slot = range - tile * a.kb / a.q;
      const int n_tile = tile / a.m_blocks, n0 = n_tile * BN, m0 = ((tile - n_tile * a.m_blocks) * a.group + member) * a.mt, rows = min(a.mt, a.m - m0);
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * NH * a.acc_cols);
      float* dst = a.part + (size_t)slot * a.slot_stride + (size_t)m0 * a.n + n0 + quarter * 32 + lane;
      if (REDUCE && threadIdx.x == 64) atomicMax(a.arr.count + tile, a.arr.ticket << 16);      // an older call's count, if one is left, is gone
      const int tiles_in = NH == 2 && n0 + BLOCK_N < a.n ? 2 : 1;      // an output that is no multiple of the unit's width ends inside its last unit
      bool ok = mbar_wait(accfull_bar(acc), acc_ph, a.wait_limit);
      if constexpr (REDUCE) ok = epilogue_all(ok);       // the four warps meet at barriers below: they give up together
      if (!__all_sync(0xffffffffu, ok)) { if (lane == 0) GIVE_UP(5, i); s_abort = 1; break; }
      tc_fence_after();
      if (rows <= 16) {
        store_few<NH>(taddr, a.acc_cols, a.cat, a.mt, dst, rows, a.n, tiles_in);
      } else {
#pragma unroll 1
        for (int hh = 0; hh < tiles_in; ++hh) store_accumulator(taddr + (uint32_t)(hh * a.acc_cols), a.cat, a.mt, dst + hh * BLOCK_N, rows, a.n);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(accempty_bar(acc));     // the MMA lane may reuse this accumulator
      if constexpr (REDUCE) {
        const int slots = ((tile + 1) * a.kb - 1) / a.q - tile * a.kb / a.q + 1;
        epilogue_barrier();
        if (threadIdx.x == 64) {                         // one fence covers what the barrier has ordered before it
          __threadfence();
          s_last = (atomicAdd(a.arr.count + tile, 1ull) & 0xffff) == (unsigned)(slots - 1);
          __threadfence();
        }
        epilogue_barrier();
        if (s_last) {
          if (threadIdx.x == 64) a.arr.count[tile] = 0ull;      // threads may enqueue on one stream in another order than their tickets'
          const size_t at = (size_t)m0 * a.n + n0;
          sum_tile(a.part + at, a.slot_stride, slots, a.out + at, rows, a.n, (int)threadIdx.x - 64);
        }
      }
      i += seg_len;
      if (++acc == a.acc_bufs) { acc = 0; acc_ph ^= 1u; }
    }
  }
  __syncwarp();                                          // the one-lane roles rejoin their warps before the block-wide barrier
  tc_fence_before();
  __syncthreads();
  if (s_abort) {                                         // let copies in flight land before the CTA retires
    for (int i = 0; i < 2000; ++i) __nanosleep(100);
  }
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, a.tmem_cols); }
}

template <int NH, bool REDUCE>
hydra_status launch(const CUtensorMap& tw, const CUtensorMap& tx, const GemmArgs& a, int grid, int smem, cudaStream_t st) {
  static PerDeviceFlag attr_done;
  if (!attr_done.get()) {
    HYDRA_CUDA(cudaFuncSetAttribute(gemm_tc_kernel<NH, REDUCE>, cudaFuncAttributeMaxDynamicSharedMemorySize, RING_BYTES_MAX + RING_EXTRA_BYTES));
    attr_done.set();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  HYDRA_CUDA(cudaLaunchKernelEx(&cfg, gemm_tc_kernel<NH, REDUCE>, tw, tx, a));
  HYDRA_LAUNCH_CHECK();
  return HYDRA_OK;
}

}  // namespace

bool gemm_tc_available() { return tensor_map_encoder_available(); }

// Tile shape: 128 or 256 weight rows per unit.
//  * Units of 256 rows take enough of them for ~4 per SM.
//  * Up to 64 activation rows 256: fewer activation bytes per weight byte, more weight bytes in flight.
//  * Above, 128: tensor memory then holds two accumulators, and fewer partial sums are left.  Except for
//  * 97 to 160 rows of an output wide enough that a tile meets one or two ranges all the same (half as many tiles as SMs): the activation tile is twice the
//    weight tile there, and an SM takes in a third less (176 rows would have two stages); and for
//  * tall row tiles with 16 and more units per SM, where the activation tile is most of what an SM takes in.
// Measured, us with 128 / 256 weight rows.  With the reduction of the partial sums:
//    rows  n x k                                      rows  n x k
//       1  2048 x 2048     4.8 / 5.6                     1  3072 x 3072    8.4 / 7.6
//       1  22016 x 4096   32.1 / 30.2                   64  22016 x 4096  42.2 / 42.4
//       1  4096 x 11008   19.0 / 17.5                   64  4096 x 11008  20.9 / 20.3
//      96  12288 x 4096   29.4 / 30.9                  128  4096 x 4096   16.0 / 19.0
//     192  22016 x 4096     77 / 82                    256  22016 x 4096   111 / 103
//     512  22016 x 4096    222 / 192                   512  4096 x 11008    96 / 91
//     512  4096 x 4096      49 / 54
// In a forward pass:
//    rows  22016 x 4096  32000 x 4096  27648 x 5120  35840 x 6656  19968 x 6656  12288 x 4096
//      80  32.0 / 32.7
//     128  37.9 / 36.6   54.0 / 51.1   58.2 / 54.5   97.8 / 90.5   56.8 / 54.1   23.0 / 23.7
//     129  39.4 / 38.8   56.3 / 52.9   63.0 / 58.8    103 / 95     60.8 / 57.9
//     144                                                                        25.0 / 25.6
//     160  47.3 / 41.8   66.8 / 56.5   74.8 / 63.0    127 / 105    73.3 / 64.5
//     192  54.2 / 56.2
//    6656 x 17920 with its norm, 128 rows: 59.4 / 61.2
struct GemmShape { int nh, mt, m_tiles; };
static GemmShape gemm_shape(int m, int n, int k) {
  // equal row tiles of a multiple of 16 rows, so that the MMA work and the activation traffic follow m
  const int row_tiles = (m + 255) / 256, mt = ((m + row_tiles - 1) / row_tiles + 15) / 16 * 16;
  const long long units = (long long)row_tiles * (n / 256) * (k / BLOCK_K), sms = sm_count();
  const bool wide = m <= 64 ? 4 * units >= 15 * sms : m <= 160 ? m > 96 && n / 256 * 2 >= sms : (mt > 192 || row_tiles > 1) && units >= 16 * sms;
  return GemmShape{wide ? 2 : 1, mt, (m + mt - 1) / mt};
}

// Sum of the cubes of the lengths of a line's segments (a segment is one sum in the tensor unit).  The unit's accumulator truncates, so the error of a sum grows
// with its length to the power 1.5 and a product's error is as the square root of this: ratios of two plans' errors agree with the measured ones to 1 %.
static double segment_cubes(long long line, int kb, int q) {
  double s = 0;
  for (long long u = 0, tile = kb, range = q; u < line;) {
    const long long end = std::min(tile, range);
    const double l = (double)(end - u);
    s += l * l * l;
    if (end == tile) tile += kb;
    if (end == range) range += q;
    u = end;
  }
  return s;
}
// Units a range when a line is shared out over at most `most` ranges of at least 4 units
static int range_units(long long line, long long most) {
  const long long r = std::max(1ll, std::min(most, line / 4));
  return (int)((line + r - 1) / r);
}
// Row tiles that walk the line together: all of them up to 16, else groups as equal as they come, unless fewer at a time are as exact as one line of all
// tiles and more are not.  Ranges that end with the tiles leave whole tiles in one sum, and a group whose size does not divide the SMs makes ranges longer: a group is taken when its
// plan's error is at most 5 % above that of the one line and its ranges at most a sixteenth longer, or an eighth if no group has such.  4096 x 4096, 9 row tiles: one line 6.58e-6, nine
// together (whole tiles) 9.25e-6 against float64, three 6.04e-6; 17 row tiles of 2048 x 2048: 3.12e-6, two nines 4.56e-6.
constexpr int GROUP_MAX = 16;            // (a prompt pass has at most 3 row tiles, 64 sequences of a 64-row tree 16)
static int row_tile_group(int m, int m_tiles, int n_tiles, int kb, int sms) {
  const long long all = (long long)n_tiles * m_tiles * kb;
  if (m_tiles == 1 || all / 4 < sms) return 1;
  const int most = (m_tiles + GROUP_MAX - 1) / GROUP_MAX;
  const int group = (m_tiles + most - 1) / most;
  if (m > 65536) return group;           // (SplitDesc::div_mt: groups of 16 whole tiles)
  const int q1 = range_units(all, sms);
  const double cubes1 = segment_cubes(all, kb, q1) / (double)all;
  for (const int part : {16, 8})
    for (int g = group; g > 1; --g) {
      const int blocks = (m_tiles + g - 1) / g;
      g = (m_tiles + blocks - 1) / blocks;
      const long long line = (long long)n_tiles * blocks * kb;
      const int q = range_units(line, sms / g);
      if ((long long)part * q <= (part + 1ll) * q1 && segment_cubes(line, kb, q) <= 1.1 * cubes1 * (double)line) return g;
    }
  return 1;
}

// Stream-K plan: equal contiguous ranges of the line, at most one CTA per SM and at least 4 k-blocks each.
struct GemmPlan { GemmShape sh; int group, ranges, max_slots; SplitDesc sd; };
static GemmPlan gemm_plan(int m, int n, int k, bool want_slots, size_t part_cap) {
  GemmPlan p{};
  p.sh = gemm_shape(m, n, k);
  SplitDesc& sd = p.sd;
  const int kb = k / BLOCK_K, sms = sm_count(), n_tiles = p.sh.nh == 2 ? (n + 255) / 256 : n / BLOCK_N;
  p.group = row_tile_group(m, p.sh.m_tiles, n_tiles, kb, sms);
  const int blocks = (p.sh.m_tiles + p.group - 1) / p.group;
  sd.kb = kb; sd.stride = (size_t)m * n; sd.bn_shift = p.sh.nh == 2 ? 8 : 7; sd.m_tiles = blocks; sd.mt = p.group * p.sh.mt;
  const int tiles = n_tiles * blocks;
  const long long line = (long long)tiles * kb;
  sd.q = range_units(line, sms / p.group);
  if (want_slots || part_cap) {
    auto slots = [&]() {                                   // ranges that touch a tile, at most: tile t begins rem units into a range
      const unsigned q = (unsigned)sd.q, kbu = (unsigned)sd.kb, top = (q + kbu - 2) / q + 1;
      unsigned mx = 1, rem = 0;
      for (int t = 0; t < tiles && mx < top; ++t, rem = (rem + kbu) % q) mx = std::max(mx, (rem + kbu - 1) / q + 1);
      return (int)mx;
    };
    p.max_slots = slots();
    // whole tiles per range need one slot
    while (part_cap && p.max_slots > 1 && (size_t)p.max_slots * sd.stride > part_cap) {
      sd.q = sd.q < kb ? sd.q + 1 : (sd.q + kb) / kb * kb;
      p.max_slots = slots();
    }
  }
  p.ranges = (int)((line + sd.q - 1) / sd.q);
  sd.set_inverses();
  return p;
}
SplitDesc gemm_tc_plan(int m, int n, int k, int* grid, int* max_slots, size_t part_cap) {
  const GemmPlan p = gemm_plan(m, n, k, max_slots != nullptr, part_cap);
  if (grid) *grid = p.ranges * p.group;
  if (max_slots) *max_slots = p.max_slots;
  return p.sd;
}

hydra_status gemm_tc(const bf16* x, int x_rows_alloc, int x_planes, const bf16* w, float* part, int m, int n, int k,
                     SplitDesc* sd_out, bool w_const, int* status, int* diag, const GemmDebug* dbg, cudaStream_t st, size_t part_cap, float* out,
                     const GemmArrivals* arrivals, int x_row0) {
  if (m <= 0 || n <= 0 || k <= 0 || n % BLOCK_N || k % BLOCK_K || (x_planes != 1 && x_planes != 2)) return HYDRA_ERR_UNSUPPORTED;
  if (((uintptr_t)x | (uintptr_t)w) & 15) return HYDRA_ERR_INVALID;
  const GemmPlan plan = gemm_plan(m, n, k, false, part_cap);
  const SplitDesc& sd = plan.sd;
  const GemmShape& sh = plan.sh;
  const int grid = plan.ranges * plan.group;
  if (x_rows_alloc < x_row0 + m) x_rows_alloc = x_row0 + m;
  x += (size_t)x_row0 * k;
  GemmArgs a{};
  a.part = part; a.slot_stride = sd.stride; a.m = m; a.n = n; a.kb = sd.kb; a.mt = sh.mt;
  a.group = plan.group; a.m_blocks = sd.m_tiles; a.total_units = ((n + (1 << sd.bn_shift) - 1) >> sd.bn_shift) * sd.m_tiles * sd.kb; a.q = sd.q; a.status = status;
  a.x_lo_rows = x_planes == 2 ? x_rows_alloc : 0; a.diag = diag;
  a.wait_limit = dbg && dbg->wait_limit ? dbg->wait_limit : WAIT_LIMIT; a.skip_unit = dbg ? dbg->skip_unit : -1; a.w_const = w_const;
  // Two planes, up to 128 rows: the hi and lo activation tiles sit back to back and form ONE MMA operand of 2 mt rows, so each
  // weight tile is read from shared memory once; taller tiles take a pass per plane.
  a.cat = x_planes == 2 && sh.mt <= 128;
  a.passes = x_planes == 2 && !a.cat ? 2 : 1;
  a.x_boxes = x_planes; a.mma_n = a.cat ? 2 * sh.mt : sh.mt;
  const int read_cols = (sh.mt + 31) / 32 * 32;          // the epilogue reads whole batches of 32 columns
  a.acc_cols = a.cat ? sh.mt + read_cols : read_cols;
  a.acc_bufs = 2 * sh.nh * a.acc_cols <= 512 ? 2 : 1;
  for (a.tmem_cols = 32; a.tmem_cols < a.acc_bufs * sh.nh * a.acc_cols;) a.tmem_cols *= 2;
  const int stage_bytes = sh.nh * A_BYTES + a.x_boxes * sh.mt * BLOCK_K * 2;
  a.stages = std::min((sh.mt > 64 ? RING_BYTES_MAX : RING_BYTES) / stage_bytes, MAX_STAGES);
  const int smem = std::max(a.stages * stage_bytes, RING_BYTES) + RING_EXTRA_BYTES;
  CUtensorMap tw, tx;
  if (!get_tensor_map(w, (uint64_t)n, (uint64_t)k, (uint32_t)(sh.nh * BLOCK_N), false, &tw) ||
      !get_tensor_map(x, (uint64_t)x_rows_alloc * x_planes - x_row0, (uint64_t)k, (uint32_t)sh.mt, false, &tx)) {      // what the buffer holds from x on; rows past it read as zeros
    set_last_error("cuTensorMapEncodeTiled", cudaErrorUnknown);
    return HYDRA_ERR_CUDA;
  }
  if (sd_out) *sd_out = sd;
  // One launch where issuing a second one is what takes the time: up to 16 rows and a weight matrix that passes in a few microseconds
  // (back to back, one launch / two: 11 x 2048 x 2048 7.1 / 9.2 us, 4 x 3456 x 640 6.8 / 9.2, 11 x 4096 x 1024 7.0 / 9.3, 8 x 640 x 5632
  // 8.6 / 9.1; with weight tiles requested before the dependency wait 11 x 4096 x 2048 took 9.2 / 8.4, 11 x 4096 x 4096 12.4 / 10.2, 64 x 512 x
  // 1024 10.2 / 8.3: the sums of a tile are one CTA's work).
  // sum_tile stores 16 bytes at a time; a result buffer off that boundary takes the second launch, which stores single floats.  (Units
  // of two weight tiles begin at 9 million weights on 148 SMs.)
  // And only while a tile has few slots, which one CTA adds eight rows at a time: a call from Python takes 9.2 us with two launches whatever these sizes, and with one 11 x 256 x
  // 4096 (17 slots at most) 8.5, 11 x 1024 x 5632 (19) 10.7, 8 x 640 x 5632 (23) 8.5, 8 x 768 x 7744 (25) 10.0, 11 x 256 x 11008 (44) 18.7.
  const int most_slots = (sd.kb + sd.q - 2) / sd.q + 1;
  if (out && arrivals && sh.nh == 1 && m <= 16 && (long long)n * k <= GEMM_ONE_LAUNCH_WEIGHTS && most_slots <= (m > 8 ? 17 : 23) && !((uintptr_t)out & 15)) {
    a.out = out; a.arr = *arrivals;
    return launch<1, true>(tw, tx, a, grid, smem, st);
  }
  const hydra_status s = sh.nh == 2 ? launch<2, false>(tw, tx, a, grid, smem, st) : launch<1, false>(tw, tx, a, grid, smem, st);
  return s == HYDRA_OK && out ? reduce_splits(part, sd, out, m, n, st) : s;
}

}  // namespace hydra
