// tcgen05 GEMM for many activation rows (long prompts, decode steps above 128 rows): two SMs work as a pair on one tile.
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include "../../include/corun.h"
#include "gemm.cuh"
#include "launch.cuh"
#include "ptx.cuh"

namespace corun {

namespace {

constexpr int PG_THREADS = 320;                     // warp 0 TMA producer, warp 1 MMA issuer, warps 2-9 epilogue
constexpr int PG_EPI = 8;                           // epilogue warps: two per TMEM lane quarter, half of the columns each
constexpr int PG_STAGES = 4;
constexpr int PG_CHAIN = 16;                        // k-blocks that are summed in one accumulator (see below)
enum : int { PG_PLAIN = 0, PG_SWIGLU = 1, PG_KV = 2 };
constexpr uint32_t PG_X_BYTES = 128 * GEMM_BLOCK_K * 2;      // 16 KiB: a CTA's 128 activation rows, hi or lo
constexpr uint32_t PG_W_BYTES = 128 * GEMM_BLOCK_K * 2;      // 16 KiB: a CTA's half of the 256 weight rows
constexpr uint32_t PG_STAGE_BYTES = 2 * PG_X_BYTES + PG_W_BYTES;
constexpr uint32_t PG_OUT_BYTES = 32 * 128;                  // an epilogue warp's staging tile: 32 rows x 32 fp32 (or hi and lo of 32 bf16)
constexpr size_t PG_SMEM = 1024 + (size_t)PG_STAGES * PG_STAGE_BYTES + PG_EPI * PG_OUT_BYTES;

// out[r, n] = sum_k W[n, k] * (Xhi[r, k] + Xlo[r, k]) for tiles of 256 rows x 256 weight rows.
//
// A cluster of two CTAs (the two SMs of a TPC) owns a tile: CTA i holds activation rows 128 i .. of it (hi and lo, the
// M side) and weight rows 128 i .. (the N side), and one thread of the first CTA issues tcgen05.mma.cta_group::2
// (M = 256, N = 256) over both; each CTA's tensor memory receives its own 128 rows x all 256 weight rows.  Per k-block
// a CTA loads 48 KiB for 8 MMAs of 128 cycles: 48 bytes per cycle, where one CTA on its own (128 rows x 256 weight
// rows) would need 64 and be bound by what the L2 delivers into an SM.  hi and lo go into the same accumulator,
// k-slice by k-slice.  Two accumulators of 256 columns alternate, so that a tile's epilogue overlaps the next tile.
//
// K is cut into `slices` (a function of N, K and the number of SMs): a slice is summed in one accumulator, the slices in
// ascending order in fp32.  A pair that has a whole tile does both itself (the running sum in the epilogue's registers);
// the tiles that do not fill a wave of the pairs are dealt out in units of `per_unit` slices, every slice leaving a partial
// matrix, and the consumer adds them in the same order (gemm_load_pair4).  So a row's result depends on its own activations
// only, not on its place among the rows nor on their number: 256 rows of the Qwen3-8B QKV projection are 24 tiles, 72 units
// of a third of K each for 74 pairs (43 us as 24 whole tiles).
//
// A slice is short because the tensor core's accumulator cuts every sum off: a product is off by 1.7e-8 (2-norm, relative) per
// MMA of a slice, K = 4096 in one accumulator (512 MMAs, hi and lo) by 9e-6, slices of 16 k-blocks by 2.2e-6 beside the 2.5e-6
// of the activations' 16 bits.  Prompts of 300 / 1003 tokens, 12 Qwen3-8B layers, against 64 bits: 1.1e-4 / 6.7e-5 with the
// gate / up matrix in one slice and 3 or 4 of the others, 9.6e-5 / 5.3e-5 so (8 k-blocks: no nearer, and 3 % slower).
//
// Launched in plain stream order (no programmatic launch): a pair's two SMs are taken and left together, never while a
// CTA of a neighbouring kernel of the stream is on one of them.
//
// The tiles are walked row tile first (pair p takes tiles p, p + pairs, ...), so that the pairs that run at the same
// time share weight tiles in L2 and the weights are read from HBM once.
//
// SWIGLU: W is a gate / up matrix ([2F, K]); a tile is `half` gate rows (first CTA) and the up rows of the same outputs
// (second CTA), always whole (the slices meet in registers), and the epilogue writes silu(gate) * up as the bf16 hi/lo pair the down GEMM reads.
// KV (gemm_pair_plan_create_kv): a tile's 256 columns are one head's 128 key and 128 value columns, stored as fp16 hi / lo
// pairs, keys by the first half of the epilogue warps, values by the second; cap: rows of one of the four matrices per head;
// kv_scale: [head][2] powers of two that keep a head's keys and values within the range of such a pair.
//
// DECODE (up to 256 rows, one row tile; row_blocks says which halves of them hold requests this step): hi and lo have an
// accumulator each, a slice's value is their sum.  With requests in rows 128 .. each CTA keeps both accumulators (512 columns:
// one buffer).  Without, a CTA's 128 operand rows are the hi and the lo parts of 64 rows, so that one MMA does what takes two
// above, and the halves of the accumulator meet through shared memory (the stages' unused lo parts): the tensor work is that
// of 128 rows, and a row has the same value either way.  (With both halves multiplied in every step, 200 slots with 30 / 60 /
// 128 requests took 2.83 / 3.06 / 3.54 ms per step of 12 Qwen3-8B layers, now 2.65 / 2.78 / 3.26; with 200 requests 4.27, now
// 4.40: the end of a slice is not hidden behind the next one.  Others: Program::wide.)
template <int MODE, bool DECODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PG_THREADS, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmHi,
                 const __grid_constant__ CUtensorMap tmLo, const __grid_constant__ CUtensorMap tmOut,
                 const __grid_constant__ CUtensorMap tmOut2, int R, int N, int KB, int row_tiles, int whole, int units, int slices,
                 int per_unit, int half, int *status, const int *row_blocks, int cap, const float *kv_scale, unsigned long long *trace) {
  // optional per-CTA timeline (debug): 8 globaltimer stamps, as the other GEMM's
#define TRACE(i) do { if (trace) trace[(size_t)blockIdx.x * 8 + (i)] = globaltimer_ns(); } while (0)
  if (threadIdx.x == 0) TRACE(0);
  constexpr bool SWIGLU = MODE == PG_SWIGLU, KV = MODE == PG_KV;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[PG_STAGES];      // used in the first CTA: both CTAs' loads of a stage
  __shared__ __align__(8) uint64_t empty_bar[PG_STAGES];     // in each CTA: the MMAs have read the stage
  __shared__ __align__(8) uint64_t tmem_full_bar[2];         // in each CTA: an accumulator is complete
  __shared__ __align__(8) uint64_t tmem_empty_bar[2];        // in the first CTA: both CTAs' epilogues have read it
  __shared__ __align__(8) uint64_t x_full_bar[4], x_free_bar[4];   // (stacked) lo sums of 32 rows x 128 columns handed over / read
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;

  // (DECODE) the step's requests are in the first rows; stacked: none in rows 128 ..
  const bool stacked = DECODE && !(*reinterpret_cast<const volatile int *>(row_blocks) & 2);
  const bool one_buffer = DECODE && !stacked;
  if (stacked && R > 128) R = 128;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < PG_STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tmem_full_bar[a]), 1);
      mbar_init(smem_u32(&tmem_empty_bar[a]), 2 * 32 * PG_EPI);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(smem_u32(&x_full_bar[i]), 32);
      mbar_init(smem_u32(&x_free_bar[i]), 32);
    }
    fence_mbar_init();
    fence_proxy_async();
    prefetch_tensormap(&tmW);
    prefetch_tensormap(&tmHi);
    prefetch_tensormap(&tmLo);
    prefetch_tensormap(&tmOut);
    prefetch_tensormap(&tmOut2);
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(&tmem_base_s), 512);   // (the permit is given back at the end: see there)
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // the other CTA's barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  if (threadIdx.x == 0) TRACE(1);
  volatile int *abort_p = &abort_flag;
  int fail = 0;

  // Work unit u: a whole tile (all slices in turn), or per_unit slices of a tile beyond the `whole` first ones.
  struct Unit { int tile, s0, s1; };
  auto unit = [&](int u) {
    if (u < whole) return Unit{u, 0, slices};
    const int v = u - whole, n = slices / per_unit, t = v / n, sl = (v - t * n) * per_unit;
    return Unit{whole + t, sl, sl + per_unit};
  };
  auto cut = [&](int sl) { return sl * KB / slices; };       // first k-block of a slice

  if (warp == 0) {
    if (elect_one()) {
      // ---------------- TMA producer (both CTAs; the bytes count on the first CTA's barrier) ----------------
      const uint64_t pol_w = l2_policy_evict_first();        // a weight tile is used by the row tiles that run now
      const uint64_t pol_x = l2_policy_evict_last();
      const uint32_t stage_tx = 2u * (uint32_t)half * 128u + (stacked ? 2u : 4u) * PG_X_BYTES;   // of both CTAs
      int it = 0;
      for (int u = pair; u < units && !fail; u += n_pairs) {
        const Unit un = unit(u);
        const int nt = un.tile / row_tiles, yx = (un.tile % row_tiles) * 256 + rank * 128;
        const int yw = SWIGLU ? nt * half + rank * (N >> 1) : nt * GEMM_TILE_N + rank * 128;
        const int kb1 = cut(un.s1);
        for (int kb = cut(un.s0); kb < kb1; ++kb, ++it) {
          const int s = it % PG_STAGES;
          if (!mbar_wait(smem_u32(&empty_bar[s]), ((uint32_t)(it / PG_STAGES) & 1u) ^ 1u, abort_p)) {
            fail = DEV_TIMEOUT_PRODUCER;
            break;
          }
          const uint32_t fb = smem_u32(&full_bar[s]), dst = base + (uint32_t)s * PG_STAGE_BYTES;
          if (rank == 0) mbar_arrive_expect_tx(fb, stage_tx);
          if (it == 0) TRACE(2);
          const uint32_t fb0 = cluster_map(fb, 0);
          tma_load_2d_pair(dst + 2 * PG_X_BYTES, &tmW, kb * GEMM_BLOCK_K, yw, fb0, pol_w);
          if (stacked) {
            tma_load_2d_pair(dst, &tmHi, kb * GEMM_BLOCK_K, 64 * rank, fb0, pol_x);
            tma_load_2d_pair(dst + PG_X_BYTES / 2, &tmLo, kb * GEMM_BLOCK_K, 64 * rank, fb0, pol_x);
          } else if (DECODE) {                      // (boxes of 64 rows)
            for (int b = 0; b < 2; ++b) {
              tma_load_2d_pair(dst + b * (PG_X_BYTES / 2), &tmHi, kb * GEMM_BLOCK_K, yx + 64 * b, fb0, pol_x);
              tma_load_2d_pair(dst + PG_X_BYTES + b * (PG_X_BYTES / 2), &tmLo, kb * GEMM_BLOCK_K, yx + 64 * b, fb0, pol_x);
            }
          } else {
            tma_load_2d_pair(dst, &tmHi, kb * GEMM_BLOCK_K, yx, fb0, pol_x);
            tma_load_2d_pair(dst + PG_X_BYTES, &tmLo, kb * GEMM_BLOCK_K, yx, fb0, pol_x);
          }
        }
      }
      TRACE(3);
      // every stage's last release has arrived before this CTA may end: an arrival of the pair's MMAs must not find the
      // shared memory given to another CTA
      for (int i = 0; i < PG_STAGES && !fail; ++i) {
        const int last = it - 1 - i;
        if (last < 0) break;
        if (!mbar_wait(smem_u32(&empty_bar[last % PG_STAGES]), (uint32_t)(last / PG_STAGES) & 1u, abort_p)) fail = DEV_TIMEOUT_PRODUCER;
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      // ---------------- MMA issuer (first CTA) ----------------
      // kind::f16: D fp32, A and B bf16, both K-major, N = 2 * half, M = 256 over the pair
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * half >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      int it = 0, seg = 0;
      for (int u = pair; u < units && !fail; u += n_pairs) {
        const Unit un = unit(u);
        for (int sl = un.s0; sl < un.s1 && !fail; ++sl, ++seg) {
          const int acc = one_buffer ? 0 : seg & 1;
          const uint32_t turn = (uint32_t)(one_buffer ? seg : seg >> 1) & 1u;
          if (!mbar_wait(smem_u32(&tmem_empty_bar[acc]), turn ^ 1u, abort_p)) { fail = DEV_TIMEOUT_MMA; break; }
          tc_fence_after();
          const uint32_t d = tmem_base + (uint32_t)acc * GEMM_TILE_N;
          const uint32_t d_lo = one_buffer ? d + GEMM_TILE_N : d;
          const int kb0 = cut(sl), kb1 = cut(sl + 1);
          for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const int s = it % PG_STAGES;
            if (!mbar_wait(smem_u32(&full_bar[s]), (uint32_t)(it / PG_STAGES) & 1u, abort_p)) { fail = DEV_TIMEOUT_MMA; break; }
            if (it == 0) TRACE(4);
            tc_fence_after();
            const uint32_t st = base + (uint32_t)s * PG_STAGE_BYTES;
            const uint64_t hi = umma_desc_sw128(st), lo = umma_desc_sw128(st + PG_X_BYTES), w = umma_desc_sw128(st + 2 * PG_X_BYTES);
#pragma unroll
            for (int k = 0; k < GEMM_BLOCK_K / 16; ++k) {
              const uint64_t adv = (uint64_t)(k * 2);
              umma_bf16_pair(d, hi + adv, w + adv, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
              if (!stacked) umma_bf16_pair(d_lo, lo + adv, w + adv, idesc, (!DECODE || kb > kb0 || k > 0) ? 1u : 0u);
            }
            umma_commit_pair(smem_u32(&empty_bar[s]));
          }
          if (!fail) umma_commit_pair(smem_u32(&tmem_full_bar[acc]));
        }
      }
      TRACE(5);
    }
  } else {
    // ---------------- epilogue: TMEM -> registers -> swizzled staging tile -> TMA store ----------------
    const int lane_base = (warp & 3) * 32, grp = (warp - 2) >> 2;   // lane quarter; half of the columns
    const uint32_t stg = base + PG_STAGES * PG_STAGE_BYTES + (uint32_t)(warp - 2) * PG_OUT_BYTES;
    uint8_t *stg_p = smem_raw + (stg - smem_u32(smem_raw));
    const uint32_t lane_off = (uint32_t)lane_base << 16;
    // stacked: lanes 64 .. of the accumulator are the lo sums of the rows in lanes 0 .. 63
    const bool lo_warp = stacked && lane_base >= 64;
    const int in_tile = stacked ? rank * 64 + (lane_base & 32) : rank * 128 + lane_base;   // this warp's 32 rows of a tile
    const uint32_t x_full = smem_u32(&x_full_bar[grp * 2 + (warp & 1)]), x_free = smem_u32(&x_free_bar[grp * 2 + (warp & 1)]);
    // (stacked) where this thread's row is handed over: 64 columns of 64 rows per stage, two stages per half of the columns
    uint8_t *const handed_p = smem_raw + (base - smem_u32(smem_raw)) + 2 * grp * PG_STAGE_BYTES + PG_X_BYTES + ((lane_base & 32) + lane) * 4;
    auto handed = [&](int i) -> float & { return *reinterpret_cast<float *>(handed_p + (i >> 6) * PG_STAGE_BYTES + (i & 63) * 256); };
    int seg = 0;
    bool ok = true;
    for (int u = pair; u < units && ok; u += n_pairs) {
      const Unit un = unit(u);
      const int nt = un.tile / row_tiles;
      const int row0 = (un.tile % row_tiles) * 256 + in_tile;   // this warp's 32 rows
      const bool part = u >= whole;                 // its slices go to partial matrices, a whole tile to the output
      auto add = [](uint32_t a, uint32_t b) { return __float_as_uint(__uint_as_float(a) + __uint_as_float(b)); };
      // first accumulator column of the sums 8 q ..; SWIGLU: blocks of 32 outputs, gate then up columns of each
      auto acc_col = [&](int q) { return SWIGLU ? grp * 32 + (q >> 3) * 64 + ((q >> 2) & 1) * half + (q & 3) * 8 : grp * 128 + q * 8; };
      auto accumulator = [&]() { return tmem_base + (uint32_t)(one_buffer ? 0 : seg & 1) * GEMM_TILE_N + lane_off; };
      auto wait_full = [&]() {                      // the segment's accumulator is complete
        ok = mbar_wait(smem_u32(&tmem_full_bar[one_buffer ? 0 : seg & 1]), (uint32_t)(one_buffer ? seg : seg >> 1) & 1u, abort_p);
        // (one row tile: every segment, or none, has rows for this warp)
        if (lo_warp && row0 < R && seg > 0) ok = ok && mbar_wait(x_free, (uint32_t)(seg - 1) & 1u, abort_p);
        ok = __all_sync(0xffffffffu, ok);
        tc_fence_after();
      };
      auto lo_ready = [&]() {                       // (stacked) the lo sums of this thread's row have been handed over
        ok = mbar_wait(x_full, (uint32_t)seg & 1u, abort_p);
        ok = __all_sync(0xffffffffu, ok);
      };
      auto read_out = [&]() {
        tc_fence_before();
        mbar_arrive_cluster(cluster_map(smem_u32(&tmem_empty_bar[one_buffer ? 0 : seg & 1]), 0));
      };
      uint32_t sum[128];                            // this thread's row: 128 columns (SWIGLU: up to 64 gate and 64 up columns), fp32
      for (int sl = un.s0; sl < un.s1; ++sl, ++seg) {
        wait_full();
        if (threadIdx.x == 64) TRACE(6);            // (the last one stays)
        if (!ok) { fail = DEV_TIMEOUT_EPILOGUE; break; }
        const uint32_t ta = accumulator();
        if (row0 < R) {                             // warp-uniform
          if (KV) {
            const int nh = N / GEMM_TILE_N;
            const float scale = __ldg(kv_scale + 2 * nt + grp);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t v[32];
              tmem_ld32(ta + (uint32_t)(grp * 128 + q * 32), v);
              if (lane == 0) bulk_wait_read<0>();
              __syncwarp();
              tmem_ld_wait();
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                __half a[8], b[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const float x = __uint_as_float(v[8 * c + j]) * scale;
                  a[j] = __float2half_rn(x);
                  b[j] = __float2half_rn(x - __half2float(a[j]));
                }
                const uint32_t off = (uint32_t)lane * 64 + (((uint32_t)c ^ (((uint32_t)lane >> 1) & 3u)) << 4);
                *reinterpret_cast<uint4 *>(stg_p + off) = *reinterpret_cast<const uint4 *>(a);
                *reinterpret_cast<uint4 *>(stg_p + PG_OUT_BYTES / 2 + off) = *reinterpret_cast<const uint4 *>(b);
              }
              fence_proxy_async();
              __syncwarp();
              if (lane == 0) {
                tma_store_2d(&tmOut, stg, q * 32, ((2 * grp) * nh + nt) * cap + row0);
                tma_store_2d(&tmOut, stg + PG_OUT_BYTES / 2, q * 32, ((2 * grp + 1) * nh + nt) * cap + row0);
                bulk_commit();
              }
            }
          } else {
            auto there = [&](int q) { return !SWIGLU || grp * 32 + (q >> 3) * 64 < half; };
            if (lo_warp || sl == un.s0 || part) {   // no sum yet: straight into the registers, all loads in flight together
              // (the first half is always there; a branch must not end between a load and its wait)
#pragma unroll
              for (int g = 0; g < (SWIGLU ? 4 : 8); ++g) tmem_ld16(ta + (uint32_t)acc_col(2 * g), *reinterpret_cast<uint32_t(*)[16]>(&sum[16 * g]));
              tmem_ld_wait();
              if (SWIGLU && there(8)) {
#pragma unroll
                for (int g = 4; g < 8; ++g) tmem_ld16(ta + (uint32_t)acc_col(2 * g), *reinterpret_cast<uint32_t(*)[16]>(&sum[16 * g]));
                tmem_ld_wait();
              }
              if (lo_warp) {
#pragma unroll
                for (int i = 0; i < 128; ++i)
                  if (there(i / 8)) handed(i) = __uint_as_float(sum[i]);
                mbar_arrive(x_full);
              } else if (stacked) {
                lo_ready();
#pragma unroll
                for (int i = 0; i < 128; ++i)
                  if (there(i / 8)) sum[i] = add(sum[i], __float_as_uint(handed(i)));
                mbar_arrive(x_free);
              } else if (DECODE) {
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                  if (!there(2 * g)) break;
                  uint32_t lo[16];
                  tmem_ld16(ta + (uint32_t)(GEMM_TILE_N + acc_col(2 * g)), lo);
                  tmem_ld_wait();
#pragma unroll
                  for (int j = 0; j < 16; ++j) sum[16 * g + j] = add(sum[16 * g + j], lo[j]);
                }
              }
            } else {
              if (stacked) lo_ready();
#pragma unroll
              for (int q = 0; q < 16; ++q) {        // (8 columns at a time: 128 running sums leave few registers)
                if (!there(q)) break;
                uint32_t v[8], lo[8];
                tmem_ld8(ta + (uint32_t)acc_col(q), v);
                if (DECODE && !stacked) {
                  tmem_ld8(ta + (uint32_t)(GEMM_TILE_N + acc_col(q)), lo);
                  tmem_ld_wait();
                } else {
                  tmem_ld_wait();
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  if (stacked) lo[j] = __float_as_uint(handed(8 * q + j));
                  if (DECODE) v[j] = add(v[j], lo[j]);
                  sum[8 * q + j] = add(sum[8 * q + j], v[j]);
                }
              }
              if (stacked) mbar_arrive(x_free);
            }
          }
        }
        if (!ok) { fail = DEV_TIMEOUT_EPILOGUE; break; }
        read_out();
        if (MODE != PG_PLAIN || row0 >= R || lo_warp || !(part || sl + 1 == un.s1)) continue;
        // a whole tile goes to the output, a slice to its partial matrix
        const int y = part ? ((un.tile - whole) * slices + sl) * 256 + in_tile : row0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int col = nt * GEMM_TILE_N + grp * 128 + q * 32;
          if (col < N) {
            if (lane == 0) bulk_wait_read<0>();     // the staging tile has been read
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 8; ++c)
              *reinterpret_cast<uint4 *>(stg_p + lane * 128 + (((uint32_t)c ^ ((uint32_t)lane & 7u)) << 4)) =
                  make_uint4(sum[32 * q + 4 * c], sum[32 * q + 4 * c + 1], sum[32 * q + 4 * c + 2], sum[32 * q + 4 * c + 3]);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(part ? &tmOut2 : &tmOut, stg, part ? grp * 128 + q * 32 : col, y);
              bulk_commit();
            }
          }
        }
      }
      if (SWIGLU && ok && row0 < R && !lo_warp) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {               // blocks of 32 outputs
          const int c0 = grp * 32 + 64 * i, col = nt * half + c0;
          if (c0 >= half || col >= (N >> 1)) break;
          if (lane == 0) bulk_wait_read<0>();       // the staging tile has been read
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 4; ++q) {             // 16 bytes = 8 outputs; 64-byte rows, 64-byte swizzle
            __nv_bfloat16 a[8], b[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float gt = __uint_as_float(sum[64 * i + 8 * q + j]);
              const float y = gt / (1.f + expf(-gt)) * __uint_as_float(sum[64 * i + 32 + 8 * q + j]);
              a[j] = __float2bfloat16_rn(y);
              b[j] = __float2bfloat16_rn(y - __bfloat162float(a[j]));
            }
            const uint32_t off = (uint32_t)lane * 64 + (((uint32_t)q ^ (((uint32_t)lane >> 1) & 3u)) << 4);
            *reinterpret_cast<uint4 *>(stg_p + off) = *reinterpret_cast<const uint4 *>(a);
            *reinterpret_cast<uint4 *>(stg_p + PG_OUT_BYTES / 2 + off) = *reinterpret_cast<const uint4 *>(b);
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&tmOut, stg, col, row0);
            tma_store_2d(&tmOut2, stg + PG_OUT_BYTES / 2, col, row0);
            bulk_commit();
          }
        }
      }
    }
    if (lane == 0) bulk_wait<0>();                  // the stores have been performed before the kernel ends
    if (threadIdx.x == 64) TRACE(7);
  }

  if (fail) {
    atomicCAS(status, 0, fail);
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);   // let copies in flight land before the shared memory is given back
  }
  tc_fence_before();
  __syncthreads();
  // The right to allocate is given back only now: a pair's release acts on both SMs, so right behind this CTA's
  // allocation it could come before the other CTA's.
  if (warp == 1) tmem_relinquish_pair();
  cluster_sync_all();                               // neither CTA leaves while the other's MMAs or arrivals may still reach it
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem_base, 512);
#undef TRACE
}

// The tiles that were left as partial matrices, added up in place (for consumers that read a plain matrix).
__global__ void __launch_bounds__(256) gemm_pair_fixup_kernel(GemmOut g, float *direct, int first_tile) {
  griddep_launch_dependents();
  griddep_wait();
  const int t = first_tile + blockIdx.x, r = (t % g.row_tiles) * 256 + blockIdx.y, n = (t / g.row_tiles) * GEMM_TILE_N + threadIdx.x;
  if (n < g.N && r < g.BN) direct[(size_t)r * g.N + n] = gemm_load_pair(g, r, n);
}

// How a launch over R rows divides its tiles: the first `whole` as whole tiles, the others in units of per_unit slices where
// that shortens the last wave.
struct PairShape { int row_tiles, whole, units, half; };
PairShape pair_shape(const GemmPairPlan &p, int R, bool narrow) {
  PairShape q{};
  q.row_tiles = (R + 255) / 256;
  q.half = 128;
  int n_tiles = p.n_tiles;
  if (p.swiglu && narrow) {
    // tiles of 96 outputs where their waves are shorter by a tenth or more (256 rows of the Qwen3-8B gate / up: two of 96
    // against two of 128, 79 us against 114; 2048 rows would gain 4 % of the waves and re-read a third more activations)
    const int F = p.N / 2, t128 = q.row_tiles * ((F + 127) / 128), t96 = q.row_tiles * ((F + 95) / 96);
    if ((t96 + p.pairs - 1) / p.pairs * 96 * 10 < (t128 + p.pairs - 1) / p.pairs * 128 * 9) { q.half = 96; n_tiles = (F + 95) / 96; }
  }
  const int tiles = q.row_tiles * n_tiles;
  q.whole = tiles;
  q.units = tiles;
  const int n = p.slices / p.per_unit;              // units of a tile
  if (n > 1 && !p.swiglu) {
    const int full = tiles / p.pairs * p.pairs, tail = tiles - full;
    // worth it where the time of the last wave that is saved (0.8 us per k-block) exceeds what writing and reading the
    // partials costs (0.06 us per slice of a tile): 16 of 16 tiles of the Qwen3-8B O projection at 256 rows 51 -> 21
    // us, not 54 of 128 at 2048 rows
    const int parts = (tail * n + p.pairs - 1) / p.pairs;
    const float saved = 0.8f * (float)(p.K / GEMM_BLOCK_K) * (float)(n - parts) / (float)n;
    if (tail && saved > 0.06f * (float)(tail * p.slices)) {
      q.whole = full;
      q.units = full + tail * n;
    }
  }
  return q;
}

// The cuts of K: units of a tile whose one row tile fills a wave, each of one or more slices of at most PG_CHAIN k-blocks as
// far as eight slices allow (each is a matrix for the consumer to read).
void pair_slices(GemmPairPlan &p) {
  const int kb = p.K / GEMM_BLOCK_K;
  // (decode: hi on its own makes half the MMAs, and the end of a slice is not hidden behind the next one)
  const int chain = !p.decode ? PG_CHAIN : p.swiglu ? 2 * PG_CHAIN : 3 * PG_CHAIN;
  if (p.swiglu) {                                   // no units: the slices meet in the epilogue's registers
    p.slices = p.per_unit = (kb + chain - 1) / chain;
    return;
  }
  int n = p.pairs / p.n_tiles;
  if (n < 1) n = p.decode ? 2 : 4;                  // more tiles than pairs: the units serve the last wave only
  if (n > 8) n = 8;
  while (n > 1 && kb / n < 8) --n;                  // a unit of fewer than 8 k-blocks costs more than it shortens
  p.per_unit = 1;
  while (kb > chain * n * p.per_unit && n * (p.per_unit + 1) <= 8) ++p.per_unit;
  p.slices = n * p.per_unit;
}

}  // namespace

size_t gemm_pair_part_floats(int N, int K, int cap, int num_sms, bool decode) {
  GemmPairPlan p;
  p.decode = decode;
  p.N = N; p.K = K; p.cap = cap; p.pairs = num_sms / 2;
  p.n_tiles = (N + GEMM_TILE_N - 1) / GEMM_TILE_N;
  pair_slices(p);
  int most = 1;
  for (int R = 256; R < cap + 256; R += 256) {
    const PairShape q = pair_shape(p, R, false);
    if ((q.units - q.whole) * p.per_unit > most) most = (q.units - q.whole) * p.per_unit;
  }
  return (size_t)most * 256 * GEMM_TILE_N;
}

int gemm_pair_plan_create(GemmPairPlan *p, int N, int K, const void *Xhi, const void *Xlo, int cap, float *out, float *part, int num_sms,
                          bool decode) {
  if (N <= 0 || N % 8 || K <= 0 || K % GEMM_BLOCK_K || cap < 1 || !out || !part || num_sms < 2) return CORUN_EINVAL;
  p->N = N; p->K = K; p->cap = cap; p->pairs = num_sms / 2; p->swiglu = false; p->out = out; p->part = part;
  p->decode = decode;
  p->n_tiles = (N + GEMM_TILE_N - 1) / GEMM_TILE_N;
  pair_slices(*p);
  int rc;
  const int box = decode ? 64 : 128;
  if ((rc = gemm_encode_map(&p->tmHi, Xhi, cap, K, box)) != 0 || (rc = gemm_encode_map(&p->tmLo, Xlo, cap, K, box)) != 0) return rc;
  if ((rc = tma_encode_store_2d(&p->tmOut, out, 1, cap, N)) != 0) return rc;
  if (p->slices > 1) {
    if ((rc = tma_encode_store_2d(&p->tmOut2, part, 1, gemm_pair_part_floats(N, K, cap, num_sms, decode) / GEMM_TILE_N, GEMM_TILE_N)) != 0) return rc;
  } else {
    p->tmOut2 = p->tmOut;
  }
  return gemm_pair_prepare();
}

GemmOut gemm_pair_out(const GemmPairPlan &p, int R, const int *zero_tiles) {
  const PairShape q = pair_shape(p, R, false);
  GemmOut g{p.out, p.part, zero_tiles, zero_tiles, p.N, 0, p.cap};
  g.row_tiles = q.row_tiles;
  g.whole = q.whole;
  g.slices = p.slices;
  return g;
}

int gemm_pair_ctas(const GemmPairPlan &p, int R, bool narrow) {
  const PairShape q = pair_shape(p, R, narrow);
  return 2 * (q.units < p.pairs ? q.units : p.pairs);
}

int gemm_pair_has_parts(const GemmPairPlan &p, int R) {
  const PairShape q = pair_shape(p, R, false);
  return q.whole < q.row_tiles * p.n_tiles ? 1 : 0;
}

cudaError_t gemm_pair_fixup_launch(const GemmPairPlan &p, int R, cudaStream_t st) {
  const PairShape q = pair_shape(p, R, false);
  const int tiles = q.row_tiles * p.n_tiles;
  if (q.whole == tiles) return cudaSuccess;
  return launch_k(gemm_pair_fixup_kernel, dim3(tiles - q.whole, R < 256 ? R : 256), dim3(256), 0, st, true, gemm_pair_out(p, R, nullptr), p.out,
                  q.whole);
}

int gemm_pair_plan_create_swiglu(GemmPairPlan *p, int F, int K, const void *Xhi, const void *Xlo, int cap, __nv_bfloat16 *out_hi,
                                 __nv_bfloat16 *out_lo, int num_sms, bool decode) {
  if (F <= 0 || F % 8 || K <= 0 || K % GEMM_BLOCK_K || cap < 1 || !out_hi || !out_lo || num_sms < 2) return CORUN_EINVAL;
  p->N = 2 * F; p->K = K; p->cap = cap; p->pairs = num_sms / 2; p->swiglu = true; p->out = nullptr;
  p->decode = decode;
  p->n_tiles = (F + 127) / 128;
  pair_slices(*p);
  int rc;
  const int box = decode ? 64 : 128;
  if ((rc = gemm_encode_map(&p->tmHi, Xhi, cap, K, box)) != 0 || (rc = gemm_encode_map(&p->tmLo, Xlo, cap, K, box)) != 0) return rc;
  if ((rc = tma_encode_store_2d(&p->tmOut, out_hi, 0, cap, F)) != 0 || (rc = tma_encode_store_2d(&p->tmOut2, out_lo, 0, cap, F)) != 0)
    return rc;
  return gemm_pair_prepare();
}

int gemm_pair_plan_create_kv(GemmPairPlan *p, int nh, int K, const void *Xhi, const void *Xlo, int cap, void *kv, int num_sms) {
  if (nh < 1 || K <= 0 || K % GEMM_BLOCK_K || cap < 32 || cap % 32 || !kv || num_sms < 2) return CORUN_EINVAL;
  p->N = nh * GEMM_TILE_N; p->K = K; p->cap = cap; p->pairs = num_sms / 2; p->swiglu = false; p->out = nullptr;
  p->n_tiles = nh;
  p->slices = p->per_unit = 1;                      // (a latent of at most 512 values)
  p->kv_heads = nh;
  int rc;
  if ((rc = gemm_encode_map(&p->tmHi, Xhi, cap, K, 128)) != 0 || (rc = gemm_encode_map(&p->tmLo, Xlo, cap, K, 128)) != 0) return rc;
  if ((rc = tma_encode_store_2d(&p->tmOut, kv, 0, (unsigned long long)4 * nh * cap, 128)) != 0) return rc;
  p->tmOut2 = p->tmOut;
  return gemm_pair_prepare();
}

int gemm_pair_prepare() {
  for (auto kernel : {gemm_pair_kernel<PG_PLAIN, false>, gemm_pair_kernel<PG_SWIGLU, false>, gemm_pair_kernel<PG_KV, false>,
                      gemm_pair_kernel<PG_PLAIN, true>, gemm_pair_kernel<PG_SWIGLU, true>}) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PG_SMEM);
    if (e != cudaSuccess) { g_last_cuda_error = (int)e; return CORUN_ECUDA; }
  }
  return CORUN_OK;
}

cudaError_t gemm_pair_launch(const GemmPairPlan &p, const CUtensorMap &tmW, int R, int *d_status, cudaStream_t st, const CUtensorMap *tmW96,
                             const float *kv_scale, unsigned long long *trace) {
  if (R < 1 || R > p.cap || (p.decode && (p.cap != 256 || !p.row_blocks)) || (p.kv_heads && !kv_scale)) return cudaErrorInvalidValue;
  const PairShape q = pair_shape(p, R, tmW96 != nullptr);
  const int pairs = q.units < p.pairs ? q.units : p.pairs;
  auto go = [&](auto kernel) {
    return launch_k(kernel, dim3(2 * pairs), dim3(PG_THREADS), PG_SMEM, st, false, q.half == 96 ? *tmW96 : tmW, p.tmHi, p.tmLo, p.tmOut, p.tmOut2,
                    R, p.N, p.K / GEMM_BLOCK_K, q.row_tiles, q.whole, q.units, p.slices, p.per_unit, q.half, d_status, p.row_blocks, p.cap, kv_scale, trace);
  };
  if (p.decode) return p.swiglu ? go(gemm_pair_kernel<PG_SWIGLU, true>) : go(gemm_pair_kernel<PG_PLAIN, true>);
  return p.kv_heads ? go(gemm_pair_kernel<PG_KV, false>) : p.swiglu ? go(gemm_pair_kernel<PG_SWIGLU, false>) : go(gemm_pair_kernel<PG_PLAIN, false>);
}

}  // namespace corun
