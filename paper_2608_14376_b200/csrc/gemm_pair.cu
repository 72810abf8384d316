// tcgen05 GEMM for many activation rows (prompts beyond one small chunk): two SMs work as a pair on one tile.
#include <cudaTypedefs.h>

#include "../../include/corun.h"
#include "gemm.cuh"
#include "launch.cuh"
#include "ptx.cuh"

namespace corun {

namespace {

constexpr int PG_THREADS = 192;                     // warp 0 TMA producer, warp 1 MMA issuer, warps 2-5 epilogue
constexpr int PG_STAGES = 4;
constexpr uint32_t PG_X_BYTES = 128 * GEMM_BLOCK_K * 2;      // 16 KiB: a CTA's 128 activation rows, hi or lo
constexpr uint32_t PG_W_BYTES = 128 * GEMM_BLOCK_K * 2;      // 16 KiB: a CTA's half of the 256 weight rows
constexpr uint32_t PG_STAGE_BYTES = 2 * PG_X_BYTES + PG_W_BYTES;
constexpr uint32_t PG_OUT_BYTES = 32 * 128;                  // one staging tile of the epilogue: 32 rows x 128 bytes
constexpr size_t PG_SMEM = 1024 + (size_t)PG_STAGES * PG_STAGE_BYTES + 4 * 2 * PG_OUT_BYTES;

// out[r, n] = sum_k W[n, k] * (Xhi[r, k] + Xlo[r, k]) for tiles of 256 rows x 256 weight rows.
//
// A cluster of two CTAs (the two SMs of a TPC) owns a tile: CTA i holds activation rows 128 i .. of it (hi and lo, the
// M side) and weight rows 128 i .. (the N side), and one thread of the first CTA issues tcgen05.mma.cta_group::2
// (M = 256, N = 256) over both; each CTA's tensor memory receives its own 128 rows x all 256 weight rows.  Per k-block
// a CTA loads 48 KiB for 8 MMAs of 128 cycles: 48 bytes per cycle, where one CTA on its own (128 rows x 256 weight
// rows) would need 64 and be bound by what the L2 delivers into an SM.  hi and lo go into the same accumulator,
// k-slice by k-slice.  Two accumulators of 256 columns alternate, so that a tile's epilogue overlaps the next tile.
//
// A tile's sum runs over the whole of K in one accumulator whatever the number of rows, the tile order or the grid:
// a row's result depends on its own activations only, not on its place among the rows nor on their number.
//
// Launched in plain stream order (no programmatic launch): a pair's two SMs are taken and left together, never while a
// CTA of a neighbouring kernel of the stream is on one of them.
//
// The tiles are walked row tile first (pair p takes tiles p, p + pairs, ...), so that the pairs that run at the same
// time share weight tiles in L2 and the weights are read from HBM once.
//
// SWIGLU: W is a gate / up matrix ([2F, K]); a tile is 128 gate rows (first CTA) and the up rows of the same outputs
// (second CTA), and the epilogue writes silu(gate) * up as the bf16 hi/lo pair the down GEMM reads.
template <bool SWIGLU>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PG_THREADS, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmHi,
                 const __grid_constant__ CUtensorMap tmLo, const __grid_constant__ CUtensorMap tmOut,
                 const __grid_constant__ CUtensorMap tmOut2, int R, int N, int KB, int row_tiles, int n_tiles, int *status) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[PG_STAGES];      // used in the first CTA: both CTAs' loads of a stage
  __shared__ __align__(8) uint64_t empty_bar[PG_STAGES];     // in each CTA: the MMAs have read the stage
  __shared__ __align__(8) uint64_t tmem_full_bar[2];         // in each CTA: an accumulator is complete
  __shared__ __align__(8) uint64_t tmem_empty_bar[2];        // in the first CTA: both CTAs' epilogues have read it
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int tiles = row_tiles * n_tiles;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < PG_STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tmem_full_bar[a]), 1);
      mbar_init(smem_u32(&tmem_empty_bar[a]), 256);
    }
    fence_mbar_init();
    fence_proxy_async();
    prefetch_tensormap(&tmW);
    prefetch_tensormap(&tmHi);
    prefetch_tensormap(&tmLo);
    prefetch_tensormap(&tmOut);
    if (SWIGLU) prefetch_tensormap(&tmOut2);
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(&tmem_base_s), 512);   // (the permit is given back at the end: see there)
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // the other CTA's barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  volatile int *abort_p = &abort_flag;
  int fail = 0;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer (both CTAs; the bytes count on the first CTA's barrier) ----------------
      const uint64_t pol_w = l2_policy_evict_first();        // a weight tile is used by the row tiles that run now
      const uint64_t pol_x = l2_policy_evict_last();
      auto load_w = [&](int it, int tile, int kb) {
        const int s = it % PG_STAGES, nt = tile / row_tiles;
        const uint32_t fb = smem_u32(&full_bar[s]);
        if (rank == 0) mbar_arrive_expect_tx(fb, 2 * PG_STAGE_BYTES);
        const int y = SWIGLU ? nt * 128 + rank * (N >> 1) : nt * GEMM_TILE_N + rank * 128;
        tma_load_2d_pair(base + (uint32_t)s * PG_STAGE_BYTES + 2 * PG_X_BYTES, &tmW, kb * GEMM_BLOCK_K, y, cluster_map(fb, 0), pol_w);
      };
      auto load_x = [&](int it, int tile, int kb) {
        const int s = it % PG_STAGES, y = (tile % row_tiles) * 256 + rank * 128;
        const uint32_t fb = cluster_map(smem_u32(&full_bar[s]), 0), dst = base + (uint32_t)s * PG_STAGE_BYTES;
        tma_load_2d_pair(dst, &tmHi, kb * GEMM_BLOCK_K, y, fb, pol_x);
        tma_load_2d_pair(dst + PG_X_BYTES, &tmLo, kb * GEMM_BLOCK_K, y, fb, pol_x);
      };
      int it = 0;
      for (int tile = pair; tile < tiles && !fail; tile += n_pairs)
        for (int kb = 0; kb < KB; ++kb, ++it) {
          if (!mbar_wait(smem_u32(&empty_bar[it % PG_STAGES]), ((uint32_t)(it / PG_STAGES) & 1u) ^ 1u, abort_p)) {
            fail = DEV_TIMEOUT_PRODUCER;
            break;
          }
          load_w(it, tile, kb);
          load_x(it, tile, kb);
        }
      // every stage's last release has arrived before this CTA may end: an arrival of the pair's MMAs must not find the
      // shared memory given to another CTA
      for (int i = 0; i < PG_STAGES && !fail; ++i) {
        const int last = it - 1 - i;                // the it-th last use of the ring
        if (last < 0) break;
        if (!mbar_wait(smem_u32(&empty_bar[last % PG_STAGES]), (uint32_t)(last / PG_STAGES) & 1u, abort_p)) fail = DEV_TIMEOUT_PRODUCER;
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      // ---------------- MMA issuer (first CTA) ----------------
      // kind::f16: D fp32, A and B bf16, both K-major, N = 256, M = 256 over the pair
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GEMM_TILE_N >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      int it = 0, seg = 0;
      for (int tile = pair; tile < tiles && !fail; tile += n_pairs, ++seg) {
        const int acc = seg & 1;
        if (!mbar_wait(smem_u32(&tmem_empty_bar[acc]), ((uint32_t)(seg >> 1) & 1u) ^ 1u, abort_p)) { fail = DEV_TIMEOUT_MMA; break; }
        tc_fence_after();
        const uint32_t d = tmem_base + (uint32_t)acc * GEMM_TILE_N;
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % PG_STAGES;
          if (!mbar_wait(smem_u32(&full_bar[s]), (uint32_t)(it / PG_STAGES) & 1u, abort_p)) { fail = DEV_TIMEOUT_MMA; break; }
          tc_fence_after();
          const uint32_t st = base + (uint32_t)s * PG_STAGE_BYTES;
          const uint64_t hi = umma_desc_sw128(st), lo = umma_desc_sw128(st + PG_X_BYTES), w = umma_desc_sw128(st + 2 * PG_X_BYTES);
#pragma unroll
          for (int k = 0; k < GEMM_BLOCK_K / 16; ++k) {
            const uint64_t adv = (uint64_t)(k * 2);
            umma_bf16_pair(d, hi + adv, w + adv, idesc, (kb > 0 || k > 0) ? 1u : 0u);
            umma_bf16_pair(d, lo + adv, w + adv, idesc, 1u);
          }
          umma_commit_pair(smem_u32(&empty_bar[s]));
        }
        if (!fail) umma_commit_pair(smem_u32(&tmem_full_bar[acc]));
      }
    }
  } else {
    // ---------------- epilogue: TMEM -> registers -> swizzled staging tile -> TMA store ----------------
    const int lane_base = (warp & 3) * 32;
    const uint32_t stg = base + PG_STAGES * PG_STAGE_BYTES + (uint32_t)(warp - 2) * 2 * PG_OUT_BYTES;
    uint8_t *stg_p = smem_raw + (stg - smem_u32(smem_raw));
    const uint32_t swz = (uint32_t)(lane & 7);
    int seg = 0, buf = 0;                           // buf: the staging tile of the next store (they alternate)
    for (int tile = pair; tile < tiles; tile += n_pairs, ++seg) {
      const int acc = seg & 1, nt = tile / row_tiles;
      const int row0 = (tile % row_tiles) * 256 + rank * 128 + lane_base;   // this warp's 32 rows
      bool ok = mbar_wait(smem_u32(&tmem_full_bar[acc]), (uint32_t)(seg >> 1) & 1u, abort_p);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { fail = DEV_TIMEOUT_EPILOGUE; break; }
      tc_fence_after();
      const uint32_t ta = tmem_base + (uint32_t)acc * GEMM_TILE_N + ((uint32_t)lane_base << 16);
      if (row0 < R) {                               // warp-uniform
        if (SWIGLU) {
          for (int c0 = 0; c0 < 128; c0 += 64) {
            const int col = nt * 128 + c0;
            if (col >= (N >> 1)) break;
            if (lane == 0) bulk_wait_read<0>();     // the staging tiles have been read
            __syncwarp();
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              uint32_t g[32], u[32];
              tmem_ld32(ta + (uint32_t)(c0 + 32 * half), g);
              tmem_ld32(ta + (uint32_t)(128 + c0 + 32 * half), u);
              tmem_ld_wait();
#pragma unroll
              for (int q = 0; q < 4; ++q) {         // 16 bytes = 8 outputs
                __nv_bfloat16 a[8], b[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const float gt = __uint_as_float(g[8 * q + j]);
                  const float y = gt / (1.f + expf(-gt)) * __uint_as_float(u[8 * q + j]);
                  a[j] = __float2bfloat16_rn(y);
                  b[j] = __float2bfloat16_rn(y - __bfloat162float(a[j]));
                }
                const uint32_t off = (uint32_t)lane * 128 + (((uint32_t)(4 * half + q) ^ swz) << 4);
                *reinterpret_cast<uint4 *>(stg_p + off) = *reinterpret_cast<const uint4 *>(a);
                *reinterpret_cast<uint4 *>(stg_p + PG_OUT_BYTES + off) = *reinterpret_cast<const uint4 *>(b);
              }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&tmOut, stg, col, row0);
              tma_store_2d(&tmOut2, stg + PG_OUT_BYTES, col, row0);
              bulk_commit();
            }
          }
        } else {
          for (int c0 = 0; c0 < GEMM_TILE_N; c0 += 32, buf ^= 1) {
            const int col = nt * GEMM_TILE_N + c0;
            if (col >= N) break;
            uint32_t v[32];
            tmem_ld32(ta + (uint32_t)c0, v);
            if (lane == 0) bulk_wait_read<1>();     // the store before the last one has read this staging tile
            __syncwarp();
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 8; ++q)
              *reinterpret_cast<uint4 *>(stg_p + buf * PG_OUT_BYTES + lane * 128 + (((uint32_t)q ^ swz) << 4)) =
                  make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&tmOut, stg + (uint32_t)buf * PG_OUT_BYTES, col, row0);
              bulk_commit();
            }
          }
        }
      }
      tc_fence_before();
      mbar_arrive_cluster(cluster_map(smem_u32(&tmem_empty_bar[acc]), 0));
    }
    if (lane == 0) bulk_wait<0>();                  // the stores have been performed before the kernel ends
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
}

}  // namespace

int gemm_pair_plan_create(GemmPairPlan *p, int N, int K, const void *Xhi, const void *Xlo, int cap, float *out, int num_sms) {
  if (N <= 0 || N % 8 || K <= 0 || K % GEMM_BLOCK_K || cap < 1 || !out || num_sms < 2) return CORUN_EINVAL;
  p->N = N; p->K = K; p->cap = cap; p->pairs = num_sms / 2; p->swiglu = false; p->out = out;
  p->n_tiles = (N + GEMM_TILE_N - 1) / GEMM_TILE_N;
  int rc;
  if ((rc = gemm_encode_map(&p->tmHi, Xhi, cap, K, 128)) != 0 || (rc = gemm_encode_map(&p->tmLo, Xlo, cap, K, 128)) != 0) return rc;
  if ((rc = tma_encode_store_2d(&p->tmOut, out, 1, cap, N)) != 0) return rc;
  p->tmOut2 = p->tmOut;
  return gemm_pair_prepare();
}

int gemm_pair_plan_create_swiglu(GemmPairPlan *p, int F, int K, const void *Xhi, const void *Xlo, int cap, __nv_bfloat16 *out_hi,
                                 __nv_bfloat16 *out_lo, int num_sms) {
  if (F <= 0 || F % 8 || K <= 0 || K % GEMM_BLOCK_K || cap < 1 || !out_hi || !out_lo || num_sms < 2) return CORUN_EINVAL;
  p->N = 2 * F; p->K = K; p->cap = cap; p->pairs = num_sms / 2; p->swiglu = true; p->out = nullptr;
  p->n_tiles = (F + 127) / 128;
  int rc;
  if ((rc = gemm_encode_map(&p->tmHi, Xhi, cap, K, 128)) != 0 || (rc = gemm_encode_map(&p->tmLo, Xlo, cap, K, 128)) != 0) return rc;
  if ((rc = tma_encode_store_2d(&p->tmOut, out_hi, 0, cap, F)) != 0 || (rc = tma_encode_store_2d(&p->tmOut2, out_lo, 0, cap, F)) != 0)
    return rc;
  return gemm_pair_prepare();
}

int gemm_pair_prepare() {
  cudaError_t e = cudaFuncSetAttribute(gemm_pair_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PG_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_pair_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PG_SMEM);
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return CORUN_ECUDA; }
  return CORUN_OK;
}

cudaError_t gemm_pair_launch(const GemmPairPlan &p, const CUtensorMap &tmW, int R, int *d_status, cudaStream_t st) {
  if (R < 1 || R > p.cap) return cudaErrorInvalidValue;
  const int row_tiles = (R + 255) / 256, tiles = row_tiles * p.n_tiles;
  const int pairs = tiles < p.pairs ? tiles : p.pairs;
  auto go = [&](auto kernel) {
    return launch_k(kernel, dim3(2 * pairs), dim3(PG_THREADS), PG_SMEM, st, false, tmW, p.tmHi, p.tmLo, p.tmOut, p.tmOut2, R, p.N,
                    p.K / GEMM_BLOCK_K, row_tiles, p.n_tiles, d_status);
  };
  return p.swiglu ? go(gemm_pair_kernel<true>) : go(gemm_pair_kernel<false>);
}

}  // namespace corun
