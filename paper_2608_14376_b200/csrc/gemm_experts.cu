// tcgen05 GEMMs of the experts of a prompt: an expert's rows in groups of up to 128, two SMs work as a pair on 512 weight rows.
#include <cuda_bf16.h>

#include "../../include/corun.h"
#include "gemm.cuh"
#include "launch.cuh"
#include "ptx.cuh"

namespace corun {

namespace {

constexpr int GE_THREADS = 320;                     // warp 0 TMA producer, warp 1 MMA issuer, warps 2-9 epilogue
constexpr int GE_STAGES = 4;
constexpr uint32_t GE_W_BYTES = 128 * GEMM_BLOCK_K * 2;      // 16 KiB: a CTA's 128 weight rows of a block
constexpr uint32_t GE_X_BYTES = 128 * GEMM_BLOCK_K * 2;      // 16 KiB: up to 128 rows, hi (first CTA) or lo (second CTA)
constexpr uint32_t GE_STAGE_BYTES = 2 * GE_W_BYTES + GE_X_BYTES;
constexpr size_t GE_SMEM = 1024 + (size_t)GE_STAGES * GE_STAGE_BYTES;

struct GemmExpertsArgs {
  float *direct;
  int N, KB, tiles_per_group, n_groups_max;
  const int *group_tab;
  const float *row_w;
  __nv_bfloat16 *sw_hi, *sw_lo;
  int *status;
};

// Group g multiplies rows g * 128 .. of Xhi / Xlo with N weight rows from the row, and the k-block, that group_tab names for it
// (three ints per group, then the number of groups in use), as the GROUPED form of gemm_rows.cu does; SWIGLU likewise: W is
// [2F, K] per group, the result row_w * silu(gate) * up as a bf16 hi / lo pair.
//
// The weights are the M operand, the rows the N operand (2 * the padded rows: W * hi, then W * lo).  A cluster of two CTAs (the
// two SMs of a TPC) owns a tile: two blocks of 256 weight rows (SWIGLU: gate and up rows of 256 outputs), 128 of each block in
// a CTA, one tcgen05.mma.cta_group::2 (M = 256) per block and k-slice.  Of the N operand the first CTA holds the hi rows and the
// second the lo rows, so that the rows enter each SM once as 128 bytes per k-block and not as 256: what bounds these products on
// one SM per tile is what the L2 delivers into an SM (2048 rows of the DeepSeek-V2-Lite layer: 3.4 GB at 9.9 TB/s, the tensor
// pipe 60 % busy).  Per k-block a CTA loads 48 KiB for 8 MMAs of 128 cycles.  Gate / up and down of those 2048 rows: 387 and 202 us
// in blocks of 64 rows on one SM per tile, 331 and 172 us so (the tensor pipe 78 and 67 % busy; 1003 rows of the Qwen3-30B-A3B layer,
// where the weights' 1.2 GB are the floor: 177 and 96 -> 168 and 88).
//
// hi and lo have an accumulator each, added at the end; K ascending.  Above 64 rows the accumulators of a tile fill tensor memory
// (the next tile begins when they are in registers), up to 64 its halves alternate.  Launched in plain stream order,
// as gemm_pair.cu.  A row's result depends neither on its place nor on the other rows.
template <bool SWIGLU>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GE_THREADS, 1)
gemm_experts_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ GemmXMaps tmX, const __grid_constant__ GemmExpertsArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[GE_STAGES];      // used in the first CTA: both CTAs' loads of a stage
  __shared__ __align__(8) uint64_t empty_bar[GE_STAGES];     // in each CTA: the MMAs have read the stage
  __shared__ __align__(8) uint64_t tmem_full_bar[2];         // in each CTA: a half of tensor memory is complete
  __shared__ __align__(8) uint64_t tmem_empty_bar[2];        // in the first CTA: both CTAs' epilogues have read it
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;
  __shared__ float row_w_s[SWIGLU ? 8 : 1][SWIGLU ? 128 : 1];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int KB = a.KB, N = a.N, F = N / 2;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < GE_STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(smem_u32(&tmem_full_bar[h]), 1);
      mbar_init(smem_u32(&tmem_empty_bar[h]), 2 * (GE_THREADS - 64));
    }
    fence_mbar_init();
    fence_proxy_async();
    prefetch_tensormap(&tmW);
#pragma unroll
    for (int i = 0; i < 3; ++i) prefetch_tensormap(rank == 0 ? &tmX.hi[i] : &tmX.lo[i]);
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(&tmem_base_s), 512);   // (the permit is given back at the end, as in gemm_pair.cu)
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // the other CTA's barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  volatile int *abort_p = &abort_flag;
  int fail = 0;

  const int n_tiles = min(a.group_tab[3 * a.n_groups_max], a.n_groups_max) * a.tiles_per_group;
  struct Tile { int g, j, wrow, wk, rows, n_pad; };
  auto tile_at = [&](int t) {
    const int g = t / a.tiles_per_group, rows = a.group_tab[3 * g + 2];
    return Tile{g, t - g * a.tiles_per_group, a.group_tab[3 * g], a.group_tab[3 * g + 1], rows, gemm_rows_padded(rows)};
  };
  // a CTA's first row of the tile's first block, and whether it has any (the last tile may end in the first CTA)
  auto own_row = [&](int j, int r) { return SWIGLU ? j * 256 + r * 128 : j * 512 + r * 256; };
  const int n_rows = SWIGLU ? F : N;
  // accumulators: block b at b * 128 columns of one half, or (more than 64 padded rows) at b * 256
  struct Halves { int next = 0; uint32_t use[2] = {0, 0}; };
  auto col_of = [](int n_pad, int half, int b) { return n_pad > 64 ? (uint32_t)b * 256u : (uint32_t)half * 256u + (uint32_t)b * 128u; };

  if (warp == 0) {
    if (elect_one()) {
      // ---------------- TMA producer (both CTAs; the bytes count on the first CTA's barrier) ----------------
      const uint64_t pol_w = l2_policy_evict_normal();       // the groups of an expert follow one another
      const uint64_t pol_x = l2_policy_evict_last();
      int it = 0;
      for (int t = pair; t < n_tiles && !fail; t += n_pairs) {
        const Tile q = tile_at(t);
        const bool mine = own_row(q.j, rank) < n_rows, other = own_row(q.j, 1) < n_rows;   // (the first CTA always has rows)
        const uint32_t tx = (other ? 4u : 2u) * GE_W_BYTES + (uint32_t)q.n_pad * 256u;     // of both CTAs
        const int y0 = q.wrow + own_row(q.j, rank), y1 = y0 + (SWIGLU ? F : 128);
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % GE_STAGES;
          if (!mbar_wait(smem_u32(&empty_bar[s]), ((uint32_t)(it / GE_STAGES) & 1u) ^ 1u, abort_p)) { fail = DEV_TIMEOUT_PRODUCER; break; }
          const uint32_t fb = smem_u32(&full_bar[s]), dst = base + (uint32_t)s * GE_STAGE_BYTES;
          if (rank == 0) mbar_arrive_expect_tx(fb, tx);
          const uint32_t fb0 = cluster_map(fb, 0);
          const int x = (q.wk + kb) * GEMM_BLOCK_K;
          if (mine) {
            tma_load_2d_pair(dst, &tmW, x, y0, fb0, pol_w);
            tma_load_2d_pair(dst + GE_W_BYTES, &tmW, x, y1, fb0, pol_w);
          }
          int r = 0;
          auto box = [&](int i, int rows) {
            tma_load_2d_pair(dst + 2 * GE_W_BYTES + (uint32_t)r * 128u, rank == 0 ? &tmX.hi[i] : &tmX.lo[i], kb * GEMM_BLOCK_K, q.g * 128 + r, fb0, pol_x);
            r += rows;
          };
          if (q.n_pad >= 64) box(0, 64);
          if (q.n_pad == 128) box(0, 64);
          if (q.n_pad & 32) box(1, 32);
          if (q.n_pad & 16) box(2, 16);
        }
      }
      // every stage's last release has arrived before this CTA may end: an arrival of the pair's MMAs must not find the
      // shared memory given to another CTA
      for (int i = 0; i < GE_STAGES && !fail; ++i) {
        const int last = it - 1 - i;
        if (last < 0) break;
        if (!mbar_wait(smem_u32(&empty_bar[last % GE_STAGES]), (uint32_t)(last / GE_STAGES) & 1u, abort_p)) fail = DEV_TIMEOUT_PRODUCER;
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      // ---------------- MMA issuer (first CTA) ----------------
      Halves hv;
      int it = 0;
      for (int t = pair; t < n_tiles && !fail; t += n_pairs) {
        const Tile q = tile_at(t);
        const bool both = q.n_pad > 64;
        const int half = both ? 0 : hv.next;
        for (int h = 0; h < 2 && !fail; ++h)
          if (both || h == half) {
            if (!mbar_wait(smem_u32(&tmem_empty_bar[h]), (hv.use[h] & 1u) ^ 1u, abort_p)) fail = DEV_TIMEOUT_MMA;
            ++hv.use[h];
          }
        if (fail) break;
        if (!both) hv.next ^= 1;
        tc_fence_after();
        // kind::f16: D fp32, A and B bf16, both K-major, N = 2 * n_pad, M = 256 over the pair
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(q.n_pad >> 2) << 17) | ((uint32_t)(256 >> 4) << 24);
        const uint32_t d0 = tmem_base + col_of(q.n_pad, half, 0), d1 = tmem_base + col_of(q.n_pad, half, 1);
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % GE_STAGES;
          if (!mbar_wait(smem_u32(&full_bar[s]), (uint32_t)(it / GE_STAGES) & 1u, abort_p)) { fail = DEV_TIMEOUT_MMA; break; }
          tc_fence_after();
          const uint32_t st = base + (uint32_t)s * GE_STAGE_BYTES;
          const uint64_t w0 = umma_desc_sw128(st), w1 = umma_desc_sw128(st + GE_W_BYTES), x = umma_desc_sw128(st + 2 * GE_W_BYTES);
#pragma unroll
          for (int k = 0; k < GEMM_BLOCK_K / 16; ++k) {
            const uint64_t adv = (uint64_t)(k * 2);
            const uint32_t more = (kb > 0 || k > 0) ? 1u : 0u;
            umma_bf16_pair(d0, w0 + adv, x + adv, idesc, more);
            umma_bf16_pair(d1, w1 + adv, x + adv, idesc, more);
          }
          umma_commit_pair(smem_u32(&empty_bar[s]));
        }
        if (fail) break;
        for (int h = 0; h < 2; ++h)
          if (both || h == half) umma_commit_pair(smem_u32(&tmem_full_bar[h]));
      }
    }
  } else {
    // ---------------- epilogue: TMEM -> registers -> global, as in gemm_rows.cu ----------------
    const int lane_base = (warp & 3) * 32, grp = (warp - 2) >> 2;
    const uint32_t t_lane = tmem_base + ((uint32_t)lane_base << 16);
    Halves hv;
    for (int t = pair; t < n_tiles; t += n_pairs) {
      const Tile q = tile_at(t);
      const bool both = q.n_pad > 64;
      const int half = both ? 0 : hv.next;
      const int n0 = own_row(q.j, rank), chunks = (q.rows + 7) >> 3;
      const size_t row0 = (size_t)q.g * 128;
      float *const my_w = row_w_s[SWIGLU ? warp - 2 : 0];          // (ahead of the wait: the rows' routing weights)
      if (SWIGLU) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k) my_w[32 * k + lane] = a.row_w[row0 + 32 * k + lane];
        __syncwarp();
      }
      bool ok = true;
      for (int h = 0; h < 2; ++h)
        if (both || h == half) {
          ok = ok && mbar_wait(smem_u32(&tmem_full_bar[h]), hv.use[h] & 1u, abort_p);
          ++hv.use[h];
        }
      if (!both) hv.next ^= 1;
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { fail = DEV_TIMEOUT_EPILOGUE; break; }
      tc_fence_after();
      const uint32_t t0 = t_lane + col_of(q.n_pad, half, 0), t1 = t_lane + col_of(q.n_pad, half, 1);
      // all sums of this thread into registers first (SWIGLU: gate and up of every other chunk of eight rows; else all rows of
      // one block): tensor memory is then free for the next tile while this one is worked on and stored
      float v[128];
      const bool live = n0 + lane_base + (SWIGLU ? 0 : grp * 128) < n_rows;   // warp-uniform
      if (live) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if ((SWIGLU ? grp + 2 * i : 2 * i) >= chunks) break;
          uint32_t x0[8], x1[8], x2[8], x3[8];
          if (SWIGLU) {
            const uint32_t at = (uint32_t)(8 * (grp + 2 * i));
            tmem_ld8(t0 + at, x0);
            tmem_ld8(t0 + (uint32_t)q.n_pad + at, x1);
            tmem_ld8(t1 + at, x2);
            tmem_ld8(t1 + (uint32_t)q.n_pad + at, x3);
          } else {
            const uint32_t tb = (grp == 0 ? t0 : t1) + (uint32_t)(16 * i);
            tmem_ld8(tb, x0);
            tmem_ld8(tb + (uint32_t)q.n_pad, x1);
            tmem_ld8(tb + 8, x2);
            tmem_ld8(tb + (uint32_t)q.n_pad + 8, x3);
          }
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            v[16 * i + j] = __uint_as_float(x0[j]) + __uint_as_float(x1[j]);
            v[16 * i + 8 + j] = __uint_as_float(x2[j]) + __uint_as_float(x3[j]);
          }
        }
      }
      tc_fence_before();
      for (int h = 0; h < 2; ++h)
        if (both || h == half) mbar_arrive_cluster(cluster_map(smem_u32(&tmem_empty_bar[h]), 0));
      if (!live) continue;
      if (SWIGLU) {
        const int f = n0 + lane_base + lane;          // (F is a multiple of 8: both lanes of a pair are inside or not)
        const bool odd = lane & 1;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int c = grp + 2 * i;
          if (c >= chunks) break;
          float y[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float gt = v[16 * i + j], w = my_w[8 * c + j];
            y[j] = __fdividef(gt, 1.f + __expf(-gt)) * v[16 * i + 8 + j];
            y[j] = w != 0.f ? w * y[j] : 0.f;
          }
          // lanes in pairs: the even one stores two outputs of row 2 i, the odd one of row 2 i + 1
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            const float got = __shfl_xor_sync(0xffffffffu, odd ? y[j] : y[j + 1], 1);
            const float v0 = odd ? got : y[j], v1 = odd ? y[j + 1] : got;
            const int r = 8 * c + j + (odd ? 1 : 0);
            const __nv_bfloat16 h0 = __float2bfloat16_rn(v0), h1 = __float2bfloat16_rn(v1);
            const __nv_bfloat162 hi = __halves2bfloat162(h0, h1),
                                 lo = __halves2bfloat162(__float2bfloat16_rn(v0 - __bfloat162float(h0)), __float2bfloat16_rn(v1 - __bfloat162float(h1)));
            if (f < F && r < q.rows) {
              const size_t o = (row0 + r) * F + (f & ~1);
              *reinterpret_cast<__nv_bfloat162 *>(a.sw_hi + o) = hi;
              *reinterpret_cast<__nv_bfloat162 *>(a.sw_lo + o) = lo;
            }
          }
        }
      } else {
        const int n = n0 + grp * 128 + lane_base + lane;   // each group of warps has a block
        float *d = a.direct + row0 * N + n;
#pragma unroll
        for (int i = 0; i < 128; ++i)
          if (i < q.rows && n < N) d[(size_t)i * N] = v[i];
      }
    }
  }

  if (fail) {
    atomicCAS(a.status, 0, fail);
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);   // let copies in flight land before the shared memory is given back
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_relinquish_pair();
  cluster_sync_all();                               // neither CTA leaves while the other's MMAs or arrivals may still reach it
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem_base, 512);
}

int create(GemmExpertsPlan *p, int N, int K, const void *Xhi, const void *Xlo, int n_groups, const int *group_tab, int num_sms) {
  if (N <= 0 || K <= 0 || K % GEMM_BLOCK_K || n_groups < 1 || !group_tab || num_sms < 2) return CORUN_EINVAL;
  p->N = N; p->K = K; p->n_groups_max = n_groups; p->group_tab = group_tab; p->pairs = num_sms / 2;
  for (auto kernel : {gemm_experts_kernel<false>, gemm_experts_kernel<true>}) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GE_SMEM);
    if (e != cudaSuccess) { g_last_cuda_error = (int)e; return CORUN_ECUDA; }
  }
  return gemm_encode_x(&p->tmX, Xhi, Xlo, (unsigned long long)n_groups * 128, K);
}

}  // namespace

int gemm_experts_plan_create(GemmExpertsPlan *p, int N, int K, const void *Xhi, const void *Xlo, int n_groups, float *direct, const int *group_tab,
                             int num_sms) {
  if (N % 128 || !direct) return CORUN_EINVAL;
  p->direct = direct;
  p->tiles_per_group = (N + 511) / 512;
  return create(p, N, K, Xhi, Xlo, n_groups, group_tab, num_sms);
}

int gemm_experts_plan_create_swiglu(GemmExpertsPlan *p, int F, int K, const void *Xhi, const void *Xlo, int n_groups, __nv_bfloat16 *out_hi,
                                    __nv_bfloat16 *out_lo, const float *row_w, const int *group_tab, int num_sms) {
  if (F <= 0 || F % 8 || !out_hi || !out_lo || !row_w) return CORUN_EINVAL;
  p->sw_hi = out_hi; p->sw_lo = out_lo; p->row_w = row_w;
  p->tiles_per_group = (F + 255) / 256;
  return create(p, 2 * F, K, Xhi, Xlo, n_groups, group_tab, num_sms);
}

cudaError_t gemm_experts_launch(const GemmExpertsPlan &p, const CUtensorMap &tmW, int *d_status, cudaStream_t st) {
  const int tiles = p.n_groups_max * p.tiles_per_group, pairs = tiles < p.pairs ? tiles : p.pairs;
  const GemmExpertsArgs a{p.direct, p.N, p.K / GEMM_BLOCK_K, p.tiles_per_group, p.n_groups_max, p.group_tab, p.row_w, p.sw_hi, p.sw_lo, d_status};
  auto go = [&](auto kernel) { return launch_k(kernel, dim3(2 * pairs), dim3(GE_THREADS), GE_SMEM, st, false, tmW, p.tmX, a); };
  return p.sw_hi ? go(gemm_experts_kernel<true>) : go(gemm_experts_kernel<false>);
}

}  // namespace corun
