// tcgen05 GEMM for up to 128 activation rows (decode steps, short prompts, the rows of an expert): the weights are the M
// operand, the rows the N operand.
#include <cuda_bf16.h>

#include "../../include/corun.h"
#include "gemm.cuh"
#include "launch.cuh"
#include "ptx.cuh"

namespace corun {

namespace {

constexpr int GR_THREADS = 320;                     // warp 0 TMA producer, warp 1 MMA issuer, warps 2-9 epilogue
constexpr int GR_MAX_STAGES = 11;
constexpr uint32_t GR_W_BYTES = 128 * GEMM_BLOCK_K * 2;      // 16 KiB: what one MMA reads of the weights

struct GemmRowsArgs {
  float *direct, *ws;
  const int *cta_start;
  int N, KB, BN, R, stages, tile_n, w_rows;         // w_rows: weight rows per box (128; SWIGLU: gate rows = up rows of a tile)
  uint32_t stage_bytes;
  const float *row_keep;
  int keep_pitch, keep_div;
  const int *group_tab;
  int tiles_per_group;
  int *status;
  unsigned long long *trace;
  __nv_bfloat16 *sw_hi, *sw_lo;
  const int *row_blocks;
};

// out[r, n] = sum_k W[n, k] * (Xhi[r, k] + Xlo[r, k]).
//
// An MMA multiplies 128 weight rows (M, accumulator lanes) by the hi and the lo parts of the rows (N = 2 * the padded rows:
// accumulator columns 0 .. are W * hi, the columns behind them W * lo); a tile is one or two such blocks of weight rows (tile_n
// = 128 or 256).  What a k-block costs beside its weights, the activations' bytes into the SM (rows x 256 bytes: an SM gets about
// 43 bytes per cycle out of L2, of which the weights at the memory's rate are 24), the MMAs and the end of a tile, is so
// proportional to the rows there are: they are counted on the device (row_blocks bits 8 .., or the group's rows).  With the
// rows as the M operand (128 lanes whatever there is, and a tile's end of 256 columns through shared memory) the end of a tile took
// 2.9 us at 8 rows of 16; here a warp stores its 32 weight rows' value of one activation row as one 128-byte segment.
// tile_n = 128 up to 32 padded rows where that leaves a CTA's share of K as it is (gemm_plan_fill).
//
// The flat space of (tile, k-block) pairs is cut into one contiguous range per CTA, a function of (N, K, SM count); role loops
// walk the range segment by segment (the part of the range that falls into one tile).  hi and lo have an accumulator each, added
// at the end; K ascending.  A row's result depends neither on its place nor on the other rows.
//
// MASKED: row r of tile column n is stored only where row_keep[r * keep_pitch + (n / 256) / keep_div] != 0 (rows that no
//   consumer will read are skipped).
// SWIGLU: W is a gate / up matrix ([2F, K]); a tile is w_rows gate rows and the up rows of the same outputs as the two blocks
//   (fewer than 128, or 64, rows are loaded of each: the other lanes hold meaningless values that are never read back; up to 64 rows the
//   MMAs read 64, half the shared memory that bounds them at few activation rows), every CTA owns whole tiles, and the epilogue writes
//   silu(gate) * up as a bf16 hi / lo pair.
// SWIGLU with MASKED: a stack of keep_pitch such matrices (keep_div tiles each); times row_keep[r, block], exact zeros where it is zero.
// GROUPED: a tile belongs to one group: group_tab holds, per group, the first weight row, the first weight k-block and the rows
//   in use, and behind its keep_pitch entries the number of groups in use (the first ones); the CTAs take the tiles of those
//   groups in turn.  The group's activations are rows group * BN .., its results rows group * BN .. of the output.
// SWIGLU with GROUPED: times row_keep[group * BN + r].
// SELECT (with GROUPED; the experts of up to 64 rows): the groups are the experts that at least one row selected, all rows of the
//   step together.  group_tab holds keep_div ints, the selected experts of every row (< 0: none); every CTA makes the ascending
//   list of them itself.  row_keep: routing weights [rows][keep_pitch]; only rows that selected the expert are stored.
template <bool MASKED, bool GROUPED, bool SWIGLU, bool SELECT>
__global__ void __launch_bounds__(GR_THREADS, 1)
gemm_rows_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ GemmXMaps tmX, const __grid_constant__ GemmRowsArgs a) {
  extern __shared__ uint8_t smem_raw[];
  // optional per-CTA timeline (debug): 8 globaltimer stamps
#define TRACE(i) do { if (a.trace) a.trace[(size_t)blockIdx.x * 8 + (i)] = globaltimer_ns(); } while (0)
  if (threadIdx.x == 0) TRACE(0);
  griddep_launch_dependents();   // the next kernel may start its prologue
  __shared__ __align__(8) uint64_t full_bar[GR_MAX_STAGES];
  __shared__ __align__(8) uint64_t empty_bar[GR_MAX_STAGES];
  __shared__ __align__(8) uint64_t tmem_full_bar[2];    // one pair per half of tensor memory
  __shared__ __align__(8) uint64_t tmem_empty_bar[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;
  __shared__ uint32_t sel_bits[SELECT ? GEMM_MAX_SELECT / 32 : 1];   // SELECT: which experts have a row
  __shared__ unsigned short sel_list[SELECT ? GEMM_MAX_SELECT : 1];  // and their list, ascending
  __shared__ int sel_n;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x, KB = a.KB, BN = a.BN, N = a.N;
  const int MT = SWIGLU ? 2 : a.tile_n >> 7;        // blocks of 128 weight rows per tile
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t w_box = (uint32_t)a.w_rows * GEMM_BLOCK_K * 2, w_bytes = (uint32_t)MT * w_box;
  const bool m64 = SWIGLU && a.w_rows <= 64;        // MMAs of 64 weight rows: 16 of them in the first lanes of each quarter
  const int sw_fb = (SWIGLU && MASKED) ? N / (2 * a.keep_pitch) : N / 2;   // SWIGLU: gate rows of a matrix
  int n_pad = gemm_rows_padded(BN);                          // padded rows (of the launch; GROUPED: of the segment)

  // the group of the CTA's i-th tile (read only after the wait for the table below)
  int g_tile = -1, g_id = 0, g_j = 0, g_wrow = 0, g_wk = 0, g_rows = 0;
  auto look = [&](int tile) {
    if (GROUPED && tile != g_tile) {
      const int t = cta + tile * (int)gridDim.x;
      g_tile = tile;
      g_id = t / a.tiles_per_group;
      g_j = t - g_id * a.tiles_per_group;
      if (SELECT) {
        g_id = sel_list[g_id];
        g_wrow = SWIGLU ? g_id * N : 0;
        g_wk = SWIGLU ? 0 : g_id * KB;
        g_rows = a.R;
        return;
      }
      g_wrow = a.group_tab[3 * g_id];
      g_wk = a.group_tab[3 * g_id + 1];
      g_rows = a.group_tab[3 * g_id + 2];
      n_pad = gemm_rows_padded(g_rows);
    }
  };
  // behind the wait for the predecessor: the rows of this step
  auto read_rows = [&]() {
    if ((!GROUPED || SELECT) && a.row_blocks) {
      griddep_wait();
      const int v = *reinterpret_cast<const volatile int *>(a.row_blocks), n = v >> 8;
      n_pad = gemm_rows_padded(min(BN, n > 0 ? n : (v & 2) ? BN : 64));
    }
  };
  // A segment's accumulators: block mt's columns start at mt * 128 of one half of tensor memory, or (more than 64 padded rows
  // in two blocks) of mt * 256: then both halves are taken.  The roles walk the same segments and count the uses alike.
  struct Halves { int next = 0; uint32_t use[2] = {0, 0}; };
  auto wide_seg = [&]() { return MT == 2 && n_pad > 64; };
  auto mt_col = [&](int half, int mt) { return wide_seg() ? (uint32_t)mt * 256u : (uint32_t)half * 256u + (uint32_t)mt * 128u; };

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(smem_u32(&tmem_full_bar[h]), 1);
      mbar_init(smem_u32(&tmem_empty_bar[h]), GR_THREADS - 64);
    }
    fence_mbar_init();
    fence_proxy_async();
    prefetch_tensormap(&tmW);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      prefetch_tensormap(&tmX.hi[i]);
      prefetch_tensormap(&tmX.lo[i]);
    }
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_s), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  volatile int *abort_p = &abort_flag;
  if (threadIdx.x == 0) TRACE(1);

  // GROUPED: the CTA walks the tiles cta, cta + grid, ... of the groups in use, every tile whole; the flat range counts the
  // k-blocks of those tiles.
  int k0, k1;
  if (SELECT) {
    if (threadIdx.x < GEMM_MAX_SELECT / 32) sel_bits[threadIdx.x] = 0u;
    __syncthreads();
    griddep_wait();
    for (int i = (int)threadIdx.x; i < a.keep_div; i += GR_THREADS) {
      const int e = *reinterpret_cast<const volatile int *>(a.group_tab + i);
      if (e >= 0) atomicOr(&sel_bits[e >> 5], 1u << (e & 31));
    }
    __syncthreads();
    if (warp == 0) {
      int n = 0;
      for (int w = 0; w < GEMM_MAX_SELECT / 32; ++w) {
        const uint32_t m = sel_bits[w];
        if ((m >> lane) & 1u) sel_list[n + __popc(m & ((1u << lane) - 1u))] = (unsigned short)(w * 32 + lane);
        n += __popc(m);
      }
      if (lane == 0) sel_n = n;
    }
    __syncthreads();
    const int used = sel_n * a.tiles_per_group;
    k0 = 0;
    k1 = cta < used ? (used - cta + (int)gridDim.x - 1) / (int)gridDim.x * KB : 0;
  } else if (GROUPED) {
    if (a.keep_div >= 0) griddep_wait();            // the group table comes from an earlier kernel (keep_div < 0: it is fixed)
    const int used = min(*reinterpret_cast<const volatile int *>(a.group_tab + 3 * a.keep_pitch), a.keep_pitch) * a.tiles_per_group;
    k0 = 0;
    k1 = cta < used ? (used - cta + (int)gridDim.x - 1) / (int)gridDim.x * KB : 0;
  } else {
    k0 = a.cta_start[cta];
    k1 = a.cta_start[cta + 1];
  }
  int fail = 0;

  if (warp == 0) {
    if (elect_one()) {
      // ---------------- TMA producer ----------------
      const uint64_t pol_w = l2_policy_evict_first();   // weights are streamed once per step
      const uint64_t pol_x = l2_policy_evict_last();    // activations are re-read by every CTA
      auto load_w = [&](uint32_t dst, int tile, int kb, uint32_t fb) {
        int row0, row1;                                 // first weight rows of the tile's blocks
        if (SWIGLU) {
          if (GROUPED) row0 = g_wrow + g_j * a.w_rows;
          else if (MASKED) row0 = tile / a.keep_div * 2 * sw_fb + tile % a.keep_div * a.w_rows;
          else row0 = tile * a.w_rows;
          row1 = row0 + sw_fb;
        } else {
          row0 = GROUPED ? g_wrow + g_j * a.tile_n : tile * a.tile_n;
          row1 = row0 + 128;
        }
        const int x = (GROUPED ? g_wk + kb : kb) * GEMM_BLOCK_K;
        tma_load_2d(dst, &tmW, x, row0, fb, pol_w);
        if (MT == 2) tma_load_2d(dst + w_box, &tmW, x, row1, fb, pol_w);
      };
      // hi rows, then lo rows: boxes of 64, 32 and 16 rows (128-byte rows; every box begins on a group of eight)
      auto load_x = [&](uint32_t dst, int kb, uint32_t fb) {
        const int x = kb * GEMM_BLOCK_K, y = GROUPED && !(SELECT && SWIGLU) ? g_id * BN : 0;   // (SELECT: every expert's gate / up reads the step's rows)
        const uint32_t lo = (uint32_t)n_pad * 128u;
        int r = 0;
        auto box = [&](int i, int rows) {
          tma_load_2d(dst + (uint32_t)r * 128u, &tmX.hi[i], x, y + r, fb, pol_x);
          tma_load_2d(dst + lo + (uint32_t)r * 128u, &tmX.lo[i], x, y + r, fb, pol_x);
          r += rows;
        };
        if (n_pad >= 64) box(0, 64);
        if (n_pad == 128) box(0, 64);
        if (n_pad & 32) box(1, 32);
        if (n_pad & 16) box(2, 16);
      };
      // The weights depend on no earlier kernel: fill the ring with weight tiles first, then wait for the predecessor (which
      // produces the activations) and add the activation tiles to the same barriers.
      const int n_pre = min(a.stages, k1 - k0);
      for (int it = 0; it < n_pre; ++it) {
        const int g = k0 + it, tile = g / KB, kb = g - tile * KB;
        look(tile);
        const uint32_t fb = smem_u32(&full_bar[it]);
        mbar_expect_tx(fb, w_bytes);                // the activations' bytes and the arrival follow behind the wait
        load_w(base + (uint32_t)it * a.stage_bytes, tile, kb, fb);
        if (it == 0) TRACE(2);
      }
      griddep_wait();
      read_rows();
      for (int it = 0; it < n_pre; ++it) {
        const int g = k0 + it, tile = g / KB, kb = g - tile * KB;
        look(tile);
        const uint32_t fb = smem_u32(&full_bar[it]);
        mbar_arrive_expect_tx(fb, (uint32_t)n_pad * 256u);
        load_x(base + (uint32_t)it * a.stage_bytes + w_bytes, kb, fb);
      }
      int s = n_pre == a.stages ? 0 : n_pre;
      uint32_t ph = n_pre == a.stages ? 0u : 1u;    // (the first release of a stage completes phase 0)
      for (int g = k0 + n_pre; g < k1; ++g) {
        const int tile = g / KB, kb = g - tile * KB;
        look(tile);
        if (!mbar_wait(smem_u32(&empty_bar[s]), ph, abort_p)) { fail = DEV_TIMEOUT_PRODUCER; break; }
        const uint32_t fb = smem_u32(&full_bar[s]), dst = base + (uint32_t)s * a.stage_bytes;
        mbar_arrive_expect_tx(fb, w_bytes + (uint32_t)n_pad * 256u);
        load_w(dst, tile, kb, fb);
        load_x(dst + w_bytes, kb, fb);
        if (++s == a.stages) { s = 0; ph ^= 1u; }
      }
      TRACE(3);
    }
  } else if (warp == 1) {
    if (elect_one()) {
      // ---------------- MMA issuer ----------------
      read_rows();
      Halves hv;
      int s = 0;
      uint32_t ph = 0;
      for (int g = k0; g < k1 && !fail;) {
        const int tile = g / KB, kb_begin = g - tile * KB;
        const int kb_end = min(KB, kb_begin + (k1 - g));
        look(tile);
        const bool both = wide_seg();
        const int half = both ? 0 : hv.next;
        for (int h = 0; h < 2 && !fail; ++h)
          if (both || h == half) {
            if (!mbar_wait(smem_u32(&tmem_empty_bar[h]), (hv.use[h] & 1u) ^ 1u, abort_p)) fail = DEV_TIMEOUT_MMA;
            ++hv.use[h];
          }
        if (fail) break;
        if (!both) hv.next ^= 1;
        tc_fence_after();
        // kind::f16: D fp32 (bits 4-5 = 1), A and B bf16 (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n_pad >> 2) << 17) | ((uint32_t)((m64 ? 64 : 128) >> 4) << 24);
        const uint32_t d0 = tmem_base + mt_col(half, 0), d1 = tmem_base + mt_col(half, 1);
        uint32_t more = 0;
        for (int kb = kb_begin; kb < kb_end; ++kb) {
          if (!mbar_wait(smem_u32(&full_bar[s]), ph, abort_p)) { fail = DEV_TIMEOUT_MMA; break; }
          if (g == k0 && kb == kb_begin) TRACE(4);
          tc_fence_after();
          const uint32_t st = base + (uint32_t)s * a.stage_bytes;
          const uint64_t w0 = umma_desc_sw128(st), w1 = umma_desc_sw128(st + w_box), x = umma_desc_sw128(st + w_bytes);
#pragma unroll
          for (int k = 0; k < GEMM_BLOCK_K / 16; ++k) {
            // advancing 16 bf16 = 32 bytes along K inside the swizzle row: +2 in 16-byte units
            const uint64_t adv = (uint64_t)(k * 2);
            umma_bf16(d0, w0 + adv, x + adv, idesc, more);
            if (MT == 2) umma_bf16(d1, w1 + adv, x + adv, idesc, more);
            more = 1u;
          }
          umma_commit(smem_u32(&empty_bar[s]));     // frees the stage once these MMAs have read it
          if (++s == a.stages) { s = 0; ph ^= 1u; }
        }
        if (fail) break;
        for (int h = 0; h < 2; ++h)
          if (both || h == half) umma_commit(smem_u32(&tmem_full_bar[h]));   // the accumulators of this segment are complete
        g += kb_end - kb_begin;
      }
      TRACE(5);
    }
  } else {
    // ---------------- epilogue: TMEM -> registers -> global ----------------
    // A warp reads the 32 lanes (weight rows) of its quarter; the two groups of four warps share the blocks, or the rows.
    const int lane_base = (warp & 3) * 32, grp = (warp - 2) >> 2;
    const uint32_t t_lane = tmem_base + ((uint32_t)lane_base << 16);
    read_rows();
    Halves hv;
    int seg = 0;
    for (int g = k0; g < k1; ++seg) {
      const int tile = g / KB, kb_begin = g - tile * KB;
      const int kb_end = min(KB, kb_begin + (k1 - g));
      const bool whole = (kb_begin == 0 && kb_end == KB);
      look(tile);
      const bool both = wide_seg();
      const int half = both ? 0 : hv.next;
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
      if (g + (kb_end - kb_begin) >= k1 && threadIdx.x == 64) TRACE(6);   // last accumulator is ready
      const int rows = GROUPED && !SELECT ? min(g_rows, n_pad) : min(a.R, n_pad), chunks = (rows + 7) >> 3;
      // which rows of a chunk of eight are stored, as bits (MASKED, SELECT: those with a weight)
      auto rows_on = [&](int c, int col) -> uint32_t {
        const int r = 8 * c + (lane & 7);
        bool on = r < rows;
        if (SELECT) on = on && a.row_keep[(size_t)r * a.keep_pitch + col] != 0.f;
        else if (MASKED && !SWIGLU) on = on && a.row_keep[(size_t)r * a.keep_pitch + col] != 0.f;
        return __ballot_sync(0xffffffffu, on) & 0xffu;
      };
      if (SWIGLU) {
        // this thread's output: gate sums in block 0, up sums in block 1, the same lane
        const int blk = MASKED ? tile / a.keep_div : 0;
        const int f0 = (GROUPED ? g_j : MASKED ? tile - blk * a.keep_div : tile) * a.w_rows;
        const int w0 = m64 ? lane_base / 2 : lane_base, f = f0 + w0 + lane, o_pitch = N / 2, col = blk * sw_fb + f;   // w0: this warp's first weight row
        // (F, the matrix and w_rows are multiples of 8: the same for both lanes of a pair)
        const bool f_ok = w0 + lane < a.w_rows && f < sw_fb && (!m64 || lane < 16);
        const int row0 = GROUPED ? g_id * BN : 0;
        const uint32_t tg = t_lane + mt_col(half, 0), tu = t_lane + mt_col(half, 1);
        if (w0 < a.w_rows) {
          for (int c = grp; c < chunks; c += 2) {
            uint32_t gh[8], gl[8], uh[8], ul[8];
            tmem_ld8(tg + (uint32_t)(8 * c), gh);
            tmem_ld8(tg + (uint32_t)(n_pad + 8 * c), gl);
            tmem_ld8(tu + (uint32_t)(8 * c), uh);
            tmem_ld8(tu + (uint32_t)(n_pad + 8 * c), ul);
            tmem_ld_wait();
            const uint32_t on = rows_on(c, g_id);
            float y[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float gt = __uint_as_float(gh[j]) + __uint_as_float(gl[j]), up = __uint_as_float(uh[j]) + __uint_as_float(ul[j]);
              y[j] = __fdividef(gt, 1.f + __expf(-gt)) * up;
              if (MASKED || GROUPED) {              // the row's routing weight for this expert; 0: not selected
                const int r = min(8 * c + j, rows - 1);
                const float w = SELECT ? a.row_keep[(size_t)r * a.keep_pitch + g_id]
                                       : GROUPED ? a.row_keep[row0 + r] : a.row_keep[(size_t)r * a.keep_pitch + blk];
                y[j] = w != 0.f ? w * y[j] : 0.f;
              }
            }
            // lanes in pairs: the even one stores two outputs of row 2 i, the odd one of row 2 i + 1
            const bool odd = lane & 1;
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
              const float got = __shfl_xor_sync(0xffffffffu, odd ? y[j] : y[j + 1], 1);
              const float y0 = odd ? got : y[j], y1 = odd ? y[j + 1] : got;
              const int r = j + (odd ? 1 : 0);
              const __nv_bfloat16 h0 = __float2bfloat16_rn(y0), h1 = __float2bfloat16_rn(y1);
              const __nv_bfloat162 hi = __halves2bfloat162(h0, h1),
                                   lo = __halves2bfloat162(__float2bfloat16_rn(y0 - __bfloat162float(h0)), __float2bfloat16_rn(y1 - __bfloat162float(h1)));
              if (f_ok && ((on >> r) & 1u)) {
                const size_t o = (size_t)(row0 + 8 * c + r) * o_pitch + (col & ~1);
                *reinterpret_cast<__nv_bfloat162 *>(a.sw_hi + o) = hi;
                *reinterpret_cast<__nv_bfloat162 *>(a.sw_lo + o) = lo;
              }
            }
          }
        }
      } else {
        const int n0 = GROUPED ? g_j * a.tile_n : tile * a.tile_n;
        const size_t pitch = whole ? (size_t)N : (size_t)a.tile_n;
        float *dst = GROUPED ? a.direct + (size_t)g_id * BN * N + n0
                             : whole ? a.direct + n0 : a.ws + (size_t)(cta * 2 + (seg == 0 ? 0 : 1)) * BN * a.tile_n;
        const int step = MT == 2 ? 1 : 2;           // two blocks: one per group of warps; one: every other chunk of rows
        for (int mt = MT == 2 ? grp : 0, c = MT == 2 ? 0 : grp; c < chunks; c += step) {
          const int at = mt * 128 + lane_base + lane;
          if (n0 + mt * 128 + lane_base >= N) break;   // columns beyond the matrix (last tile); warp-uniform
          const uint32_t ta = t_lane + mt_col(half, mt) + (uint32_t)(8 * c);
          uint32_t h[8], l[8];
          tmem_ld8(ta, h);
          tmem_ld8(ta + (uint32_t)n_pad, l);
          tmem_ld_wait();
          uint32_t on = rows_on(c, SELECT ? g_id : MASKED ? n0 / GEMM_TILE_N / a.keep_div : 0);
          if (n0 + at >= N) on = 0;
          float *d = dst + (size_t)(8 * c) * pitch + at;
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if ((on >> j) & 1u) d[(size_t)j * pitch] = __uint_as_float(h[j]) + __uint_as_float(l[j]);
        }
      }
      tc_fence_before();
      for (int h = 0; h < 2; ++h)
        if (both || h == half) mbar_arrive(smem_u32(&tmem_empty_bar[h]));
      g += kb_end - kb_begin;
    }
    if (threadIdx.x == 64) TRACE(7);
  }

  if (fail) {
    atomicCAS(a.status, 0, fail);
    // let copies that are still in flight land before the shared memory is given back
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, 512);
#undef TRACE
}

template <typename F>
cudaError_t each_kernel(F f) {
  cudaError_t e = f(gemm_rows_kernel<false, false, false, false>);
  if (e == cudaSuccess) e = f(gemm_rows_kernel<true, false, false, false>);
  if (e == cudaSuccess) e = f(gemm_rows_kernel<false, false, true, false>);
  if (e == cudaSuccess) e = f(gemm_rows_kernel<true, false, true, false>);
  if (e == cudaSuccess) e = f(gemm_rows_kernel<false, true, false, false>);
  if (e == cudaSuccess) e = f(gemm_rows_kernel<false, true, true, false>);
  if (e == cudaSuccess) e = f(gemm_rows_kernel<false, true, false, true>);
  if (e == cudaSuccess) e = f(gemm_rows_kernel<false, true, true, true>);
  return e;
}

}  // namespace

int gemm_rows_stages(GemmPlan *p) {
  const int mt = p->sw_half ? 2 : p->tile_n / 128, box = p->sw_half ? p->sw_half : 128;
  const size_t w = (size_t)mt * box * GEMM_BLOCK_K * 2;
  p->stage_bytes = (uint32_t)(w + (size_t)gemm_rows_padded(p->BN) * 256);
  // an MMA always reads 128 weight rows: what the last stage leaves behind the second block's rows must be readable
  const size_t over = GR_W_BYTES - (size_t)box * GEMM_BLOCK_K * 2, fixed = 1024 + over;
  int stages = (int)((GEMM_ROWS_MAX_SMEM - fixed) / p->stage_bytes);
  if (stages > GR_MAX_STAGES) stages = GR_MAX_STAGES;
  if (stages < 2) return CORUN_EINVAL;
  p->stages = stages;
  p->smem_bytes = fixed + (size_t)stages * p->stage_bytes;
  return CORUN_OK;
}

int gemm_encode_x(GemmXMaps *m, const void *Xhi, const void *Xlo, unsigned long long rows, int K) {
  static const int box[3] = {64, 32, 16};
  for (int i = 0; i < 3; ++i) {
    int rc;
    if ((rc = tma_encode_2d(&m->hi[i], Xhi, 0, rows, K, box[i], GEMM_BLOCK_K)) != 0) return rc;
    if ((rc = tma_encode_2d(&m->lo[i], Xlo, 0, rows, K, box[i], GEMM_BLOCK_K)) != 0) return rc;
  }
  return CORUN_OK;
}

cudaError_t gemm_rows_prepare() {
  return each_kernel([](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_ROWS_MAX_SMEM); });
}

cudaError_t gemm_rows_launch(const GemmPlan &p, const CUtensorMap *tmW_override, int *d_status, cudaStream_t st, unsigned long long *trace,
                             bool pdl) {
  const GemmRowsArgs a{p.direct, p.ws, p.d_cta_start, p.N, p.KB, p.BN, p.R, p.stages, p.tile_n, p.sw_half ? p.sw_half : 128, p.stage_bytes,
                       p.row_keep, p.keep_pitch, p.keep_div, p.group_tab, p.tiles_per_group, d_status, trace, p.sw_hi, p.sw_lo, p.row_blocks};
  auto go = [&](auto kernel) {
    return launch_k(kernel, dim3(p.grid), dim3(GR_THREADS), p.smem_bytes, st, pdl, tmW_override ? *tmW_override : p.tmW, p.tmX, a);
  };
  const bool masked = p.row_keep != nullptr;
  if (p.select) return p.sw_hi ? go(gemm_rows_kernel<false, true, true, true>) : go(gemm_rows_kernel<false, true, false, true>);
  if (p.group_tab) return p.sw_hi ? go(gemm_rows_kernel<false, true, true, false>) : go(gemm_rows_kernel<false, true, false, false>);
  if (p.sw_hi) return masked ? go(gemm_rows_kernel<true, false, true, false>) : go(gemm_rows_kernel<false, false, true, false>);
  return masked ? go(gemm_rows_kernel<true, false, false, false>) : go(gemm_rows_kernel<false, false, false, false>);
}

}  // namespace corun
