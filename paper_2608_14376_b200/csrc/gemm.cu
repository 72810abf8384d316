// tcgen05 / TMEM / TMA GEMM for sm_100a with a static, shape-keyed work partition.
#include "gemm.cuh"

#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdlib>
#include <vector>

#include "../../include/corun.h"
#include "launch.cuh"
#include "ptx.cuh"

namespace corun {

int g_last_cuda_error = 0;
bool g_use_pdl = !(getenv("CORUN_NO_PDL") && atoi(getenv("CORUN_NO_PDL")) != 0);

namespace {

constexpr int MAX_STAGES = 8;
constexpr int GEMM_MAX_DYN_SMEM = 209 * 1024;
constexpr uint32_t W_TILE_BYTES = GEMM_TILE_N * GEMM_BLOCK_K * 2;          // 32 KiB
constexpr uint32_t A_BLOCK_BYTES = GEMM_ROW_BLOCK * GEMM_BLOCK_K * 2;      // 16 KiB: what one MMA reads of A

// More than 128 rows (gemm_rows.cu has the kernel for fewer).  Role loops walk the CTA's flat k-block range [k0, k1) segment
// by segment; a segment is the part of the range that falls into one weight tile.
//
// Operands: A = activations (hi or lo), 128 rows per MMA, K-major, 128-byte
// swizzle; B = 256 weight rows, same layout; D = fp32 [128 rows x 256 weight
// rows] in TMEM (lane = activation row, column = weight row), one accumulator
// per block of 128 activation rows.
// MASKED: the optional store mask of the epilogue (a separate instantiation, so that the plain kernel is
// exactly the code it was without it).
// *row_blocks (bit b: rows 128 b .. hold active rows; written by an earlier kernel of the step, or null = both) says which
// blocks of 128 rows exist this step: an absent block is neither loaded nor multiplied nor stored (its output rows keep what
// they held: nobody reads rows without a request); with one block left its two accumulator buffers alternate.  A row's value
// does not depend on which blocks exist.
template <bool MASKED>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
gemm_streamk_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmHi,
                    const __grid_constant__ CUtensorMap tmLo, float *__restrict__ direct, float *__restrict__ ws,
                    const int *__restrict__ cta_start, int N, int KB, int BN, int R, int stages, uint32_t idesc,
                    const float *row_keep, int keep_pitch, int keep_div, int *status, unsigned long long *trace, const int *row_blocks) {
  extern __shared__ uint8_t smem_raw[];
  // optional per-CTA timeline (debug): 8 globaltimer stamps
#define TRACE(i) do { if (trace) trace[(size_t)blockIdx.x * 8 + (i)] = globaltimer_ns(); } while (0)
  if (threadIdx.x == 0) TRACE(0);
  griddep_launch_dependents();   // the next kernel may start its prologue
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t empty_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t tmem_full_bar[2];    // one pair per accumulator buffer
  __shared__ __align__(8) uint64_t tmem_empty_bar[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x;
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  // the hi tiles of both blocks (128 rows each, whatever BN is), then the lo tiles
  const uint32_t lo_off = 2u * A_BLOCK_BYTES;
  constexpr uint32_t stage_bytes = W_TILE_BYTES + 4u * A_BLOCK_BYTES;
  constexpr int n_rb = 2;                           // blocks of 128 activation rows
  int bmask = 3, n_acc = 1;
  uint32_t tx_bytes = 0;
  auto read_blocks = [&]() {
    if (row_blocks) { griddep_wait(); bmask = *reinterpret_cast<const volatile int *>(row_blocks) & 3; }
    if (bmask == 0) bmask = 1;                      // a step without requests: block 0 is computed and ignored
    n_acc = bmask == 3 ? 1 : 2;
    tx_bytes = W_TILE_BYTES + (uint32_t)__popc(bmask) * 2 * A_BLOCK_BYTES;
  };
  auto acc_col = [&](int acc, int b) { return (uint32_t)(n_acc == 2 ? acc : b) * GEMM_TILE_N; };

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < stages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tmem_full_bar[a]), 1);
      mbar_init(smem_u32(&tmem_empty_bar[a]), 128);
    }
    fence_mbar_init();
    fence_proxy_async();
    prefetch_tensormap(&tmW);
    prefetch_tensormap(&tmHi);
    prefetch_tensormap(&tmLo);
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
  const int k0 = cta_start[cta], k1 = cta_start[cta + 1];
  int fail = 0;

  if (warp == 0) {
    if (elect_one()) {
      // ---------------- TMA producer ----------------
      const uint64_t pol_w = l2_policy_evict_first();   // weights are streamed once per step
      const uint64_t pol_x = l2_policy_evict_last();    // activations are re-read by every CTA
      auto load_w = [&](uint32_t dst, int tile, int kb, uint32_t fb) {
        tma_load_2d(dst, &tmW, kb * GEMM_BLOCK_K, tile * GEMM_TILE_N, fb, pol_w);
        tma_load_2d(dst + W_TILE_BYTES / 2, &tmW, kb * GEMM_BLOCK_K, tile * GEMM_TILE_N + GEMM_W_BOX, fb, pol_w);
      };
      // The weights depend on no earlier kernel: fill the ring with weight tiles first, then wait for
      // the predecessor (which produces the activations) and add the activation tiles to the same
      // barriers.
      const int n_pre = min(stages, k1 - k0);
      for (int it = 0; it < n_pre; ++it) {
        const int g = k0 + it, tile = g / KB, kb = g - tile * KB;
        const uint32_t fb = smem_u32(&full_bar[it]);
        mbar_expect_tx(fb, W_TILE_BYTES);           // the activations' bytes and the arrival follow behind the wait
        load_w(tiles_base + (uint32_t)it * stage_bytes, tile, kb, fb);
        if (it == 0) TRACE(2);
      }
      griddep_wait();
      read_blocks();
      auto load_x = [&](uint32_t dst, int kb, uint32_t fb) {
#pragma unroll
        for (int b = 0; b < 2; ++b)
          if ((bmask >> b) & 1) {
            tma_load_2d(dst + W_TILE_BYTES + (uint32_t)b * A_BLOCK_BYTES, &tmHi, kb * GEMM_BLOCK_K, GEMM_ROW_BLOCK * b, fb, pol_x);
            tma_load_2d(dst + W_TILE_BYTES + lo_off + (uint32_t)b * A_BLOCK_BYTES, &tmLo, kb * GEMM_BLOCK_K, GEMM_ROW_BLOCK * b, fb, pol_x);
          }
      };
      for (int it = 0; it < n_pre; ++it) {
        const int g = k0 + it, kb = g % KB;
        const uint32_t fb = smem_u32(&full_bar[it]);
        mbar_arrive_expect_tx(fb, tx_bytes - W_TILE_BYTES);
        load_x(tiles_base + (uint32_t)it * stage_bytes, kb, fb);
      }
      int it = n_pre;
      for (int g = k0 + n_pre; g < k1; ++g, ++it) {
        const int tile = g / KB, kb = g - tile * KB;
        const int s = it % stages;
        const uint32_t ph = (uint32_t)(it / stages) & 1u;
        if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1u, abort_p)) { fail = DEV_TIMEOUT_PRODUCER; break; }
        const uint32_t fb = smem_u32(&full_bar[s]);
        const uint32_t dst = tiles_base + (uint32_t)s * stage_bytes;
        mbar_arrive_expect_tx(fb, tx_bytes);
        load_w(dst, tile, kb, fb);
        load_x(dst, kb, fb);
      }
      TRACE(3);
    }
  } else if (warp == 1) {
    if (elect_one()) {
      // ---------------- MMA issuer ----------------
      read_blocks();
      int it = 0, seg = 0;
      for (int g = k0; g < k1 && !fail; ++seg) {
        const int tile = g / KB, kb_begin = g - tile * KB;
        const int kb_end = min(KB, kb_begin + (k1 - g));
        const int acc = seg % n_acc;
        const uint32_t use = (uint32_t)(seg / n_acc);     // how often this buffer has been used before
        if (!mbar_wait(smem_u32(&tmem_empty_bar[acc]), (use & 1u) ^ 1u, abort_p)) { fail = DEV_TIMEOUT_MMA; break; }
        tc_fence_after();
        for (int kb = kb_begin; kb < kb_end; ++kb, ++it) {
          const int s = it % stages;
          const uint32_t ph = (uint32_t)(it / stages) & 1u;
          if (!mbar_wait(smem_u32(&full_bar[s]), ph, abort_p)) { fail = DEV_TIMEOUT_MMA; break; }
          if (it == 0) TRACE(4);
          tc_fence_after();
          const uint32_t w_addr = tiles_base + (uint32_t)s * stage_bytes;
          const uint64_t w_desc = umma_desc_sw128(w_addr);
          for (int rb = 0; rb < n_rb; ++rb) {
            if (!((bmask >> rb) & 1)) continue;
            const uint64_t hi_desc = umma_desc_sw128(w_addr + W_TILE_BYTES + (uint32_t)rb * A_BLOCK_BYTES);
            const uint64_t lo_desc = umma_desc_sw128(w_addr + W_TILE_BYTES + lo_off + (uint32_t)rb * A_BLOCK_BYTES);
            const uint32_t d_tmem = tmem_base + acc_col(acc, rb);
#pragma unroll
            for (int k = 0; k < GEMM_BLOCK_K / 16; ++k) {
              // advancing 16 bf16 = 32 bytes along K inside the swizzle row: +2 in 16-byte units
              const uint64_t adv = (uint64_t)(k * 2);
              umma_bf16(d_tmem, hi_desc + adv, w_desc + adv, idesc, (kb > kb_begin || k > 0) ? 1u : 0u);
              umma_bf16(d_tmem, lo_desc + adv, w_desc + adv, idesc, 1u);
            }
          }
          umma_commit(smem_u32(&empty_bar[s]));   // frees the stage once these MMAs have read it
        }
        if (fail) break;
        umma_commit(smem_u32(&tmem_full_bar[acc]));    // accumulators of this segment are complete
        g += kb_end - kb_begin;
      }
      TRACE(5);
    }
  } else {
    // ---------------- epilogue: TMEM -> registers -> global ----------------
    const int lane_base = (warp & 3) * 32;          // the TMEM lanes this warp may read
    read_blocks();
    int seg = 0;
    for (int g = k0; g < k1; ++seg) {
      const int tile = g / KB, kb_begin = g - tile * KB;
      const int kb_end = min(KB, kb_begin + (k1 - g));
      const bool whole = (kb_begin == 0 && kb_end == KB);
      const int acc = seg % n_acc;
      const uint32_t use = (uint32_t)(seg / n_acc);
      bool ok = mbar_wait(smem_u32(&tmem_full_bar[acc]), use & 1u, abort_p);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { fail = DEV_TIMEOUT_EPILOGUE; break; }
      tc_fence_after();
      if (g + (kb_end - kb_begin) >= k1 && threadIdx.x == 64) TRACE(6);   // last accumulator is ready
      const int n0 = tile * GEMM_TILE_N;
      // optional: rows whose entry for this tile's column group is zero are not stored (nobody reads them)
      const float *keep = MASKED ? row_keep + tile / keep_div : nullptr;
      for (int rb = 0; rb < n_rb; ++rb) {
        if (!((bmask >> rb) & 1)) continue;
        const int row_base = rb * GEMM_ROW_BLOCK + lane_base;
        const int rows_valid = whole ? R : BN;      // partials keep the padded row count
        if (row_base >= rows_valid) continue;        // warp-uniform: nothing of this warp's lanes is needed
        const int row = row_base + lane;
        const bool row_ok = row < rows_valid && (!MASKED || row >= R || keep[(size_t)row * keep_pitch] != 0.f);
        float *dst = whole ? direct + (size_t)row * N + n0
                           : ws + ((size_t)(cta * 2 + (seg == 0 ? 0 : 1)) * BN + row) * GEMM_TILE_N;
        const bool vec_ok = whole ? ((N & 3) == 0) : true;
        for (int c0 = 0; c0 < GEMM_TILE_N; c0 += 16) {
          if (whole && n0 + c0 >= N) break;          // columns beyond the matrix (last tile)
          uint32_t v[16];
          tmem_ld16(tmem_base + ((uint32_t)lane_base << 16) + acc_col(acc, rb) + (uint32_t)c0, v);
          tmem_ld_wait();
          if (!row_ok) continue;
          if (vec_ok && (!whole || n0 + c0 + 16 <= N)) {
#pragma unroll
            for (int j = 0; j < 16; j += 4)
              *reinterpret_cast<float4 *>(dst + c0 + j) =
                  make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]), __uint_as_float(v[j + 2]),
                              __uint_as_float(v[j + 3]));
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (n0 + c0 + j < N) dst[c0 + j] = __uint_as_float(v[j]);
          }
        }
      }
      tc_fence_before();
      mbar_arrive(smem_u32(&tmem_empty_bar[acc]));
      g += kb_end - kb_begin;
    }
    if (threadIdx.x == 64) TRACE(7);
  }

  if (fail) {
    atomicCAS(status, 0, fail);
    // let copies that are still in flight land before the shared memory is given back
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

// Split tiles of the rows there are, 16 bytes per thread, up to FIXUP_SHARES blocks per tile.  Bound by its blocks' launches: with a
// block per tile and row (295 tiles, 128 rows of the DeepSeek-V2-Lite LM head) 31 us.  The LM head with it, with up to 1 / 2 / 4 / 8 / 16
// blocks per tile: those 128 rows 131.7 / 124.7 / 118.3 / 119.0 / 118.3 us, 40 rows of Qwen3-8B (vocabulary 151936) 208.1 / 205.9 / 203.9 /
// 205.0 / 205.7.
constexpr int FIXUP_THREADS = 256, FIXUP_SHARES = 4;
__global__ void __launch_bounds__(FIXUP_THREADS) gemm_fixup_kernel(GemmOut g, float *direct, const int *split_tiles, int rows, const int *row_blocks) {
  griddep_launch_dependents();
  griddep_wait();
  if (row_blocks) {
    const int n = *reinterpret_cast<const volatile int *>(row_blocks) >> 8;
    if (n > 0 && n < rows) rows = n;
  }
  const int lg = g.tile_shift - 2, t = split_tiles[blockIdx.x], n = (t << g.tile_shift) + 4 * ((int)threadIdx.x & ((1 << lg) - 1));
  for (int r = (int)blockIdx.y * (FIXUP_THREADS >> lg) + ((int)threadIdx.x >> lg); r < rows; r += (int)gridDim.y * (FIXUP_THREADS >> lg)) {
    if ((g.N & 3) == 0) {
      if (n < g.N) *reinterpret_cast<float4 *>(direct + (size_t)r * g.N + n) = gemm_load4(g, r, n);
    } else {
      for (int k = 0; k < 4; ++k)
        if (n + k < g.N) direct[(size_t)r * g.N + n + k] = gemm_load(g, r, n + k);
    }
  }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}

}  // namespace

int tma_encode_2d(CUtensorMap *m, const void *base, int is_fp16, unsigned long long rows, int cols, int box_rows,
                  int box_cols) {
  auto enc = get_encode();
  if (!enc) { g_last_cuda_error = 99999; return CORUN_ECUDA; }
  if (((uintptr_t)base & 15u) || (cols % 8) || (box_cols * 2 != 128 && box_cols * 2 != 32) || box_rows > 256 || box_rows < 1)
    return CORUN_EINVAL;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, is_fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                   const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   box_cols * 2 == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) g_last_cuda_error = 100000 + (int)r;
  return r == CUDA_SUCCESS ? CORUN_OK : CORUN_ECUDA;
}

int tma_encode_store_2d(CUtensorMap *m, const void *base, int is_fp32, unsigned long long rows, int cols) {
  auto enc = get_encode();
  if (!enc) { g_last_cuda_error = 99999; return CORUN_ECUDA; }
  const int eb = is_fp32 ? 4 : 2;
  if (((uintptr_t)base & 15u) || (cols * eb) % 16 || rows < 1) return CORUN_EINVAL;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * eb};
  cuuint32_t box[2] = {32, 32};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, is_fp32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims,
                   strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, is_fp32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_NONE,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) g_last_cuda_error = 100000 + (int)r;
  return r == CUDA_SUCCESS ? CORUN_OK : CORUN_ECUDA;
}

int tma_encode_fp16_nd(CUtensorMap *m, const void *base, int nd, const unsigned long long *dims, const unsigned long long *strides,
                       const unsigned *box) {
  auto enc = get_encode();
  if (!enc) { g_last_cuda_error = 99999; return CORUN_ECUDA; }
  if (nd < 2 || nd > 5 || ((uintptr_t)base & 15u) || box[0] * 2 != 128) return CORUN_EINVAL;
  cuuint64_t d[5], s[4];
  cuuint32_t b[5], estr[5] = {1, 1, 1, 1, 1};
  for (int i = 0; i < nd; ++i) {
    if (dims[i] < 1 || box[i] < 1 || box[i] > 256) return CORUN_EINVAL;
    d[i] = dims[i];
    b[i] = box[i];
  }
  for (int i = 0; i < nd - 1; ++i) {
    if (strides[i] % 16) return CORUN_EINVAL;
    s[i] = strides[i];
  }
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, (cuuint32_t)nd, const_cast<void *>(base), d, s, b, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) g_last_cuda_error = 100000 + (int)r;
  return r == CUDA_SUCCESS ? CORUN_OK : CORUN_ECUDA;
}

int tma_encode_fp16_4d(CUtensorMap *m, const void *base, const unsigned long long dims[4], const unsigned long long strides[3],
                       const unsigned box[4]) {
  return tma_encode_fp16_nd(m, base, 4, dims, strides, box);
}

int gemm_encode_map(CUtensorMap *m, const void *base, int rows, int K, int box_rows) {
  if (K % GEMM_BLOCK_K) return CORUN_EINVAL;
  return tma_encode_2d(m, base, 0, (unsigned long long)rows, K, box_rows, GEMM_BLOCK_K);
}

// The activations' tensor maps and the ring of a plan whose N, K, BN, tile_n and sw_half are set: x_rows rows of hi and lo.
static int plan_operands(GemmPlan *p, const void *Xhi, const void *Xlo, unsigned long long x_rows) {
  int rc;
  if (p->BN <= GEMM_MAX_ROWS) {
    if ((rc = gemm_rows_stages(p)) != 0) return rc;
    return gemm_encode_x(&p->tmX, Xhi, Xlo, x_rows, p->K);
  }
  const size_t stage = W_TILE_BYTES + 4 * (size_t)A_BLOCK_BYTES;
  const int stages = (int)((GEMM_MAX_DYN_SMEM - 1024) / stage);
  p->stages = stages < MAX_STAGES ? stages : MAX_STAGES;
  if (p->stages < 2) return CORUN_EINVAL;
  p->smem_bytes = stage * p->stages + 1024;
  // kind::f16 instruction descriptor: D fp32 (bits 4-5 = 1), A and B bf16 (bits 7-9, 10-12 = 1),
  // both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28.
  p->idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GEMM_TILE_N >> 3) << 17) | ((uint32_t)(GEMM_ROW_BLOCK >> 4) << 24);
  if ((rc = gemm_encode_map(&p->tmX.hi[0], Xhi, (int)x_rows, p->K, GEMM_ROW_BLOCK)) != 0) return rc;
  return gemm_encode_map(&p->tmX.lo[0], Xlo, (int)x_rows, p->K, GEMM_ROW_BLOCK);
}

int gemm_plan_fill(GemmPlan *p, const void *W, int N, int K, const void *Xhi, const void *Xlo, int R, int BN,
                   float *direct, float *ws, int num_sms, int *tab, int tab_cap, int *tab_ints) {
  if (N <= 0 || K <= 0 || K % GEMM_BLOCK_K || BN % 16 || BN < 16 || BN > 256 || R < 1 || R > BN) return CORUN_EINVAL;
  p->N = N; p->K = K; p->R = R; p->BN = BN;
  p->KB = K / GEMM_BLOCK_K;
  // With several CTAs per tile the ranges are cut tile by tile (the same number of CTAs for every tile, a few
  // SMs left out): no CTA then crosses a tile boundary, so none has two epilogues in a row, and above 128
  // rows -- where the two row blocks of a tile fill TMEM and the epilogue of a segment cannot overlap the MMAs
  // of the next -- none stops in the middle of its range.
  // At least four k-blocks per CTA: with fewer, the consumer's extra partials cost more than the shorter stream saves.
  struct Cut { int tile_n, n_tiles, grid, per_tile; };
  auto cut = [&](int tile_n) {
    Cut c{tile_n, (N + tile_n - 1) / tile_n, 0, 0};
    const long long total = (long long)c.n_tiles * p->KB;
    c.grid = (int)(total < num_sms ? total : num_sms);
    c.per_tile = c.grid >= 2 * c.n_tiles ? c.grid / c.n_tiles : 0;
    if (c.per_tile > 2 && c.per_tile > (p->KB + 3) / 4) c.per_tile = p->KB > 8 ? (p->KB + 3) / 4 : 2;
    if (c.per_tile) c.grid = c.per_tile * c.n_tiles;
    return c;
  };
  // Up to GEMM_NARROW_ROWS rows a tile is half as wide where a CTA's share of K does not grow with it: whole tiles, and matrices so small
  // that the four k-blocks bound it, which twice the CTAs then stream (a step of one row of a decoder of width 1024 483 us, 489 in wide
  // tiles).  Elsewhere half as many CTAs would share a tile's K and an accumulator sum twice the k-blocks, and it cuts every sum off
  // (gemm_pair.cu): sums of positive products of 6144 x 4096 / 4096 x 12288 2.5e-6 / 7.9e-6 off 64 bits instead of 9.9e-7 / 2.5e-6.  Nor is
  // that faster: 8 rows of Qwen3-8B's QKV, O and down 11.15 / 9.4 / 18.65 us in narrow tiles, 9.85 / 8.05 / 16.95 in wide ones.
  const Cut wide = cut(GEMM_TILE_N), narrow = cut(GEMM_TILE_N / 2);
  auto share = [&](const Cut &c) { return std::min((double)p->KB, c.per_tile ? (double)p->KB / c.per_tile : (double)c.n_tiles * p->KB / c.grid); };
  const Cut own = BN <= GEMM_NARROW_ROWS && share(narrow) <= share(wide) ? narrow : wide;
  p->tile_n = own.tile_n;
  p->n_tiles = own.n_tiles;
  p->grid = own.grid;
  const int per_tile = own.per_tile;
  const long long total = (long long)p->n_tiles * p->KB;
  if (total * (long long)p->grid >= (1ll << 31)) return CORUN_EINVAL;
  p->direct = direct;
  p->ws = ws;
  int rc;
  if ((rc = gemm_encode_map(&p->tmW, W, N, K, GEMM_W_BOX)) != 0) return rc;
  if ((rc = plan_operands(p, Xhi, Xlo, BN)) != 0) return rc;

  const int n_ints = p->grid + 1 + 3 * p->n_tiles;
  if (n_ints > tab_cap) return CORUN_ELIMIT;
  int *cs = tab, *cb = cs + p->grid + 1, *ce = cb + p->n_tiles, *sp = ce + p->n_tiles;
  for (int c = 0; c <= p->grid; ++c)
    cs[c] = per_tile ? (c / per_tile) * p->KB + (int)((long long)(c % per_tile) * p->KB / per_tile)
                     : (int)((long long)c * total / p->grid);
  p->n_split_tiles = 0;
  for (int t = 0, c = 0; t < p->n_tiles; ++t) {
    const int first = t * p->KB, last = first + p->KB - 1;
    while (cs[c + 1] <= first) ++c;
    cb[t] = 2 * c + (cs[c] < first ? 1 : 0);   // a CTA that began before the tile wrote its second slot
    int d = c;
    while (cs[d + 1] <= last) ++d;
    ce[t] = d;
    if (c != d) sp[p->n_split_tiles++] = t;
  }
  *tab_ints = n_ints;
  return CORUN_OK;
}

void gemm_plan_bind_tables(GemmPlan *p, int *d_tab) {
  p->d_cta_start = d_tab;
  p->d_tile_first = d_tab + p->grid + 1;
  p->d_tile_cend = p->d_tile_first + p->n_tiles;
  p->d_split_tiles = p->d_tile_cend + p->n_tiles;
}

int gemm_plan_create(GemmPlan *p, const void *W, int N, int K, const void *Xhi, const void *Xlo, int R, int BN,
                     float *direct, float *ws, int num_sms) {
  if (N <= 0 || K <= 0 || K % GEMM_BLOCK_K) return CORUN_EINVAL;
  const int n_tiles = (N + GEMM_TILE_N / 2 - 1) / (GEMM_TILE_N / 2);   // (of the narrower tiles)
  std::vector<int> tab((size_t)num_sms + 1 + 3 * (size_t)n_tiles);
  int n_ints = 0;
  int rc = gemm_plan_fill(p, W, N, K, Xhi, Xlo, R, BN, direct, ws, num_sms, tab.data(), (int)tab.size(), &n_ints);
  if (rc != CORUN_OK) return rc;
  int *d_tab = nullptr;
  if (cudaMalloc(&d_tab, (size_t)n_ints * sizeof(int)) != cudaSuccess) return CORUN_ENOMEM;
  cudaError_t me = cudaMemcpy(d_tab, tab.data(), (size_t)n_ints * sizeof(int), cudaMemcpyHostToDevice);
  if (me != cudaSuccess) { g_last_cuda_error = (int)me; cudaFree(d_tab); return CORUN_ECUDA; }
  gemm_plan_bind_tables(p, d_tab);
  cudaError_t ae = gemm_prepare_kernel();
  if (ae != cudaSuccess) { g_last_cuda_error = (int)ae; return CORUN_ECUDA; }
  return CORUN_OK;
}

int gemm_swiglu_half(int F, int num_sms) {
  int half = ((F + num_sms - 1) / num_sms + 7) / 8 * 8;
  if (half < 64) half = 64;
  if (half > GEMM_TILE_N / 2) half = GEMM_TILE_N / 2;
  return half;
}

int gemm_plan_create_swiglu(GemmPlan *p, const void *W, int F, int K, const void *Xhi, const void *Xlo, int R, int BN,
                            __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, int num_sms) {
  if (F <= 0 || F % 8 || K <= 0 || K % GEMM_BLOCK_K || BN % 16 || BN < 16 || BN > GEMM_MAX_ROWS || R < 1 || R > BN || !out_hi || !out_lo ||
      num_sms < 1)
    return CORUN_EINVAL;
  // as many whole tiles as there are SMs, if the matrix is large enough: the narrowest tile (a multiple of 8 gate
  // rows, at least 64) that still gives every CTA at most one
  const int HALF = gemm_swiglu_half(F, num_sms);
  p->sw_half = HALF;
  p->N = 2 * F; p->K = K; p->R = R; p->BN = BN;
  p->n_tiles = (F + HALF - 1) / HALF;
  p->KB = K / GEMM_BLOCK_K;
  p->grid = p->n_tiles < num_sms ? p->n_tiles : num_sms;
  if ((long long)p->n_tiles * p->KB >= (1ll << 31)) return CORUN_EINVAL;
  p->direct = nullptr;
  p->ws = nullptr;
  p->sw_hi = out_hi;
  p->sw_lo = out_lo;
  int rc;
  if ((rc = gemm_encode_map(&p->tmW, W, 2 * F, K, HALF)) != 0) return rc;
  if ((rc = plan_operands(p, Xhi, Xlo, BN)) != 0) return rc;
  // whole tiles only: CTA c takes tiles [c * n_tiles / grid, (c + 1) * n_tiles / grid)
  std::vector<int> tab((size_t)p->grid + 1);
  for (int c = 0; c <= p->grid; ++c) tab[(size_t)c] = (int)((long long)c * p->n_tiles / p->grid) * p->KB;
  int *d_tab = nullptr;
  if (cudaMalloc(&d_tab, tab.size() * sizeof(int)) != cudaSuccess) return CORUN_ENOMEM;
  cudaError_t me = cudaMemcpy(d_tab, tab.data(), tab.size() * sizeof(int), cudaMemcpyHostToDevice);
  if (me != cudaSuccess) { g_last_cuda_error = (int)me; cudaFree(d_tab); return CORUN_ECUDA; }
  p->d_cta_start = d_tab;
  p->d_tile_first = p->d_tile_cend = p->d_split_tiles = nullptr;
  p->n_split_tiles = 0;
  cudaError_t ae = gemm_prepare_kernel();
  if (ae != cudaSuccess) { g_last_cuda_error = (int)ae; return CORUN_ECUDA; }
  return CORUN_OK;
}

int gemm_swiglu_blocks_half(int Fb, int n_blocks, int num_sms) {
  // the widest tile (a multiple of 8 gate rows that divides Fb, 64..128) for which the busiest CTA streams the
  // fewest weight rows; wider tiles mean fewer MMA instructions per byte, so ties go to the wider one
  int best = 0;
  long long best_cost = 0;
  for (int half = GEMM_TILE_N / 2; half >= 64; half -= 8) {
    if (Fb % half) continue;
    const long long tiles = (long long)n_blocks * (Fb / half);
    const long long cost = (tiles + num_sms - 1) / num_sms * half;
    if (!best || cost < best_cost) { best = half; best_cost = cost; }
  }
  return best;
}

int gemm_plan_create_swiglu_blocks(GemmPlan *p, const void *W, int n_blocks, int Fb, int K, const void *Xhi, const void *Xlo,
                                   int R, int BN, __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, const float *row_scale,
                                   int num_sms) {
  if (n_blocks < 1 || Fb <= 0 || Fb % 8 || K <= 0 || K % GEMM_BLOCK_K || BN % 16 || BN < 16 || BN > GEMM_MAX_ROWS || R < 1 || R > BN ||
      !out_hi || !out_lo || !row_scale || num_sms < 1)
    return CORUN_EINVAL;
  const int HALF = gemm_swiglu_blocks_half(Fb, n_blocks, num_sms);
  if (!HALF) return CORUN_EINVAL;
  p->sw_half = HALF;
  p->N = n_blocks * 2 * Fb; p->K = K; p->R = R; p->BN = BN;
  p->n_tiles = n_blocks * (Fb / HALF);
  p->KB = K / GEMM_BLOCK_K;
  p->grid = p->n_tiles < num_sms ? p->n_tiles : num_sms;
  if ((long long)p->n_tiles * p->KB >= (1ll << 31)) return CORUN_EINVAL;
  p->direct = nullptr;
  p->ws = nullptr;
  p->sw_hi = out_hi;
  p->sw_lo = out_lo;
  p->row_keep = row_scale;
  p->keep_pitch = n_blocks;
  p->keep_div = Fb / HALF;
  int rc;
  if ((rc = gemm_encode_map(&p->tmW, W, n_blocks * 2 * Fb, K, HALF)) != 0) return rc;
  if ((rc = plan_operands(p, Xhi, Xlo, BN)) != 0) return rc;
  // whole tiles only: CTA c takes tiles [c * n_tiles / grid, (c + 1) * n_tiles / grid)
  std::vector<int> tab((size_t)p->grid + 1);
  for (int c = 0; c <= p->grid; ++c) tab[(size_t)c] = (int)((long long)c * p->n_tiles / p->grid) * p->KB;
  int *d_tab = nullptr;
  if (cudaMalloc(&d_tab, tab.size() * sizeof(int)) != cudaSuccess) return CORUN_ENOMEM;
  cudaError_t me = cudaMemcpy(d_tab, tab.data(), tab.size() * sizeof(int), cudaMemcpyHostToDevice);
  if (me != cudaSuccess) { g_last_cuda_error = (int)me; cudaFree(d_tab); return CORUN_ECUDA; }
  p->d_cta_start = d_tab;
  p->d_tile_first = p->d_tile_cend = p->d_split_tiles = nullptr;
  p->n_split_tiles = 0;
  cudaError_t ae = gemm_prepare_kernel();
  if (ae != cudaSuccess) { g_last_cuda_error = (int)ae; return CORUN_ECUDA; }
  return CORUN_OK;
}

int gemm_plan_create_grouped(GemmPlan *p, const void *W, long long w_rows, int w_cols, int N, int K, const void *Xhi,
                             const void *Xlo, int n_groups, int BN, float *direct, const int *group_tab, int num_sms) {
  if (N <= 0 || N % GEMM_TILE_N || K <= 0 || K % GEMM_BLOCK_K || w_cols % GEMM_BLOCK_K || BN % 16 || BN < 16 || BN > GEMM_MAX_ROWS ||
      n_groups < 1 || !group_tab || w_rows < N || num_sms < 1)
    return CORUN_EINVAL;
  p->N = N; p->K = K; p->R = BN; p->BN = BN;
  p->n_tiles = n_groups * (N / GEMM_TILE_N);
  p->KB = K / GEMM_BLOCK_K;
  p->grid = p->n_tiles < num_sms ? p->n_tiles : num_sms;
  p->keep_pitch = n_groups;                         // where the table's count of groups in use sits
  p->direct = direct;
  p->ws = nullptr;
  p->group_tab = group_tab;
  p->tiles_per_group = N / GEMM_TILE_N;
  int rc;
  if ((rc = tma_encode_2d(&p->tmW, W, 0, (unsigned long long)w_rows, w_cols, GEMM_W_BOX, GEMM_BLOCK_K)) != 0) return rc;
  if ((rc = plan_operands(p, Xhi, Xlo, (unsigned long long)n_groups * BN)) != 0) return rc;
  p->d_cta_start = p->d_tile_first = p->d_tile_cend = p->d_split_tiles = nullptr;   // the kernel derives its tiles itself
  p->n_split_tiles = 0;
  cudaError_t ae = gemm_prepare_kernel();
  if (ae != cudaSuccess) { g_last_cuda_error = (int)ae; return CORUN_ECUDA; }
  return CORUN_OK;
}

int gemm_plan_create_grouped_swiglu(GemmPlan *p, const void *W, long long w_rows, int F, int K, int half, const void *Xhi,
                                    const void *Xlo, int n_groups, int BN, __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo,
                                    const float *row_scale, const int *group_tab, int num_sms) {
  if (F <= 0 || half < 64 || half > GEMM_TILE_N / 2 || half % 8 || F % half || K <= 0 || K % GEMM_BLOCK_K || BN % 16 || BN < 16 ||
      BN > GEMM_MAX_ROWS || n_groups < 1 || !group_tab || !out_hi || !out_lo || !row_scale || w_rows < 2 * F || num_sms < 1)
    return CORUN_EINVAL;
  p->sw_half = half;
  p->N = 2 * F; p->K = K; p->R = BN; p->BN = BN;
  p->tiles_per_group = F / half;
  p->n_tiles = n_groups * p->tiles_per_group;
  p->KB = K / GEMM_BLOCK_K;
  p->grid = p->n_tiles < num_sms ? p->n_tiles : num_sms;
  p->keep_pitch = n_groups;
  p->direct = nullptr;
  p->ws = nullptr;
  p->sw_hi = out_hi;
  p->sw_lo = out_lo;
  p->row_keep = row_scale;
  p->group_tab = group_tab;
  int rc;
  if ((rc = tma_encode_2d(&p->tmW, W, 0, (unsigned long long)w_rows, K, half, GEMM_BLOCK_K)) != 0) return rc;
  if ((rc = plan_operands(p, Xhi, Xlo, (unsigned long long)n_groups * BN)) != 0) return rc;
  p->d_cta_start = p->d_tile_first = p->d_tile_cend = p->d_split_tiles = nullptr;   // the kernel derives its tiles itself
  p->n_split_tiles = 0;
  cudaError_t ae = gemm_prepare_kernel();
  if (ae != cudaSuccess) { g_last_cuda_error = (int)ae; return CORUN_ECUDA; }
  return CORUN_OK;
}

int gemm_plan_create_select_up(GemmPlan *p, const void *W, int NB, int F, int K, int half, const void *Xhi, const void *Xlo, int R, int BN,
                               __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, const float *w, const int *sel, int n_sel, int num_sms) {
  if (NB > GEMM_MAX_SELECT) return CORUN_EINVAL;
  int rc = gemm_plan_create_grouped_swiglu(p, W, (long long)NB * 2 * F, F, K, half, Xhi, Xlo, NB, BN, out_hi, out_lo, w, sel, num_sms);
  if (rc) return rc;
  p->R = R; p->keep_pitch = NB; p->keep_div = n_sel; p->select = true;
  return gemm_encode_x(&p->tmX, Xhi, Xlo, (unsigned long long)BN, K);   // one set of rows
}

int gemm_plan_create_select_down(GemmPlan *p, const void *W, int NB, int N, int F, const void *Xhi, const void *Xlo, int R, int BN,
                                 float *direct, const float *w, const int *sel, int n_sel, int num_sms) {
  if (NB > GEMM_MAX_SELECT) return CORUN_EINVAL;
  const int rc = gemm_plan_create_grouped(p, W, N, NB * F, N, F, Xhi, Xlo, NB, BN, direct, sel, num_sms);
  if (rc) return rc;
  p->R = R; p->row_keep = w; p->keep_pitch = NB; p->keep_div = n_sel; p->select = true;
  return CORUN_OK;
}

cudaError_t gemm_prepare_kernel() {
  cudaError_t e = gemm_rows_prepare();
  for (auto kernel : {gemm_streamk_kernel<false>, gemm_streamk_kernel<true>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_MAX_DYN_SMEM);
  return e;
}

void gemm_plan_destroy(GemmPlan *p) {
  if (p->d_cta_start) cudaFree(p->d_cta_start);
  p->d_cta_start = nullptr;
}

cudaError_t gemm_launch(const GemmPlan &p, const CUtensorMap *tmW_override, int *d_status, cudaStream_t st,
                        unsigned long long *trace, bool pdl) {
  if (p.BN <= GEMM_MAX_ROWS) return gemm_rows_launch(p, tmW_override, d_status, st, trace, pdl);
  const bool masked = p.row_keep != nullptr;
  auto go = [&](auto kernel) {
    return launch_k(kernel, dim3(p.grid), dim3(GEMM_THREADS), p.smem_bytes, st, pdl, tmW_override ? *tmW_override : p.tmW, p.tmX.hi[0], p.tmX.lo[0],
                    p.direct, p.ws, p.d_cta_start, p.N, p.KB, p.BN, p.R, p.stages, p.idesc, p.row_keep, p.keep_pitch, p.keep_div, d_status, trace,
                    p.row_blocks);
  };
  return masked ? go(gemm_streamk_kernel<true>) : go(gemm_streamk_kernel<false>);
}

int gemm_plan_rebase(GemmPlan *q, const GemmPlan &p, const void *Xhi, const void *Xlo, float *direct, __nv_bfloat16 *sw_hi,
                     __nv_bfloat16 *sw_lo, const int *row_blocks) {
  if (p.BN > GEMM_MAX_ROWS) return CORUN_EINVAL;    // (the other kernel's maps have other boxes)
  *q = p;
  q->direct = direct;
  q->sw_hi = sw_hi;
  q->sw_lo = sw_lo;
  q->row_blocks = row_blocks;
  return gemm_encode_x(&q->tmX, Xhi, Xlo, p.BN, p.K);
}

cudaError_t gemm_fixup_launch(const GemmPlan &p, cudaStream_t st, bool pdl, int rows) {
  if (p.n_split_tiles == 0) return cudaSuccess;
  const int R = rows ? rows : p.R, per = FIXUP_THREADS / (p.tile_n / 4), shares = (R + per - 1) / per;
  return launch_k(gemm_fixup_kernel, dim3(p.n_split_tiles, shares < FIXUP_SHARES ? shares : FIXUP_SHARES), dim3(FIXUP_THREADS), 0, st, pdl, p.out(),
                  p.direct, p.d_split_tiles, R, rows ? nullptr : p.row_blocks);
}

}  // namespace corun
