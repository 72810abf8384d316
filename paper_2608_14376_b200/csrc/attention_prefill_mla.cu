// Causal attention of a prefill chunk of a decoder with multi-head latent attention: the chunk's rows are consecutive
// tokens, so the heads' keys and values are decompressed once per cached token (one GEMM over the latents) and a tile of
// 128 query tokens shares every key / value tile.  The decode form (absorbed, one query token at a time over the latents)
// does 2176 multiply-adds per query, key and head and streams a request's whole latent cache once per token: 118 us per
// 256 tokens of a chunk; here it is 960, and the cache is read once per chunk.
//
// The cached latents are fp16 and enter the GEMM exactly (bf16 hi + lo); its fp32 results are kept as fp16 hi + lo pairs,
// queries and weights are hi + lo pairs too, and of the products only lo * lo is left out.  Such a pair holds 22 bits of values
// between 2^-13 and 2^15 only, so what goes into one is scaled by powers of two: keys and values per layer and head by what
// the weights allow at most (mla_kv_scale_kernel), a row's query by its own largest value.  The scales leave with the scores
// and with the division by the weights' sum, exactly.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math_constants.h>

#include "launch.cuh"
#include "mla.cuh"
#include "ptx.cuh"

namespace corun {

namespace {

constexpr int ML_THREADS = 352;                     // warp 0 TMA of the keys, warp 1 MMA, warps 2-5 softmax, warps 6-9 output, warp 10 TMA of the values
constexpr int ML_KEYS = 64;                         // keys per block
constexpr uint32_t ML_BOX = ML_KEYS * 128;          // [64 tokens x 64 dims] fp16
constexpr uint32_t ML_Q_BYTES = 3 * 128 * 128;      // hi or lo: [3 blocks of 64 dims][128 rows x 128 B]
constexpr uint32_t ML_K_BYTES = 5 * ML_BOX;         // hi, lo of the 128 no-rope dims, the rotary key
constexpr uint32_t ML_V_BYTES = 4 * ML_BOX;         // hi, lo
constexpr uint32_t ML_P_COL = 128, ML_O_COL = 256;  // tensor memory: scores, weights, outputs
constexpr size_t ML_SMEM = 1024 + 2 * ML_Q_BYTES + 2 * ML_K_BYTES + ML_V_BYTES;

__device__ __forceinline__ uint32_t ml_swz(int row, int chunk) { return (uint32_t)(row * 128 + ((chunk ^ (row & 7)) << 4)); }
__device__ __forceinline__ float ml_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// 2^e with x * 2^e <= 2^top, as large as that (1 for zero and for what is not finite; within 2^-60 .. 2^60)
__device__ __forceinline__ float ml_pow2_below(float x, int top) {
  if (!(x > 0.f) || x > 3.0e38f) return 1.f;
  int e;
  frexpf(x, &e);                                    // x < 2^e
  e = top - e;
  return __int_as_float(((e < -60 ? -60 : e > 60 ? 60 : e) + 127) << 23);
}
// eight fp32 -> fp16 hi and lo parts, 16 bytes each
__device__ __forceinline__ void ml_split8(const float *x, uint4 &hi, uint4 &lo) {
  __half2 h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = __floats2half2_rn(x[2 * i], x[2 * i + 1]);
    const float2 f = __half22float2(h[i]);
    l[i] = __floats2half2_rn(x[2 * i] - f.x, x[2 * i + 1] - f.y);
  }
  hi = *reinterpret_cast<const uint4 *>(h);
  lo = *reinterpret_cast<const uint4 *>(l);
}

// The largest power of two that keeps a head's keys (blockIdx.y 0) or values (1) at 2^10 or below: |sum_c w_c g_c x_c| <=
// rank * max |w_c g_c| for a normalised latent x (the sum of its squares is rank); what is met in practice lies some 2^6 below.
__global__ void __launch_bounds__(256)
mla_kv_scale_kernel(const __nv_bfloat16 *__restrict__ wkv_b, const __nv_bfloat16 *__restrict__ gains, MlaDims d, float *__restrict__ scale) {
  __shared__ float most[8];
  const int h = blockIdx.x, part = blockIdx.y, width = part ? d.vh : d.nope;
  const __nv_bfloat16 *w = wkv_b + ((size_t)h * (d.nope + d.vh) + (part ? d.nope : 0)) * d.rank;
  float m = 0.f;
  for (int i = 8 * threadIdx.x; i < width * d.rank; i += 8 * 256) {
    const uint4 a = *reinterpret_cast<const uint4 *>(w + i);
    const __nv_bfloat16 *x = reinterpret_cast<const __nv_bfloat16 *>(&a), *g = gains + i % d.rank;
#pragma unroll
    for (int j = 0; j < 8; ++j) m = fmaxf(m, fabsf(__bfloat162float(x[j]) * __bfloat162float(g[j])));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) most[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) m = fmaxf(m, most[i]);
    scale[2 * h + part] = ml_pow2_below(m * (float)d.rank, 10);
  }
}

// The latents of the segments' cached tokens as a bf16 hi / lo pair (exact) and their rotary keys (fp16), one warp per token.
__global__ void __launch_bounds__(256)
mla_gather_kernel(const __grid_constant__ MlaSegs g, MlaCache cache, int rank, int rope, int total, __nv_bfloat16 *__restrict__ c_hi,
                  __nv_bfloat16 *__restrict__ c_lo, __half *__restrict__ kr) {
  griddep_launch_dependents();
  griddep_wait();
  const int t = (int)blockIdx.x * 8 + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= total) return;
  int s = 0;
  while (s + 1 < g.n && t >= g.off[s + 1]) ++s;
  const int pos = t - g.off[s];
  if (pos >= g.len[s]) return;                      // the rest of a segment's last block: never weighted
  const int blk = cache.block_table[(size_t)g.slot[s] * cache.max_blocks + pos / KV_BLOCK];
  for (int c = lane; c < (rank + rope) / 8; c += 32) {
    const uint4 raw = *reinterpret_cast<const uint4 *>(mla_cache_at(cache, rank + rope, blk, pos % KV_BLOCK, 8 * c));
    if (8 * c >= rank) {
      *reinterpret_cast<uint4 *>(kr + (size_t)t * 64 + 8 * c - rank) = raw;
      continue;
    }
    const __half *x = reinterpret_cast<const __half *>(&raw);
    __nv_bfloat16 a[8], b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float v = __half2float(x[i]);
      a[i] = __float2bfloat16_rn(v);
      b[i] = __float2bfloat16_rn(v - __bfloat162float(a[i]));
    }
    *reinterpret_cast<uint4 *>(c_hi + (size_t)t * rank + 8 * c) = *reinterpret_cast<const uint4 *>(a);
    *reinterpret_cast<uint4 *>(c_lo + (size_t)t * rank + 8 * c) = *reinterpret_cast<const uint4 *>(b);
  }
}

// One CTA per (head, tile of 128 chunk rows = consecutive tokens of one request).  Per block of 64 keys:
//   S[128 x 64] = Qhi Khi + Qlo Khi + Qhi Klo (12 k-slices) into one of two TMEM buffers;
//   softmax warps, a thread per row: running maximum, P = exp2(S - max) as fp16 hi and lo into one of two TMEM buffers, the factor
//     by which the earlier sums shrink;
//   O'[128 x 128] = Phi Vhi + Plo Vhi + Phi Vlo (4 k-slices), P from tensor memory, into one of two TMEM buffers;
//   output warps, a thread per row: O = O * factor + O', in registers.
// MMAs on different accumulators may overtake one another, so none writes what another one may still read: scores of block j + 2
// overwrite those of block j, which the softmax has read when it hands over its weights; the weights of block j + 2 are written
// behind the commit of its scores, which are issued behind the values of block j and so complete no earlier.  The
// keys of two blocks are in shared memory.  (One key buffer, weights through shared memory and one producer for keys and values, so that
// a block's keys were requested behind the values before them, and queries and results by a thread per row: 2505 tokens of 16 heads
// 160 us per layer, now 125.)  What bounds a block are its 32 MMAs of 48 and 12 of 64 cycles.
// Every reduction runs in one fixed order that depends on the row's own position only.  All waits are bounded.
__global__ void __launch_bounds__(ML_THREADS, 1)
mla_prefill_kernel(const __grid_constant__ CUtensorMap tmKV, const __grid_constant__ CUtensorMap tmR, const __nv_bfloat16 *__restrict__ qn_hi,
                   const __nv_bfloat16 *__restrict__ qn_lo, const float *__restrict__ q_rope, Rows rows, int rows_per_head, int nh, int rope,
                   int cap, const int *__restrict__ tile_base, float scale_log2e, const float2 *__restrict__ kv_scale, __nv_bfloat16 *__restrict__ ao_hi,
                   __nv_bfloat16 *__restrict__ ao_lo, int *status) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t kfull[2], kempty[2], vfull, vempty, s_full[2], p_ready[2], o_full[2], o_free[2], c_ready[4], l_ready;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;
  __shared__ float corr_s[4][128], l_s[128], row_scale_s[128];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int h = blockIdx.x, tile = (int)gridDim.y - 1 - (int)blockIdx.y;   // the last tiles (the most keys) first
  const int row0 = tile * 128;
  const float2 kvs = __ldg(kv_scale + h);           // the head's keys and values are stored times these
  // the tile's rows with a token are the first ones
  const int n_rows = __syncthreads_count(tid < 128 && row0 + tid < rows.R && rows.active[row0 + tid] != 0);
  if (n_rows == 0) return;
  const int n_blocks = rows.pos[row0 + n_rows - 1] / ML_KEYS + 1, base_tok = tile_base[tile];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t q_hi = base, q_lo = base + ML_Q_BYTES, k_ring = q_lo + ML_Q_BYTES, v_buf = k_ring + 2 * ML_K_BYTES;
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&vfull), 1); mbar_init(smem_u32(&vempty), 1);
    mbar_init(smem_u32(&l_ready), 128);
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&kfull[i]), 1); mbar_init(smem_u32(&kempty[i]), 1);
      mbar_init(smem_u32(&s_full[i]), 1); mbar_init(smem_u32(&p_ready[i]), 128);
      mbar_init(smem_u32(&o_full[i]), 1); mbar_init(smem_u32(&o_free[i]), 128);
    }
    for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&c_ready[i]), 128);
    fence_mbar_init();
    fence_proxy_async();
    prefetch_tensormap(&tmKV);
    prefetch_tensormap(&tmR);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_s), 512);        // scores 2 x 64 columns, weights (hi, lo) 2 x 64, outputs 2 x 128
    tmem_relinquish();
  }
  if (warp >= 2 && warp < 10) {
    // the query tile: row m = token m, 128 no-rope dims (four per lane), then the rotary ones (two per lane), zeros beyond them: a
    // warp takes a row at a time, four in flight
    for (int m0 = warp - 2; m0 < 128; m0 += 32) {
      uint2 a[4], b[4];
      float2 p[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int r = row0 + m0 + 8 * k;
        const bool on = r < rows.R;
        const size_t o = ((size_t)h * rows_per_head + r) * 128 + 4 * lane;
        a[k] = on ? *reinterpret_cast<const uint2 *>(qn_hi + o) : make_uint2(0u, 0u);
        b[k] = on ? *reinterpret_cast<const uint2 *>(qn_lo + o) : make_uint2(0u, 0u);
        p[k] = on && 2 * lane < rope ? *reinterpret_cast<const float2 *>(q_rope + ((size_t)r * nh + h) * rope + 2 * lane) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int m = m0 + 8 * k;
        const __nv_bfloat16 *pa = reinterpret_cast<const __nv_bfloat16 *>(&a[k]), *pb = reinterpret_cast<const __nv_bfloat16 *>(&b[k]);
        float x[6], most = 0.f;                     // the rotary ones at the scale of the keys beside theirs
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = __bfloat162float(pa[i]) + __bfloat162float(pb[i]);
        x[4] = p[k].x * kvs.x;
        x[5] = p[k].y * kvs.x;
#pragma unroll
        for (int i = 0; i < 6; ++i) most = fmaxf(most, fabsf(x[i]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, o));
        const float q_scale = ml_pow2_below(most, 14);
        if (lane == 0) row_scale_s[m] = scale_log2e / q_scale / kvs.x;
        __half hi[6], lo[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          const float y = x[i] * q_scale;
          hi[i] = __float2half_rn(y);
          lo[i] = __float2half_rn(y - __half2float(hi[i]));
        }
        const uint32_t on = (uint32_t)(lane >> 4) * (128 * 128) + ml_swz(m, (lane & 15) >> 1) + (uint32_t)(lane & 1) * 8;
        const uint32_t orr = 2u * (128 * 128) + ml_swz(m, lane >> 2) + (uint32_t)(lane & 3) * 4;
        const __half2 h01 = __halves2half2(hi[0], hi[1]), h23 = __halves2half2(hi[2], hi[3]), l01 = __halves2half2(lo[0], lo[1]), l23 = __halves2half2(lo[2], lo[3]);
        *reinterpret_cast<uint2 *>(base_ptr + on) = make_uint2(*reinterpret_cast<const uint32_t *>(&h01), *reinterpret_cast<const uint32_t *>(&h23));
        *reinterpret_cast<uint2 *>(base_ptr + ML_Q_BYTES + on) = make_uint2(*reinterpret_cast<const uint32_t *>(&l01), *reinterpret_cast<const uint32_t *>(&l23));
        *reinterpret_cast<__half2 *>(base_ptr + orr) = __halves2half2(hi[4], hi[5]);
        *reinterpret_cast<__half2 *>(base_ptr + ML_Q_BYTES + orr) = __halves2half2(lo[4], lo[5]);
      }
    }
    fence_proxy_async();                            // the MMAs read these tiles through the async proxy
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  bool failed = false;
  // warps 2-5 and 6-9: this thread's row
  const int quad = warp & 3, tl = quad * 32 + lane;
  const bool real = tl < n_rows;

  if (warp == 0 || warp == 10) {
    if (elect_one()) {
      // ---------------- TMA producers ----------------
      const uint64_t pol = l2_policy_evict_last();  // the tiles of the same head read the same keys and values
      for (int j = 0; j < n_blocks && !failed; ++j) {
        const int tok = base_tok + j * ML_KEYS, kb = j & 1;
        auto y = [&](int part) { return (part * nh + h) * cap + tok; };   // part: key hi, key lo, value hi, value lo
        if (warp == 0) {
          const uint32_t fb = smem_u32(&kfull[kb]), dst = k_ring + (uint32_t)kb * ML_K_BYTES;
          if (j > 1 && !mbar_wait(smem_u32(&kempty[kb]), (uint32_t)((j >> 1) - 1) & 1u, &abort_flag)) { failed = true; break; }
          mbar_arrive_expect_tx(fb, ML_K_BYTES);
          for (int i = 0; i < 4; ++i) tma_load_2d(dst + (uint32_t)i * ML_BOX, &tmKV, (i & 1) * 64, y(i >> 1), fb, pol);
          tma_load_2d(dst + 4 * ML_BOX, &tmR, 0, tok, fb, pol);
        } else {
          if (j > 0 && !mbar_wait(smem_u32(&vempty), (uint32_t)(j - 1) & 1u, &abort_flag)) { failed = true; break; }
          mbar_arrive_expect_tx(smem_u32(&vfull), ML_V_BYTES);
          for (int i = 0; i < 4; ++i)
            tma_load_2d(v_buf + (uint32_t)i * ML_BOX, &tmKV, (i & 1) * 64, y(2 + (i >> 1)), smem_u32(&vfull), pol);
        }
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      // ---------------- MMA issuer ----------------
      const uint32_t idesc_s = (1u << 4) | ((uint32_t)(ML_KEYS >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      const uint32_t idesc_o = (1u << 4) | (1u << 16) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);   // values MN-major
      auto scores = [&](int j) {
        const int sb = j & 1;
        if (!mbar_wait(smem_u32(&kfull[sb]), (uint32_t)(j >> 1) & 1u, &abort_flag)) { failed = true; return; }
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)sb * 64, k_buf = k_ring + (uint32_t)sb * ML_K_BYTES;
#pragma unroll
        for (int ks = 0; ks < 12; ++ks) {
          const uint64_t adv = (uint64_t)((ks & 3) * 2);
          const uint32_t b = (uint32_t)(ks >> 2);
          const uint64_t qh = umma_desc_sw128(q_hi + b * (128 * 128)) + adv, ql = umma_desc_sw128(q_lo + b * (128 * 128)) + adv;
          const uint64_t kh = umma_desc_sw128(k_buf + (ks < 8 ? b : 4u) * ML_BOX) + adv;
          umma_bf16(d, qh, kh, idesc_s, ks > 0 ? 1u : 0u);   // operand format (fp16) is in idesc
          umma_bf16(d, ql, kh, idesc_s, 1u);
          if (ks < 8) umma_bf16(d, qh, umma_desc_sw128(k_buf + (2 + b) * ML_BOX) + adv, idesc_s, 1u);   // (the rotary key is fp16 as cached)
        }
        umma_commit(smem_u32(&kempty[sb]));
        umma_commit(smem_u32(&s_full[sb]));
      };
      scores(0);
      if (n_blocks > 1 && !failed) scores(1);
      for (int j = 0; j < n_blocks && !failed; ++j) {
        const int b = j & 1;
        if (!mbar_wait(smem_u32(&p_ready[b]), (uint32_t)(j >> 1) & 1u, &abort_flag)) { failed = true; break; }
        if (!mbar_wait(smem_u32(&vfull), (uint32_t)j & 1u, &abort_flag)) { failed = true; break; }
        if (j >= 2 && !mbar_wait(smem_u32(&o_free[b]), (uint32_t)((j >> 1) - 1) & 1u, &abort_flag)) { failed = true; break; }
        tc_fence_after();
        const uint32_t p = tmem + ML_P_COL + (uint32_t)b * 64, d = tmem + ML_O_COL + (uint32_t)b * 128;
#pragma unroll
        for (int ks = 0; ks < ML_KEYS / 16; ++ks) {
          const uint32_t ph = p + (uint32_t)(8 * ks), pl = ph + 32;   // 16 tokens of weights are 8 columns
          // values [128 dims x 16 tokens], MN-major: blocks of 64 dims a box apart, groups of 8 tokens 1 KiB apart
          const uint64_t vh = umma_desc_sw128_mn(v_buf + (uint32_t)ks * 2048, ML_BOX, 1024u);
          const uint64_t vl = umma_desc_sw128_mn(v_buf + 2 * ML_BOX + (uint32_t)ks * 2048, ML_BOX, 1024u);
          umma_f16_ts(d, ph, vh, idesc_o, ks > 0 ? 1u : 0u);
          umma_f16_ts(d, pl, vh, idesc_o, 1u);
          umma_f16_ts(d, ph, vl, idesc_o, 1u);
        }
        umma_commit(smem_u32(&vempty));
        umma_commit(smem_u32(&o_full[b]));
        if (j + 2 < n_blocks) scores(j + 2);
      }
    }
  } else if (warp < 6) {
    // ---------------- softmax: one thread per row ----------------
    const int pos = real ? rows.pos[row0 + tl] : -1;
    const float scale = row_scale_s[tl];            // scores to the base-2 domain, without the operands' scales
    float mx = -CUDART_INF_F, l = 0.f;
    for (int j = 0; j < n_blocks; ++j) {
      const int sb = j & 1;
      bool ok = mbar_wait(smem_u32(&s_full[sb]), (uint32_t)(j >> 1) & 1u, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { failed = true; break; }
      tc_fence_after();
      uint32_t sv[4][16];
#pragma unroll
      for (int x = 0; x < 4; ++x) tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(sb * 64 + 16 * x), sv[x]);
      tmem_ld_wait();
      const int lim = pos - j * ML_KEYS;            // keys 0 .. lim of the block are visible
      float m4[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
      for (int i = 0; i < ML_KEYS; ++i) m4[i & 3] = fmaxf(m4[i & 3], i <= lim ? __uint_as_float(sv[i >> 4][i & 15]) * scale : -CUDART_INF_F);
      const float bm = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      const float m_new = fmaxf(mx, bm), m_use = m_new == -CUDART_INF_F ? 0.f : m_new;   // (rows without a token: nothing visible)
      const float corr = ml_ex2(mx - m_use);
      mx = m_new;
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      float p[ML_KEYS];
#pragma unroll
      for (int i = 0; i < ML_KEYS; ++i) {
        p[i] = i <= lim ? ml_ex2(fmaf(__uint_as_float(sv[i >> 4][i & 15]), scale, -m_use)) : 0.f;
        acc[i & 3] += p[i];
      }
      l = l * corr + ((acc[0] + acc[1]) + (acc[2] + acc[3]));
      const uint32_t pt = tmem + ((uint32_t)(quad * 32) << 16) + ML_P_COL + (uint32_t)(sb * 64);
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint4 h0, l0, h1, l1;
        ml_split8(&p[16 * c], h0, l0);
        ml_split8(&p[16 * c + 8], h1, l1);
        tmem_st8(pt + (uint32_t)(8 * c), {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w});
        tmem_st8(pt + (uint32_t)(32 + 8 * c), {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w});
      }
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(smem_u32(&p_ready[sb]));
      corr_s[j & 3][tl] = corr;                     // (block j - 4's has been read: its output was, before the scores of this block were issued)
      mbar_arrive(smem_u32(&c_ready[j & 3]));
    }
    l_s[tl] = l;
    mbar_arrive(smem_u32(&l_ready));
  } else {
    // ---------------- output: one thread per row, 128 dims in registers ----------------
    float o[128];
#pragma unroll
    for (int i = 0; i < 128; ++i) o[i] = 0.f;
    for (int j = 0; j < n_blocks; ++j) {
      const int ob = j & 1;
      bool ok = mbar_wait(smem_u32(&c_ready[j & 3]), (uint32_t)(j >> 2) & 1u, &abort_flag);
      ok = ok && mbar_wait(smem_u32(&o_full[ob]), (uint32_t)(j >> 1) & 1u, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { failed = true; break; }
      const float corr = corr_s[j & 3][tl];
      tc_fence_after();
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        uint32_t v[8];
        tmem_ld8(tmem + ((uint32_t)(quad * 32) << 16) + ML_O_COL + (uint32_t)(ob * 128 + 8 * q), v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) o[8 * q + i] = fmaf(o[8 * q + i], corr, __uint_as_float(v[i]));
      }
      tc_fence_before();
      mbar_arrive(smem_u32(&o_free[ob]));
    }
    bool ok = !failed && mbar_wait(smem_u32(&l_ready), 0u, &abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    // bf16 hi / lo through the query tiles' shared memory (all MMAs have read them), then whole rows
    auto at = [&](int row, int c) { return (uint32_t)(row * 256 + ((c ^ (row & 7)) << 4)); };
    if (ok) {
      const float inv = 1.f / l_s[tl] / kvs.y;      // (rows without a token: not stored)
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        __nv_bfloat16 a[8], b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float y = o[8 * q + i] * inv;
          a[i] = __float2bfloat16_rn(y);
          b[i] = __float2bfloat16_rn(y - __bfloat162float(a[i]));
        }
        *reinterpret_cast<uint4 *>(base_ptr + at(tl, q)) = *reinterpret_cast<const uint4 *>(a);
        *reinterpret_cast<uint4 *>(base_ptr + ML_Q_BYTES + at(tl, q)) = *reinterpret_cast<const uint4 *>(b);
      }
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");  // warps 6-9 (whatever failed)
    if (ok) {
#pragma unroll 4
      for (int k = 0; k < 16; ++k) {
        const int u = k * 128 + tid - 192, row = u >> 4, c = u & 15;
        if (row < n_rows) {
          const size_t to = ((size_t)(row0 + row) * nh + h) * 128 + 8 * c;
          *reinterpret_cast<uint4 *>(ao_hi + to) = *reinterpret_cast<const uint4 *>(base_ptr + at(row, c));
          *reinterpret_cast<uint4 *>(ao_lo + to) = *reinterpret_cast<const uint4 *>(base_ptr + ML_Q_BYTES + at(row, c));
        }
      }
    }
  }
  __syncwarp();
  if (failed || abort_flag) {
    if (lane == 0) atomicCAS(status, 0, DEV_TIMEOUT_EPILOGUE);
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);   // let copies in flight land before the CTA retires
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

}  // namespace

cudaError_t launch_mla_gather(const MlaSegs &g, const MlaCache &cache, int rank, int rope, int total, __nv_bfloat16 *c_hi,
                              __nv_bfloat16 *c_lo, __half *kr, cudaStream_t st) {
  return launch_k(mla_gather_kernel, dim3((total + 7) / 8), dim3(256), 0, st, true, g, cache, rank, rope, total, c_hi, c_lo, kr);
}

cudaError_t launch_mla_kv_scale(const __nv_bfloat16 *wkv_b, const __nv_bfloat16 *gains, const MlaDims &d, float2 *scale, cudaStream_t st) {
  mla_kv_scale_kernel<<<dim3(d.nh, 2), 256, 0, st>>>(wkv_b, gains, d, reinterpret_cast<float *>(scale));
  return cudaGetLastError();
}

cudaError_t mla_prefill_prepare() {
  return cudaFuncSetAttribute(mla_prefill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ML_SMEM);
}

cudaError_t launch_mla_prefill(const CUtensorMap &tmKV, const CUtensorMap &tmR, const __nv_bfloat16 *qn_hi, const __nv_bfloat16 *qn_lo,
                               const float *q_rope, const Rows &rows, int rows_per_head, const MlaDims &d, int cap, const int *tile_base,
                               float scale, const float2 *kv_scale, __nv_bfloat16 *ao_hi, __nv_bfloat16 *ao_lo, int *d_status, cudaStream_t st) {
  return launch_k(mla_prefill_kernel, dim3(d.nh, (rows.R + 127) / 128), dim3(ML_THREADS), ML_SMEM, st, false, tmKV, tmR, qn_hi, qn_lo, q_rope,
                  rows, rows_per_head, d.nh, d.rope, cap, tile_base, scale * 1.4426950408889634f, kv_scale, ao_hi, ao_lo, d_status);
}

}  // namespace corun
