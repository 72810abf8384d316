// Causal attention of a prefill chunk: the chunk's rows are consecutive tokens of ONE request, so a tile of
// query rows shares every key / value tile it reads (the decode kernel reads them once per query row).
//
// One CTA per (tile of 128 / G consecutive tokens, kv head), G = query heads per kv head.  The 128 rows of the tile are the
// (token, head) pairs; row m = token m / G, head m % G.  It walks the blocks of 128 cached tokens (8 pages) from position 0
// to the tile's last token once:
//   S[128 rows x 128 keys] = Q * K^T on tcgen05.mma (M = 128, N = 128, fp16, Q as a hi/lo pair: two MMAs per k-slice) into
//     one of two TMEM buffers;
//   softmax warps, a thread per row (TMEM lane = row): P = exp2(S - the block's own maximum) as fp16 to shared memory (causal
//     mask: key position <= the row's own position), and the factor between this block's scale and the earlier ones';
//   O'[128 x hd] = P * V, one MMA per page, into one of two TMEM buffers;
//   output warps, a thread per row: O and O' to the larger of the two maxima and added, in registers; at the end O / sum ->
//     bf16 hi/lo.
// A block's largest weight is exactly 1 in fp16 and the factors are fp32, so the keys that carry a row have unrounded weights
// (relative to the running maximum only one of them did: prompts of 300 / 1003 tokens through 12 Qwen3-8B layers were
// 1.1e-4 / 6.7e-5 off a 64-bit evaluation).
// The scores of block j + 1 are issued ahead of the values of block j.  (A kernel that walked the blocks twice, exact maxima
// first, over a cluster of two CTAs per tile took 40 MMAs per block instead of 24: 6001 tokens of the Qwen3-8B shape, last
// chunk of 1905 rows, 479 us per layer.)
// Roles: warp 0 streams the keys and warp 10 the values with TMA (rings of two; one 4-dimensional box per (page, head)
// tile), warp 1 issues the MMAs, warps 2-5 are the softmax, warps 6-9 the output.
//
// A page's keys land as [2 groups of 8 tokens][hd / 64][8 tokens][64 dims]: for the scores a K-major operand whose groups of
// eight rows lie hd / 64 KiB apart, for the values (cached alike) an MN-major one.
//
// Every reduction has one fixed order (per thread: four interleaved partial sums over a block's keys in ascending order, then
// a fixed tree; blocks ascending) that depends on the row's own position only.  All waits are bounded.
#include <cuda_fp16.h>
#include <math_constants.h>

#include "launch.cuh"
#include "ops.cuh"
#include "ptx.cuh"

namespace corun {

namespace {

constexpr int PF_THREADS = 352;
constexpr int PF_KEYS = 128;                        // keys per block
constexpr int PF_PAGES = PF_KEYS / KV_BLOCK;        // 8
constexpr int PF_RING = 2;                          // key and value ring depth

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pf_swz(int row, int chunk) { return (uint32_t)(row * 128 + ((chunk ^ (row & 7)) << 4)); }

template <int HD>
struct PfLayout {
  static constexpr int NHALF = HD / 64;
  static constexpr int Q_BYTES = NHALF * 128 * 128;           // one of hi / lo: [half][128 rows x 128 B]
  static constexpr int P_BYTES = 2 * 128 * 128;               // one weight tile: [key half][128 rows x 128 B]
  static constexpr int PAGE_BYTES = NHALF * KV_BLOCK * 128;   // one page's keys (values) of one head
  static constexpr int B_BYTES = PF_PAGES * PAGE_BYTES;       // a block of keys (values)
  static constexpr size_t SMEM = (size_t)2 * Q_BYTES + P_BYTES + 2 * PF_RING * B_BYTES + 1024;
};

template <int HD, int GROUP>
__global__ void __launch_bounds__(PF_THREADS, 1)
attn_prefill_kernel(const __grid_constant__ CUtensorMap tmKV, const float *__restrict__ q, Rows rows, int nq, KvLayout kv,
                    __nv_bfloat16 *__restrict__ out_hi, __nv_bfloat16 *__restrict__ out_lo, int *status) {
  using L = PfLayout<HD>;
  constexpr int TPT = 128 / GROUP;                  // tokens per tile
  constexpr int KSTEPS = HD / 16;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t kfull[PF_RING], kempty[PF_RING], vfull[PF_RING], vempty[PF_RING], s_full[2], s_free[2], o_full[2], o_free[2],
      p_ready, p_free, c_ready[2], l_ready;
  __shared__ float corr_s[2][128], l_s[128];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // heads fastest, the last tiles (the most key blocks) first: the short ones fill the last wave
  const int tile = (int)gridDim.y - 1 - (int)blockIdx.y, g = blockIdx.x, row0 = tile * TPT;
  griddep_wait();                                   // q and the chunk's own keys / values come from the kernel before
  // the tile's rows with a token are the first ones
  const int n_tok = __syncthreads_count(tid < TPT && row0 + tid < rows.R && rows.active[row0 + tid] != 0);
  griddep_launch_dependents();
  if (n_tok == 0) return;                           // padding only
  const int ctx_tile = rows.pos[row0 + n_tok - 1] + 1;
  const int n_blocks = (ctx_tile + PF_KEYS - 1) / PF_KEYS;
  const int slot = rows.slot[row0];
  auto pages_of = [&](int b) { return min(PF_PAGES, (ctx_tile - b * PF_KEYS + KV_BLOCK - 1) / KV_BLOCK); };   // the last block may be partial

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t q_hi = base, q_lo = base + L::Q_BYTES, p_tile = q_lo + L::Q_BYTES, k_ring = p_tile + L::P_BYTES,
                 v_ring = k_ring + PF_RING * L::B_BYTES;
  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < PF_RING; ++i) {
      mbar_init(smem_u32(&kfull[i]), 1); mbar_init(smem_u32(&kempty[i]), 1);
      mbar_init(smem_u32(&vfull[i]), 1); mbar_init(smem_u32(&vempty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&s_full[i]), 1); mbar_init(smem_u32(&s_free[i]), 128);   // scores in TMEM / read by every row thread
      mbar_init(smem_u32(&o_full[i]), 1); mbar_init(smem_u32(&o_free[i]), 128);   // the same for a block's output
    }
    mbar_init(smem_u32(&p_ready), 128);             // every row thread has written its weights
    mbar_init(smem_u32(&p_free), 1);                // the value MMAs have read the weight tile
    for (int i = 0; i < 2; ++i) mbar_init(smem_u32(&c_ready[i]), 128);            // the rows' factors of a block
    mbar_init(smem_u32(&l_ready), 128);
    fence_mbar_init();
    fence_proxy_async();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_s), 512);        // 2 x 128 columns of scores, 2 x 128 of output
    tmem_relinquish();
  }
  if (warp >= 2 && warp < 10) {
    // ---- the query tile: row m = (token m / G, head m % G) as fp16 hi and lo tiles (q = hi + lo)
    const int m = (tid - 64) & 127, dh = (tid - 64) >> 7;   // row, and which half of the head dimension
    const int t = m / GROUP, h = m % GROUP;
    const bool real = row0 + t < rows.R;
    const float *qr = q + ((size_t)(real ? row0 + t : row0) * nq + (size_t)g * GROUP + h) * HD;
#pragma unroll 4
    for (int d = dh * (HD / 2); d < (dh + 1) * (HD / 2); d += 8) {
      __half hi[8], lo[8];
#pragma unroll
      for (int j = 0; j < 8; j += 4) {
        const float4 v = real ? *reinterpret_cast<const float4 *>(qr + d + j) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          hi[j + i] = __float2half_rn(x[i]);
          lo[j + i] = __float2half_rn(x[i] - __half2float(hi[j + i]));
        }
      }
      const uint32_t off = (uint32_t)(d >> 6) * (128 * 128) + pf_swz(m, (d & 63) >> 3);
      *reinterpret_cast<uint4 *>(base_ptr + off) = *reinterpret_cast<const uint4 *>(hi);
      *reinterpret_cast<uint4 *>(base_ptr + L::Q_BYTES + off) = *reinterpret_cast<const uint4 *>(lo);
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
  const bool real = tl / GROUP < n_tok;

  if (warp == 0 || warp == 10) {
    // ---------------- producers: lane l fetches page l of a block, its page number read one block ahead of its use
    const bool keys = warp == 0;
    const uint64_t pol = l2_policy_evict_last();    // the tiles of the same request read the same cache rows
    const int *table = kv.block_table + (size_t)slot * kv.max_blocks;
    int page_next = lane < pages_of(0) ? table[lane] : 0;
    for (int j = 0; j < n_blocks; ++j) {
      const int buf = j % PF_RING, n_pages = pages_of(j), page = page_next;
      if (j + 1 < n_blocks) page_next = lane < pages_of(j + 1) ? table[(j + 1) * PF_PAGES + lane] : 0;
      if (j >= PF_RING) {
        bool ok = mbar_wait(smem_u32(keys ? &kempty[buf] : &vempty[buf]), (uint32_t)(j / PF_RING - 1) & 1u, &abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) { failed = true; break; }
      }
      const uint32_t fb = smem_u32(keys ? &kfull[buf] : &vfull[buf]);
      if (lane == 0) mbar_arrive_expect_tx(fb, (uint32_t)(n_pages * L::PAGE_BYTES));
      __syncwarp();
      if (lane < n_pages)                           // the page's (head) tile in one box; the last dimension counts groups of 8 tokens
        tma_load_4d((keys ? k_ring : v_ring) + (uint32_t)(buf * L::B_BYTES + lane * L::PAGE_BYTES), &tmKV, 0, 0, 0,
                    (page * 2 * kv.n_kv + (keys ? 0 : kv.n_kv) + g) * (KV_BLOCK / 8), fb, pol);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: the scores of block j, then the values of block j - 1
    if (elect_one()) {
      // fp16 x fp16 -> fp32; N at bit 17 (>> 3), M = 128 at bit 24 (>> 4); the values are an MN-major B operand
      const uint32_t idesc_s = (1u << 4) | ((uint32_t)(PF_KEYS >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      const uint32_t idesc_o = (1u << 4) | (1u << 16) | ((uint32_t)(HD >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      for (int j = 0; j <= n_blocks && !failed; ++j) {
        if (j < n_blocks) {
          const int buf = j % PF_RING, sb = j & 1;
          if (j >= 2 && !mbar_wait(smem_u32(&s_free[sb]), (uint32_t)((j >> 1) - 1) & 1u, &abort_flag)) { failed = true; break; }
          if (!mbar_wait(smem_u32(&kfull[buf]), (uint32_t)(j / PF_RING) & 1u, &abort_flag)) { failed = true; break; }
          tc_fence_after();
          const uint32_t kt = k_ring + (uint32_t)(buf * L::B_BYTES), st = tmem + (uint32_t)sb * 128;
#pragma unroll
          for (int ks = 0; ks < KSTEPS; ++ks) {
            const uint64_t adv = (uint64_t)((ks & 3) * 2);
            const uint64_t bk = umma_desc_sw128_sbo(kt + (uint32_t)(ks >> 2) * 1024u, L::NHALF * 1024u) + adv;
            const uint64_t ah = umma_desc_sw128(q_hi + (uint32_t)(ks >> 2) * (128 * 128)) + adv;
            const uint64_t al = umma_desc_sw128(q_lo + (uint32_t)(ks >> 2) * (128 * 128)) + adv;
            umma_bf16(st, ah, bk, idesc_s, ks > 0 ? 1u : 0u);    // operand format (fp16) is in idesc
            umma_bf16(st, al, bk, idesc_s, 1u);
          }
          umma_commit(smem_u32(&kempty[buf]));
          umma_commit(smem_u32(&s_full[sb]));
        }
        if (j >= 1) {
          const int i = j - 1, buf = i % PF_RING, ob = i & 1;
          if (!mbar_wait(smem_u32(&p_ready), (uint32_t)i & 1u, &abort_flag)) { failed = true; break; }
          if (!mbar_wait(smem_u32(&vfull[buf]), (uint32_t)(i / PF_RING) & 1u, &abort_flag)) { failed = true; break; }
          if (i >= 2 && !mbar_wait(smem_u32(&o_free[ob]), (uint32_t)((i >> 1) - 1) & 1u, &abort_flag)) { failed = true; break; }
          tc_fence_after();
          const int n_pages = pages_of(i);
          const uint32_t vt = v_ring + (uint32_t)(buf * L::B_BYTES), d = tmem + 256 + (uint32_t)ob * 128;
          for (int p = 0; p < n_pages; ++p) {
            const uint64_t a = umma_desc_sw128(p_tile + (uint32_t)(p >> 2) * (128 * 128)) + (uint64_t)((p & 3) * 2);
            umma_bf16(d, a, umma_desc_sw128_mn(vt + (uint32_t)(p * L::PAGE_BYTES), 1024u, L::NHALF * 1024u), idesc_o, p > 0 ? 1u : 0u);
          }
          umma_commit(smem_u32(&vempty[buf]));
          umma_commit(smem_u32(&p_free));
          umma_commit(smem_u32(&o_full[ob]));
        }
      }
    }
  } else if (warp < 6) {
    // ---------------- softmax: one thread per row
    const int pos = real ? rows.pos[row0 + tl / GROUP] : -1;       // keys 0..pos are visible to this row
    const float sscale = (HD == 128 ? 0.08838834764831845f : 0.125f) * 1.4426950408889634f;   // log2(e)/sqrt(hd)
    uint8_t *p_ptr = base_ptr + 2 * L::Q_BYTES;
    float mx = -CUDART_INF_F, l = 0.f;
    for (int j = 0; j < n_blocks; ++j) {
      const int sb = j & 1;
      bool ok = mbar_wait(smem_u32(&s_full[sb]), (uint32_t)(j >> 1) & 1u, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { failed = true; break; }
      tc_fence_after();
      const uint32_t st = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(sb * 128);
      uint32_t sv[8][16];
#pragma unroll
      for (int x = 0; x < 8; ++x) tmem_ld16(st + (uint32_t)(16 * x), sv[x]);
      tmem_ld_wait();
      tc_fence_before();
      mbar_arrive(smem_u32(&s_free[sb]));           // the scores are in registers: their buffer may be overwritten
      const int lim = pos - j * PF_KEYS;            // keys 0 .. lim of the block are visible
      const bool masked = lim < PF_KEYS - 1;        // only the row's last block (or padding) needs the mask
      float bm = -CUDART_INF_F;
      if (!masked) {
#pragma unroll
        for (int i = 0; i < PF_KEYS; ++i) bm = fmaxf(bm, __uint_as_float(sv[i >> 4][i & 15]));
      } else {
#pragma unroll
        for (int i = 0; i < PF_KEYS; ++i)
          if (i <= lim) bm = fmaxf(bm, __uint_as_float(sv[i >> 4][i & 15]));
      }
      bm *= sscale;
      const float ref = bm == -CUDART_INF_F ? 0.f : bm;              // (nothing visible in this block: all its weights are 0)
      // the larger maximum is the scale from here on: a factor for the sums so far (not negative), or for this block (its sign bit set)
      const bool up = bm >= mx;
      const float factor = ex2_approx(up ? mx - ref : bm - mx), corr = up ? factor : -factor;
      mx = fmaxf(mx, bm);
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          float p0 = ex2_approx(fmaf(__uint_as_float(sv[x][i]), sscale, -ref));
          float p1 = ex2_approx(fmaf(__uint_as_float(sv[x][i + 1]), sscale, -ref));
          if (masked) {
            if (16 * x + i > lim) p0 = 0.f;
            if (16 * x + i + 1 > lim) p1 = 0.f;
          }
          acc[i & 3] += p0;
          acc[(i + 1) & 3] += p1;
          const __half2 h2 = __floats2half2_rn(p0, p1);
          sv[x][i >> 1] = *reinterpret_cast<const uint32_t *>(&h2);   // (the scores up to i + 1 have been used)
        }
      const float sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
      l = up ? fmaf(l, factor, sum) : fmaf(sum, factor, l);
      if (j > 0) {                                  // the value MMAs of the block before must have read the weight tile,
        bool okp = mbar_wait(smem_u32(&p_free), (uint32_t)(j - 1) & 1u, &abort_flag);
        if (j > 1) okp = okp && mbar_wait(smem_u32(&o_free[sb]), (uint32_t)((j >> 1) - 1) & 1u, &abort_flag);   // the output warps the factors of block j - 2
        okp = __all_sync(0xffffffffu, okp);
        if (!okp) { failed = true; break; }
      }
      corr_s[sb][tl] = corr;
      // weights as the A operand of the value MMA: [key half][row][64 keys], 128-byte swizzle
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        uint8_t *pw = p_ptr + (size_t)(x >> 2) * (128 * 128);
        *reinterpret_cast<uint4 *>(pw + pf_swz(tl, 2 * (x & 3))) = make_uint4(sv[x][0], sv[x][1], sv[x][2], sv[x][3]);
        *reinterpret_cast<uint4 *>(pw + pf_swz(tl, 2 * (x & 3) + 1)) = make_uint4(sv[x][4], sv[x][5], sv[x][6], sv[x][7]);
      }
      fence_proxy_async();
      mbar_arrive(smem_u32(&p_ready));
      mbar_arrive(smem_u32(&c_ready[sb]));
    }
    l_s[tl] = l;
    mbar_arrive(smem_u32(&l_ready));
  } else {
    // ---------------- output: one thread per row, all dims in registers
    float o[HD];
#pragma unroll
    for (int i = 0; i < HD; ++i) o[i] = 0.f;
    for (int j = 0; j < n_blocks; ++j) {
      const int ob = j & 1;
      bool ok = mbar_wait(smem_u32(&c_ready[ob]), (uint32_t)(j >> 1) & 1u, &abort_flag);
      ok = ok && mbar_wait(smem_u32(&o_full[ob]), (uint32_t)(j >> 1) & 1u, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { failed = true; break; }
      const float corr = corr_s[ob][tl];
      const float f_old = signbit(corr) ? 1.f : corr, f_new = signbit(corr) ? -corr : 1.f;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < HD / 8; ++c) {
        uint32_t v[8];
        tmem_ld8(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(256 + ob * 128 + 8 * c), v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) o[8 * c + i] = fmaf(o[8 * c + i], f_old, __uint_as_float(v[i]) * f_new);
      }
      tc_fence_before();
      mbar_arrive(smem_u32(&o_free[ob]));
    }
    bool ok = !failed && mbar_wait(smem_u32(&l_ready), 0u, &abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    if (ok && real) {
      const float inv = 1.f / l_s[tl];
      const size_t at = ((size_t)(row0 + tl / GROUP) * nq + (size_t)g * GROUP + tl % GROUP) * HD;
#pragma unroll
      for (int c = 0; c < HD / 8; ++c) {
        __nv_bfloat16 a[8], b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float y = o[8 * c + i] * inv;
          a[i] = __float2bfloat16_rn(y);
          b[i] = __float2bfloat16_rn(y - __bfloat162float(a[i]));
        }
        *reinterpret_cast<uint4 *>(out_hi + at + 8 * c) = *reinterpret_cast<const uint4 *>(a);
        *reinterpret_cast<uint4 *>(out_lo + at + 8 * c) = *reinterpret_cast<const uint4 *>(b);
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

template <int HD, int GROUP>
cudaError_t pf_prepare() {
  return cudaFuncSetAttribute(attn_prefill_kernel<HD, GROUP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PfLayout<HD>::SMEM);
}

}  // namespace

cudaError_t attention_prefill_prepare() {
  cudaError_t e = cudaSuccess;
  for (auto prepare : {pf_prepare<128, 1>, pf_prepare<128, 2>, pf_prepare<128, 4>, pf_prepare<128, 8>, pf_prepare<64, 1>, pf_prepare<64, 2>,
                       pf_prepare<64, 4>, pf_prepare<64, 8>})
    if (e == cudaSuccess) e = prepare();
  return e;
}

cudaError_t launch_attention_prefill(const CUtensorMap &tmKV, const float *q, const Rows &rows, int nq, const KvLayout &kv,
                                     __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, int *d_status, cudaStream_t st) {
  const int group = nq / kv.n_kv;
  if (group * kv.n_kv != nq) return cudaErrorInvalidValue;
  if (group != 1 && group != 2 && group != 4 && group != 8) return cudaErrorInvalidValue;
  const int tpt = 128 / group;
  const dim3 grid(kv.n_kv, (rows.R + tpt - 1) / tpt);
#define CORUN_PF_CASE(HD_, G_) \
  if (kv.hd == HD_ && group == G_)   \
    return launch_k(attn_prefill_kernel<HD_, G_>, grid, dim3(PF_THREADS), PfLayout<HD_>::SMEM, st, true, tmKV, q, rows, nq, kv, out_hi, out_lo, d_status);
  CORUN_PF_CASE(128, 1) CORUN_PF_CASE(128, 2) CORUN_PF_CASE(128, 4) CORUN_PF_CASE(128, 8)
  CORUN_PF_CASE(64, 1) CORUN_PF_CASE(64, 2) CORUN_PF_CASE(64, 4) CORUN_PF_CASE(64, 8)
#undef CORUN_PF_CASE
  return cudaErrorInvalidValue;
}

}  // namespace corun
