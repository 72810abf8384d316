// Causal attention of a prefill chunk: the chunk's rows are consecutive tokens of ONE request, so a tile of
// query rows shares every key / value tile it reads (the decode kernel reads them once per query row).
//
// One CTA per (tile of 128 / G consecutive tokens, kv head), G = query heads per kv head.  The 128 rows of the tile are the
// (token, head) pairs; row m = token m / G, head m % G.  It walks the blocks of 128 cached tokens (8 pages) from position 0
// to the tile's last token once:
//   S[128 rows x 128 keys] = Q * K^T on tcgen05.mma (M = 128, N = 128, fp16, Q as a hi/lo pair: two MMAs per k-slice) into
//     one of two TMEM buffers;
//   softmax warps, a thread per row (TMEM lane = row): P = exp2(S - the block's own maximum) as fp16 into one of two TMEM buffers
//     of 64 columns (causal mask: key position <= the row's own position), and the block's maximum and sum;
//   O'[128 x hd] = P * V, P from tensor memory, one MMA per page, into one of two (hd 128: the one) TMEM buffers;
//   output warps, a thread per row and half of the dims: the factor between this block's scale and the earlier ones', O and O' to
//     the larger of the two maxima and added, in registers; at the end O / sum -> bf16 hi/lo.
// A block's largest weight is exactly 1 in fp16 and the factors are fp32, so the keys that carry a row have unrounded weights
// (relative to the running maximum only one of them did: prompts of 300 / 1003 tokens through 12 Qwen3-8B layers were
// 1.1e-4 / 6.7e-5 off a 64-bit evaluation).
// Weights relative to the block's own maximum also make the blocks' softmax independent of each other: two groups of four warps take
// the even and the odd blocks, so that one block's loads, maxima and exponentials run beside the other's and beside the MMAs (24 of
// 64 cycles per block, beside 1024 cycles of exponentials and 1650 of TMA: 16 boxes of 4 KB at 103).
// Measured per layer of the Qwen3-8B shape, this kernel / one softmax group with weights through shared memory, a thread per row
// for queries and results: 77 tokens 9.5 / 15.7 us, 1003 tokens 29.8 / 41.3, 6001 tokens 610 / 830.
// MMAs on different accumulators may overtake one another, so none writes what another one may still read: a block's scores,
// weights and output have places of their own.  Scores of block j + 2 overwrite those of block j, which the softmax has read when it
// hands over its weights; the weights of block j + 2 are written behind the commit of its scores, which are issued behind the
// values of block j and so complete no earlier; the one output buffer of hd 128 is read while the scores of block j + 2 are
// multiplied.
// Roles: warps 0-3 and 4-7 softmax, 8-11 and 12-15 output, warp 16 streams the keys and warp 17 the values with TMA (rings of two; one
// 4-dimensional box per (page, head) tile), warp 18 issues the MMAs.
//
// A page's keys land as [2 groups of 8 tokens][hd / 64][8 tokens][64 dims]: for the scores a K-major operand whose groups of
// eight rows lie hd / 64 KiB apart, for the values (cached alike) an MN-major one.
//
// Every reduction has one fixed order (per thread: four interleaved partial sums over a block's keys in ascending order, then
// a fixed tree; blocks ascending) that depends on the row's own position only.  All waits are bounded.
#include <cuda_fp16.h>
#include <math_constants.h>
#include <type_traits>

#include "launch.cuh"
#include "ops.cuh"
#include "ptx.cuh"

namespace corun {

namespace {

constexpr int PF_THREADS = 608;
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
  static constexpr int PAGE_BYTES = NHALF * KV_BLOCK * 128;   // one page's keys (values) of one head
  static constexpr int B_BYTES = PF_PAGES * PAGE_BYTES;       // a block of keys (values)
  static constexpr int O_BUFS = HD == 64 ? 2 : 1;             // of the 512 columns: 2 x 128 scores, 2 x 64 weights, 128 output
  static constexpr uint32_t P_COL = 256, O_COL = 384;
  static constexpr size_t SMEM = (size_t)2 * Q_BYTES + 2 * PF_RING * B_BYTES + 1024;
};

template <int HD, int GROUP>
__global__ void __launch_bounds__(PF_THREADS, 1)
attn_prefill_kernel(const __grid_constant__ CUtensorMap tmKV, const float *__restrict__ q, Rows rows, int nq, KvLayout kv,
                    __nv_bfloat16 *__restrict__ out_hi, __nv_bfloat16 *__restrict__ out_lo, int *status) {
  using L = PfLayout<HD>;
  constexpr int TPT = 128 / GROUP;                  // tokens per tile
  constexpr int KSTEPS = HD / 16, O_BUFS = L::O_BUFS;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t kfull[PF_RING], kempty[PF_RING], vfull[PF_RING], vempty[PF_RING], s_full[2], p_ready[2], o_full[O_BUFS],
      o_free[O_BUFS], c_ready[4];
  __shared__ float max_s[4][128], sum_s[4][128];    // a block's maximum and sum per row, four blocks in turn
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // heads fastest, the last tiles (the most key blocks) first: the short ones fill the last wave
  const int tile = (int)gridDim.y - 1 - (int)blockIdx.y, g = blockIdx.x, row0 = tile * TPT;
  if (tid == 0) {                                   // (ahead of the wait: touches nothing that another kernel writes)
    abort_flag = 0;
    for (int i = 0; i < PF_RING; ++i) {
      mbar_init(smem_u32(&kfull[i]), 1); mbar_init(smem_u32(&kempty[i]), 1);
      mbar_init(smem_u32(&vfull[i]), 1); mbar_init(smem_u32(&vempty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&s_full[i]), 1);           // scores in TMEM
      mbar_init(smem_u32(&p_ready[i]), 128);        // every row thread has read them and written its weights
    }
    for (int i = 0; i < O_BUFS; ++i) {
      mbar_init(smem_u32(&o_full[i]), 1); mbar_init(smem_u32(&o_free[i]), 256);   // a block's output in TMEM / read by both groups
    }
    for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&c_ready[i]), 128);            // the rows' maxima and sums of a block
    fence_mbar_init();
    fence_proxy_async();
    prefetch_tensormap(&tmKV);
  }
  griddep_wait();                                   // q and the chunk's own keys / values come from the kernel before
  q = after_wait(q);
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
  const uint32_t q_hi = base, q_lo = base + L::Q_BYTES, k_ring = q_lo + L::Q_BYTES, v_ring = k_ring + PF_RING * L::B_BYTES;
  bool failed = false;
  // producers: lane l fetches page l of a block, its page number read one block ahead of its use
  const int *table = kv.block_table + (size_t)slot * kv.max_blocks;
  const bool keys = warp == 16;
  int page_next = 0;
  auto fetch = [&](int j) {
    const int buf = j % PF_RING, n_pages = pages_of(j), page = page_next;
    if (j + 1 < n_blocks) page_next = lane < pages_of(j + 1) ? table[(j + 1) * PF_PAGES + lane] : 0;
    if (j >= PF_RING) {
      bool ok = mbar_wait(smem_u32(keys ? &kempty[buf] : &vempty[buf]), (uint32_t)(j / PF_RING - 1) & 1u, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { failed = true; return; }
    }
    const uint32_t fb = smem_u32(keys ? &kfull[buf] : &vfull[buf]);
    if (lane == 0) mbar_arrive_expect_tx(fb, (uint32_t)(n_pages * L::PAGE_BYTES));
    __syncwarp();
    if (lane < n_pages)                             // the page's (head) tile in one box; the last dimension counts groups of 8 tokens
      tma_load_4d((keys ? k_ring : v_ring) + (uint32_t)(buf * L::B_BYTES + lane * L::PAGE_BYTES), &tmKV, 0, 0, 0,
                  (page * 2 * kv.n_kv + (keys ? 0 : kv.n_kv) + g) * (KV_BLOCK / 8), fb, l2_policy_evict_last());   // the tiles of the same request read the same cache rows
  };
  if (warp == 18) {
    tmem_alloc(smem_u32(&tmem_base_s), 512);        // (PfLayout)
    tmem_relinquish();
  } else if (warp >= 16) {
    page_next = lane < pages_of(0) ? table[lane] : 0;
    for (int j = 0; j < n_blocks && j < PF_RING; ++j) fetch(j);   // beside the query tile
  } else {
    // ---- the query tile: row m = (token m / G, head m % G) as fp16 hi and lo tiles (q = hi + lo).  A row is HD / 4 lanes, so that a
    // warp reads 512 contiguous bytes (a thread per row: 5.9 us of the 13.4 of a tile with one block of keys)
    constexpr int LPR = HD / 4, RPW = 32 / LPR;     // lanes per row, rows of a warp at a time
    const int d = 4 * (lane % LPR);
    float4 v[8 / RPW];
#pragma unroll
    for (int k = 0; k < 8 / RPW; ++k) {
      const int m = RPW * (warp + 16 * k) + lane / LPR, t = m / GROUP;
      v[k] = row0 + t < rows.R ? *reinterpret_cast<const float4 *>(q + ((size_t)(row0 + t) * nq + (size_t)g * GROUP + m % GROUP) * HD + d)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 8 / RPW; ++k) {
      const int m = RPW * (warp + 16 * k) + lane / LPR;
      const float x[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
      __half hi[4], lo[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        hi[i] = __float2half_rn(x[i]);
        lo[i] = __float2half_rn(x[i] - __half2float(hi[i]));
      }
      const uint32_t off = (uint32_t)(d >> 6) * (128 * 128) + pf_swz(m, (d & 63) >> 3) + (uint32_t)((d & 4) * 2);
      *reinterpret_cast<uint2 *>(base_ptr + off) = *reinterpret_cast<const uint2 *>(hi);
      *reinterpret_cast<uint2 *>(base_ptr + L::Q_BYTES + off) = *reinterpret_cast<const uint2 *>(lo);
    }
    fence_proxy_async();                            // the MMAs read these tiles through the async proxy
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  // warps 0-15: this thread's row
  const int quad = warp & 3, tl = quad * 32 + lane;
  const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
  const bool real = tl / GROUP < n_tok;

  if (warp == 16 || warp == 17) {
    // ---------------- producers
    for (int j = PF_RING; j < n_blocks && !failed; ++j) fetch(j);
  } else if (warp == 18) {
    // ---------------- MMA issuer: the values of block j, then the scores of block j + 2
    if (elect_one()) {
      // fp16 x fp16 -> fp32; N at bit 17 (>> 3), M = 128 at bit 24 (>> 4); the values are an MN-major B operand
      const uint32_t idesc_s = (1u << 4) | ((uint32_t)(PF_KEYS >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      const uint32_t idesc_o = (1u << 4) | (1u << 16) | ((uint32_t)(HD >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      auto scores = [&](int j) {
        const int buf = j % PF_RING, sb = j & 1;
        if (!mbar_wait(smem_u32(&kfull[buf]), (uint32_t)(j / PF_RING) & 1u, &abort_flag)) { failed = true; return; }
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
      };
      scores(0);
      if (n_blocks > 1 && !failed) scores(1);
      for (int j = 0; j < n_blocks && !failed; ++j) {
        const int buf = j % PF_RING, b = j & 1, ob = j % O_BUFS;
        if (!mbar_wait(smem_u32(&p_ready[b]), (uint32_t)(j >> 1) & 1u, &abort_flag)) { failed = true; break; }
        if (!mbar_wait(smem_u32(&vfull[buf]), (uint32_t)(j / PF_RING) & 1u, &abort_flag)) { failed = true; break; }
        if (j >= O_BUFS && !mbar_wait(smem_u32(&o_free[ob]), (uint32_t)(j / O_BUFS - 1) & 1u, &abort_flag)) { failed = true; break; }
        tc_fence_after();
        const int n_pages = pages_of(j);
        const uint32_t vt = v_ring + (uint32_t)(buf * L::B_BYTES), p = tmem + L::P_COL + (uint32_t)b * 64,
                       d = tmem + L::O_COL + (uint32_t)(ob * HD);
        for (int i = 0; i < n_pages; ++i)           // 16 tokens of weights are 8 columns
          umma_f16_ts(d, p + (uint32_t)(8 * i), umma_desc_sw128_mn(vt + (uint32_t)(i * L::PAGE_BYTES), 1024u, L::NHALF * 1024u), idesc_o, i > 0 ? 1u : 0u);
        umma_commit(smem_u32(&vempty[buf]));
        umma_commit(smem_u32(&o_full[ob]));
        if (j + 2 < n_blocks) scores(j + 2);
      }
    }
  } else if (warp < 8) {
    // ---------------- softmax: one thread per row; warps 0-3 the even blocks, warps 4-7 the odd ones
    const int pos = real ? rows.pos[row0 + tl / GROUP] : -1;       // keys 0..pos are visible to this row
    const float sscale = (HD == 128 ? 0.08838834764831845f : 0.125f) * 1.4426950408889634f;   // log2(e)/sqrt(hd)
    const int sb = warp >> 2;
    const uint32_t st = t_lane + (uint32_t)(sb * 128), pt = t_lane + L::P_COL + (uint32_t)(sb * 64);
    for (int j = sb; j < n_blocks; j += 2) {
      bool ok = mbar_wait(smem_u32(&s_full[sb]), (uint32_t)(j >> 1) & 1u, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { failed = true; break; }
      tc_fence_after();
      const int lim = pos - j * PF_KEYS;            // keys 0 .. lim of the block are visible
      // the scores twice, 16 at a time, the next ones requested ahead: first their maximum, then the weights.  (No branch ends
      // between a load and its wait.)
      float bm, acc[4] = {0.f, 0.f, 0.f, 0.f};
      auto block = [&](auto masked) {
        constexpr bool M = decltype(masked)::value;
        uint32_t v[2][16];
        float m4[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
        tmem_ld16(st, v[0]);
        auto largest = [&](const uint32_t (&x)[16], int left) {
#pragma unroll
          for (int i = 0; i < 16; ++i) m4[i & 3] = fmaxf(m4[i & 3], M && i > left ? -CUDART_INF_F : __uint_as_float(x[i]));
        };
#pragma unroll 1
        for (int c = 0; c < 8; c += 2) {            // (small code: a tile of a short prompt runs it once, from a cold instruction cache)
          tmem_ld_wait();
          tmem_ld16(st + (uint32_t)(16 * c + 16), v[1]);
          largest(v[0], lim - 16 * c);
          tmem_ld_wait();
          tmem_ld16(st + (uint32_t)((16 * c + 32) & 127), v[0]);     // (the last one begins the second pass)
          largest(v[1], lim - 16 * c - 16);
        }
        bm = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * sscale;
        const float ref = bm == -CUDART_INF_F ? 0.f : bm;            // (nothing visible in this block: all its weights are 0)
        auto weights = [&](const uint32_t (&x)[16], int left, uint32_t at) {
          uint32_t w[8];
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            float p0 = ex2_approx(fmaf(__uint_as_float(x[i]), sscale, -ref));
            float p1 = ex2_approx(fmaf(__uint_as_float(x[i + 1]), sscale, -ref));
            if (M && i > left) p0 = 0.f;
            if (M && i + 1 > left) p1 = 0.f;
            acc[i & 3] += p0;
            acc[(i + 1) & 3] += p1;
            const __half2 h2 = __floats2half2_rn(p0, p1);
            w[i >> 1] = *reinterpret_cast<const uint32_t *>(&h2);
          }
          tmem_st8(at, w);
        };
#pragma unroll 1
        for (int c = 0; c < 8; c += 2) {
          tmem_ld_wait();
          tmem_ld16(st + (uint32_t)(16 * c + 16), v[1]);
          weights(v[0], lim - 16 * c, pt + (uint32_t)(8 * c));
          tmem_ld_wait();
          tmem_ld16(st + (uint32_t)(c < 6 ? 16 * c + 32 : 112), v[0]);   // (the last one is not used)
          weights(v[1], lim - 16 * c - 16, pt + (uint32_t)(8 * c + 8));
        }
        tmem_ld_wait();
      };
      // only a row's last block (or padding) needs the mask
      if (__any_sync(0xffffffffu, lim < PF_KEYS - 1)) block(std::true_type{});
      else block(std::false_type{});
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(smem_u32(&p_ready[sb]));
      // (block j - 4's have been read: its output was, before the scores of this block were issued)
      max_s[j & 3][tl] = bm;
      sum_s[j & 3][tl] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
      mbar_arrive(smem_u32(&c_ready[j & 3]));
    }
  } else {
    // ---------------- output: one thread per row and half of the dims, in registers
    constexpr int HH = HD / 2;
    const int dh = (warp - 8) >> 2;
    float o[HH], mx = -CUDART_INF_F, l = 0.f;
#pragma unroll
    for (int i = 0; i < HH; ++i) o[i] = 0.f;
    for (int j = 0; j < n_blocks; ++j) {
      const int ob = j % O_BUFS;
      bool ok = mbar_wait(smem_u32(&c_ready[j & 3]), (uint32_t)(j >> 2) & 1u, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { failed = true; break; }
      // the larger maximum is the scale from here on: a factor for the sums so far, or for this block
      const float bm = max_s[j & 3][tl], sum = sum_s[j & 3][tl], ref = bm == -CUDART_INF_F ? 0.f : bm;
      const bool up = bm >= mx;
      const float factor = ex2_approx(up ? mx - ref : bm - mx);
      mx = fmaxf(mx, bm);
      l = up ? fmaf(l, factor, sum) : fmaf(sum, factor, l);
      const float f_old = up ? factor : 1.f, f_new = up ? 1.f : factor;
      ok = mbar_wait(smem_u32(&o_full[ob]), (uint32_t)(j / O_BUFS) & 1u, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { failed = true; break; }
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < HH / 16; ++c) {
        uint32_t v[16];
        tmem_ld16(t_lane + L::O_COL + (uint32_t)(ob * HD + dh * HH + 16 * c), v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) o[16 * c + i] = fmaf(o[16 * c + i], f_old, __uint_as_float(v[i]) * f_new);
      }
      tc_fence_before();
      mbar_arrive(smem_u32(&o_free[ob]));
    }
    // bf16 hi / lo through the query tiles' shared memory (all MMAs have read them), then whole rows (a thread per row: 4 us)
    constexpr int CH = HD / 8;                      // 16-byte pieces of a row
    auto at = [&](int row, int c) { return (uint32_t)(row * HD * 2 + ((c ^ (row & 7)) << 4)); };
    const float inv = 1.f / l;                      // (rows without a token: not stored)
#pragma unroll
    for (int c = 0; c < CH / 2; ++c) {
      __nv_bfloat16 a[8], b[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float y = o[8 * c + i] * inv;
        a[i] = __float2bfloat16_rn(y);
        b[i] = __float2bfloat16_rn(y - __bfloat162float(a[i]));
      }
      *reinterpret_cast<uint4 *>(base_ptr + at(tl, dh * (CH / 2) + c)) = *reinterpret_cast<const uint4 *>(a);
      *reinterpret_cast<uint4 *>(base_ptr + L::Q_BYTES + at(tl, dh * (CH / 2) + c)) = *reinterpret_cast<const uint4 *>(b);
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");  // warps 8-15 (whatever failed)
    if (!failed) {
#pragma unroll
      for (int k = 0; k < 128 * CH / 256; ++k) {
        const int u = k * 256 + tid - 256, row = u / CH, c = u % CH;
        if (row / GROUP < n_tok) {
          const size_t to = ((size_t)(row0 + row / GROUP) * nq + (size_t)g * GROUP + row % GROUP) * HD + 8 * c;
          *reinterpret_cast<uint4 *>(out_hi + to) = *reinterpret_cast<const uint4 *>(base_ptr + at(row, c));
          *reinterpret_cast<uint4 *>(out_lo + to) = *reinterpret_cast<const uint4 *>(base_ptr + L::Q_BYTES + at(row, c));
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
  if (warp == 18) tmem_dealloc(tmem, 512);
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
