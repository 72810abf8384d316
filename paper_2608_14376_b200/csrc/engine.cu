// Host side of the C ABI: engine state, paged KV pool, the row program
// (decode graph / eager prefill) and the debug accessors.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/corun.h"
#include "../../include/corun_debug.h"
#include "gemm.cuh"
#include "mla.cuh"
#include "moe.cuh"
#include "ops.cuh"

using namespace corun;


#define CK(call)                                   \
  do {                                             \
    cudaError_t _e = (call);                       \
    if (_e != cudaSuccess) {                       \
      g_last_cuda_error = (int)_e;                 \
      return CORUN_ECUDA;                          \
    }                                              \
  } while (0)
#define RC(call)                  \
  do {                            \
    int _r = (call);              \
    if (_r != CORUN_OK) return _r; \
  } while (0)

namespace {

typedef __nv_bfloat16 bf16;

// Device memory of one owner, handed out from a few blocks: an allocation of a few MB or more costs 0.35 ms whatever its
// size, and an engine has some sixty buffers.
struct DevMem {
  std::vector<void *> blocks;
  char *cur = nullptr;
  size_t left = 0, next = (size_t)32 << 20;
  // Room for `bytes` in one block of that size, if there is as much: what follows fits it and leaves nothing over.
  void reserve(size_t bytes) {
    void *q = nullptr;
    if (cudaMalloc(&q, bytes) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    blocks.push_back(q);
    cur = (char *)q;
    left = bytes;
  }
  void release() {
    for (void *p : blocks) cudaFree(p);
    blocks.clear();
    cur = nullptr;
    left = 0;
  }
};

// Buffers and GEMM plans of the row program at one fixed row count.
struct Program {
  int R = 0, BN = 0;
  float *h = nullptr, *q = nullptr, *part_acc = nullptr, *part_ml = nullptr;
  float *qkv_out = nullptr, *o_out = nullptr, *gu_out = nullptr, *down_out = nullptr, *logits = nullptr, *ws = nullptr;
  bf16 *xn_hi = nullptr, *xn_lo = nullptr, *ao_hi = nullptr, *ao_lo = nullptr, *ff_hi = nullptr, *ff_lo = nullptr;
  int *row_token = nullptr, *row_pos = nullptr, *row_active = nullptr, *row_slot = nullptr, *do_sample = nullptr;
  int *row_blocks = nullptr;   // decode program: which blocks of rows hold a request this step (GemmPlan::row_blocks)
  // decode program: the step's rows are the slots with a request first (prepare_rows); the slot's row, and the
  // slots' sampling state at the rows' places
  int *slot_row = nullptr, *row_step = nullptr;
  float *row_temp = nullptr, *row_top_p = nullptr;
  int *sampled = nullptr, *att_work = nullptr, *att_n_work = nullptr, *att_pool = nullptr;
  GemmPlan p_qkv, p_o, p_gu, p_down, p_lm;
  // Mixture-of-Experts feed-forward layers: p_gu / p_down are then the GEMMs over all experts' gate / up rows
  // and over the concatenated hidden activations; moe_w the rows' routing weights
  float *moe_w = nullptr;
  RouterScratch router_rs{};
  // selected-experts form (decode up to 64 rows): only the experts that a row selected are streamed; p_gug / p_dng are its
  // GEMMs, hg / yg hold [expert][BN] rows, moe_sel every row's experts.  Measured per step, 12 layers of the Qwen3-30B-A3B
  // shape, against every row through every expert: 1 row of 1 2.84 -> 0.99 ms, 8 of 8 2.95 -> 1.72, 16 of 32 3.05 -> 2.38, 20 of 64
  // 3.28 -> 2.60, 40 of 64 3.50 -> 3.44, 64 of 64 (nearly all experts selected) 3.76 -> 3.95.
  bool select = false;
  int *moe_sel = nullptr;
  // grouped form of the experts' GEMMs: the rows of an expert gathered into blocks of 64 (prompts: of 128, on pairs of SMs)
  bool grouped = false;
  MoeGroups grp{};
  GemmPlan p_gug, p_dng;
  GemmExpertsPlan x_gu, x_down;          // (prompts: blocks of 128)
  bf16 *xg_hi = nullptr, *xg_lo = nullptr, *hg_hi = nullptr, *hg_lo = nullptr;
  float *gug_out = nullptr, *yg_out = nullptr;
  int *plain_tiles = nullptr;            // zeros: the table that makes a plain matrix readable as a GEMM result
  // multi-head latent attention: head-major matrices of RPH rows per head for the grouped up-projections
  // (p_uk: q_lat = W_uk^T q_nope; p_uv: [. | o] = W_kv_b o_lat), the attention's partials, and the dense
  // feed-forward GEMMs of the layers that have no experts
  int RPH = 0;
  bf16 *qn_hi = nullptr, *qn_lo = nullptr, *ol_hi = nullptr, *ol_lo = nullptr;
  float *q_lat = nullptr, *q_rope = nullptr, *uv_out = nullptr, *mla_po = nullptr;
  float2 *mla_ml = nullptr;
  int *tab_uk = nullptr, *tab_uv = nullptr;
  GemmPlan p_uk, p_uv, p_gu_d, p_down_d;
  bool has_layers = false, has_lm = false;
  // Prefill: up to `cap` rows at a time (R: the rows of the chunk at hand).  Long prompts: the projections on pairs of SMs
  // (gemm_pair.cu), their results plain matrices, the SwiGLU in the gate / up GEMM's epilogue.  Short prompts (shorts): the
  // dense projections in blocks of SHORT_ROWS rows through the decode GEMM (s_*: one plan per block, blocks of 64 rows
  // without a row left out), the token-wise kernels behind a projection block by block; attention and experts over all
  // rows as for long ones.
  bool pair = false;
  int cap = 0;
  // Decode above 128 rows (wide): the dense projections and the LM head on pairs of SMs too, with expert layers from 129 rows
  // on, else from WIDE_ROWS rows on: below, the fixed cost of a pair GEMM (clusters, no programmatic launch; 15 us for the
  // matrices of the hidden-1024 decoder) outweighs what the steps of more than 128 requests save.
  // ms per step of 12 layers, one-SM GEMMs / pairs, at three counts of requests: Qwen3-8B 140 slots (25, 125, 139 requests)
  // 2.44 2.91 3.79 / 2.61 3.03 3.61, 200 slots (30, 128, 200) 2.69 3.36 4.75 / 2.65 3.26 4.39, 256 slots (40, 128, 256) 2.87 3.38
  // 5.33 / 2.73 3.17 4.82; hidden 1024 140 slots .99 1.28 1.53 / 1.09 1.39 1.55, 200 slots 1.03 1.33 1.84 / 1.10 1.41 1.76, 256
  // slots (25, 128, 256) 1.06 1.36 2.17 / 1.10 1.41 1.87; Qwen3-30B-A3B 140 slots (25, 128, 139) 3.51 4.50 4.88 / 3.46 4.44 4.71.
  bool wide = false;
  GemmPairPlan b_lm;
  bool shorts = false;
  std::vector<GemmPlan> s_qkv, s_o, s_gu, s_down;
  GemmPairPlan b_qkv, b_o, b_gu, b_down, b_router;
  float *router_out = nullptr, *pair_part = nullptr;
  size_t pair_part_floats = 0;           // (decode) room of pair_part
  // Latent attention of long prompts over decompressed keys and values (attention_prefill_mla.cu): the gathered latents of
  // the chunk's requests, up to kv_cap tokens, their keys and values, and the chunk's segments
  bool mla_tiles = false;
  int kv_cap = 0, kv_tokens = 0;
  GemmPairPlan b_kv;
  bf16 *c_hi = nullptr, *c_lo = nullptr;
  __half *kr = nullptr, *kvd = nullptr;
  int *tile_base = nullptr;
  CUtensorMap tm_kvd, tm_kr;
  MlaSegs segs{};
  uint32_t *moe_mask = nullptr;
  DevMem allocs;
};

// Prompts of up to PREFILL_SMALL tokens are short (Program::shorts), longer ones long.  Which one depends on the prompt's
// own length only, so a prompt's values do not depend on what is prefilled with it.  Prompts of 65 / 96 / 128 / 160 / 192 / 256 tokens
// through 12 Qwen3-8B layers: 1.63 / 1.75 / 2.0 / 3.1 / 3.25 / 3.75 ms in blocks of SHORT_ROWS, 2.55 / 2.43 / 2.56 / 2.6 / 2.7 / 2.8 on
// pairs of SMs.  There GEMMs of a Qwen3-8B layer take 299 us for 512 rows, 543 for 1024 and 1049 for 2048, hence chunks as large as the
// buffers allow.  PREFILL_BIG 2048 -> 4096: 3000 tokens through 12 Qwen3-30B-A3B layers 15.1 -> 12.7 ms, 2505 through 9 DeepSeek-V2-Lite
// layers 12.1 -> 9.9 (one pass over the experts and not two); prompts one behind the other through 12 Qwen3-8B layers, 2500 / 4096 /
// 6001 tokens 21.9 / 34.5 / 53.3 -> 20.3 / 33.8 / 52.7.
constexpr int PREFILL_SMALL = 128, PREFILL_BIG = 4096;
// Rows of a long prompt's chunk that the latent attention takes at a time (its partial results are kept per row).
constexpr int MLA_ROWS = 256;
constexpr int SHORT_ROWS = 128;
constexpr int WIDE_ROWS = 192;               // see Program::wide
static_assert(PREFILL_BIG <= MOE_MANY_ROWS, "a chunk of a long prompt is grouped in one go");
// (a request of a long prompt's chunk begins on a tile of 128 rows and has more than one, but for the first and the last)
static_assert(PREFILL_BIG / 256 + 1 <= MLA_MAX_SEGS, "latent attention gathers all requests of a chunk");
static_assert(PREFILL_BIG / SHORT_ROWS <= 32, "the staging buffer holds 32 blocks and 32 tiles");
// corun_get_logits: a row goes to the host by way of pinned memory, from LOGITS_SPLIT values on in two pieces, the first copied
// on to the caller while the second arrives.  A piece costs some 3 us of calls.  A call for 151936 / 102400 / 32000 values: 60 /
// 48 / 30 us straight into the caller's pageable memory, 59 / 38 / 20 in one piece, 54 / 37 / 21 in two, 55 / 41 / 27 in four.
constexpr int LOGITS_PIECES = 2, LOGITS_SPLIT = 65536;

}  // namespace

struct corun_engine {
  corun_shape sh{};
  int B = 0, max_ctx = 0, max_blocks = 0, max_splits = 0, chunk = 0, num_sms = 0;
  int whole_pairs = 0;               // ablation: attention without parallelism inside a (row, kv head) pair
  int64_t pool_blocks = 0;
  cudaStream_t st = nullptr;
  bool own_stream = false;
  const void *w0_qkv = nullptr, *w0_o = nullptr, *w0_gu = nullptr, *w0_down = nullptr;
  // borrowed weights
  const bf16 *embed = nullptr, *lm_head = nullptr, *final_norm = nullptr;
  std::vector<const bf16 *> attn_norm, mlp_norm;
  std::vector<CUtensorMap> tm_qkv, tm_o, tm_gu, tm_down;
  std::vector<CUtensorMap> tb_qkv, tb_o, tb_gu, tb_down, tb_router, tb_gu96, tb_uv;   // boxes of 128 rows (96): the GEMMs on pairs of SMs
  CUtensorMap tb_lm;
  std::vector<CUtensorMap> tb_gu_half;     // dense layers of a decoder with expert layers: the box of the GEMM with SwiGLU
  std::vector<CUtensorMap> tm_gu_half;     // dense gate / up matrices with the box of the GEMM with SwiGLU in its epilogue
  std::vector<CUtensorMap> tm_k4;        // per layer: the pages (keys and values alike) as [8-token group][64-dim half][8 tokens][64 dims]: one box per (page, head) tile
  // Mixture-of-Experts feed-forward layers (E = 0: dense).  sh.ffn is then (E + S) * F.
  int moe_E = 0, moe_K = 0, moe_F = 0, moe_S = 0, moe_renorm = 0;
  std::vector<const bf16 *> router;      // per layer: [E, H], borrowed
  // multi-head latent attention (corun_init_mla): sh.head_dim is the value width, the cache holds rank + rope
  // halfs per token; layers below first_dense have a dense feed-forward of width dense_ffn
  bool mla = false;
  MlaDims md{};
  int first_dense = 0, dense_ffn = 0, mla_splits = 0;
  bool wide = false;                     // Program::wide of the decode program
  bool big_mla_tiles = false;            // Program::mla_tiles of the prefill program
  std::vector<const bf16 *> kv_norm;
  bf16 *w_ukT = nullptr;                 // [L][nh * rank][nope]: the key up-projections transposed
  float2 *kv_scale = nullptr;            // [L][nh]: scales of decompressed keys and values (launch_mla_kv_scale)
  std::vector<CUtensorMap> tm_uk, tm_uv, tm_c, tm_cv, tm_gu_d, tm_down_d;
  const void *w0_uv = nullptr, *w0_gu_d = nullptr, *w0_down_d = nullptr;
  // KV
  __half *kv_pool = nullptr;
  size_t layer_stride = 0;
  int *d_block_table = nullptr;
  // Pages are handed out in aligned runs of kv_run consecutive pool pages (1; 4 for latent caches created with
  // kv_block = 64: the latent attention kernel then fetches a run with one TMA box).  free_blocks / slot_blocks hold
  // RUN indices; the block table holds pages (run * kv_run + i).
  int kv_run = 1;
  std::vector<int> free_blocks;
  std::vector<std::vector<int>> slot_blocks;
  float2 *d_rope = nullptr;
  // slot state: device
  int *d_in_use = nullptr, *d_ctx = nullptr, *d_step = nullptr, *d_pending = nullptr;
  float *d_temp = nullptr, *d_top_p = nullptr;
  float *pf_logits = nullptr;            // [B, vocab]: a slot's logits after its prefill (the decode logits are by row)
  std::vector<int> logits_row;           // per slot: its row of the last decode step it took part in, -1 = pf_logits
  uint64_t *d_seeds = nullptr;
  uint8_t *d_active = nullptr;
  int *d_out_tokens = nullptr, *d_status = nullptr;
  // slot state: host mirrors
  std::vector<int> in_use, ctx, reserve, step;
  // pinned staging (one allocation)
  void *h_pinned = nullptr;
  uint8_t *h_active = nullptr;
  uint64_t *h_seeds = nullptr;
  int *h_out_tokens = nullptr, *h_status = nullptr;
  int *h_rows = nullptr;          // prefill staging: rows [4][chunk], blocks of rows, group tables of the latent projections
  int *h_table = nullptr;         // [B][max_blocks]: the block table as it was last sent (a slot's row changes only while it is free)
  int *h_first = nullptr;         // [B]: first tokens of a prefill call's requests
  float *h_logits = nullptr;      // [vocab]: a row of logits on its way to the caller
  cudaEvent_t ev_logits[LOGITS_PIECES] = {};
  bool staged_valid = false, in_flight = false;
  Program dec, pre, big, lm1;
  // prefill-only per-row sampling arrays (length FINISH_ROWS)
  float *d_pf_temp = nullptr, *d_pf_top_p = nullptr;
  uint64_t *d_pf_seed = nullptr;
  int *d_pf_step = nullptr, *d_pf_one = nullptr, *d_pf_tok = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t graph_exec = nullptr;
  bool eager = false;
  unsigned long long *step_trace = nullptr;   // debug (CORUN_TRACE_STEP=1): GEMM timelines of a whole step
  int stop_after = -1;            // debug: eager decode stops after this many stages of layer 0
  int decode_launches = 0;
  DevMem allocs;
};

namespace {

template <typename T>
int dmalloc(std::vector<void *> &keep, T **p, size_t n, bool zero = true) {
  void *q = nullptr;
  if (n == 0) n = 1;
  cudaError_t e = cudaMalloc(&q, n * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();                             // (handled here: not the error of the next launch)
    g_last_cuda_error = (int)e;
    return CORUN_ENOMEM;
  }
  keep.push_back(q);
  if (zero && cudaMemset(q, 0, n * sizeof(T)) != cudaSuccess) return CORUN_ECUDA;
  *p = (T *)q;
  return CORUN_OK;
}

template <typename T>
int dmalloc(DevMem &m, T **p, size_t n, bool zero = true) {
  const size_t bytes = ((n ? n : 1) * sizeof(T) + 1023) / 1024 * 1024;
  if (bytes > m.left) {
    size_t want = m.next;
    if (bytes >= want) want = bytes;
    else if (m.next < ((size_t)256 << 20)) m.next *= 2;
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, want);
    if (e != cudaSuccess && want > bytes) { cudaGetLastError(); e = cudaMalloc(&q, want = bytes); }
    if (e != cudaSuccess) {
      cudaGetLastError();
      g_last_cuda_error = (int)e;
      return CORUN_ENOMEM;
    }
    m.blocks.push_back(q);
    if (want == bytes) {                            // a block of its own: the current one goes on
      if (zero && cudaMemset(q, 0, bytes) != cudaSuccess) return CORUN_ECUDA;
      *p = (T *)q;
      return CORUN_OK;
    }
    m.cur = (char *)q;
    m.left = want;
  }
  if (zero && cudaMemset(m.cur, 0, bytes) != cudaSuccess) return CORUN_ECUDA;
  *p = (T *)m.cur;
  m.cur += bytes;
  m.left -= bytes;
  return CORUN_OK;
}

int pad16(int x) { return (x + 15) / 16 * 16; }

void mla_group_table(std::vector<int> &t, int nh, int rows_per_head, int BG, int R, int w_rows, int count_at);
int program_create_groups(corun_engine *e, Program &P, int R, int lg_rows, char *room = nullptr);

// fuse_swiglu: the gate / up GEMM writes silu(gate) * up itself (dense feed-forward, up to 128 padded rows: the
// decode program while it is bound by the weight stream; whole tiles on fewer CTAs would cost a prefill chunk,
// which is bound by the tensor pipe, a third of its gate / up rate).
int program_create(corun_engine *e, Program &P, int R, bool layers, bool lm, bool grouped = false, bool fuse_swiglu = false) {
  const corun_shape &s = e->sh;
  const int H = s.hidden, QD = s.n_q_heads * s.head_dim, KD = s.n_kv_heads * s.head_dim, F = s.ffn, V = s.vocab;
  const MlaDims &md = e->md;
  // columns of the q / k / v (MLA: q / kv_a) projection
  const int QKVN = e->mla ? md.nh * (md.nope + md.rope) + md.rank + md.rope : QD + 2 * KD;
  const int Fd = e->dense_ffn;                      // MLA: width of the dense feed-forward layers beside expert layers
  const int Fmax = F > Fd ? F : Fd;
  P.R = R;
  P.BN = pad16(R);
  P.has_layers = layers;
  P.has_lm = lm;
  P.wide = layers && lm && e->wide;
  const int RB = P.wide ? 256 : P.BN, RR = P.wide ? 256 : R;   // rows of the projections' inputs and outputs
  auto &A = P.allocs;
  RC(dmalloc(A, &P.xn_hi, (size_t)RB * H));
  RC(dmalloc(A, &P.xn_lo, (size_t)RB * H));
  if (!P.wide || e->moe_E) RC(dmalloc(A, &P.ws, gemm_ws_floats(e->num_sms, P.BN)));
  RC(dmalloc(A, &P.row_token, R));
  RC(dmalloc(A, &P.row_pos, R));
  RC(dmalloc(A, &P.row_active, R));
  RC(dmalloc(A, &P.row_slot, R));
  RC(dmalloc(A, &P.do_sample, R));
  RC(dmalloc(A, &P.sampled, R));
  RC(dmalloc(A, &P.row_blocks, 1));
  RC(dmalloc(A, &P.slot_row, R));
  RC(dmalloc(A, &P.row_step, R));
  RC(dmalloc(A, &P.row_temp, R));
  RC(dmalloc(A, &P.row_top_p, R));
  if (layers) {
    RC(dmalloc(A, &P.h, (size_t)R * H));
    if (!e->mla) {
      RC(dmalloc(A, &P.q, (size_t)R * QD));
      RC(dmalloc(A, &P.part_acc, (size_t)R * s.n_q_heads * e->max_splits * s.head_dim));
      RC(dmalloc(A, &P.part_ml, (size_t)R * s.n_q_heads * e->max_splits * 2));
      RC(dmalloc(A, &P.att_work, (size_t)R * e->max_splits * e->sh.n_kv_heads));
      RC(dmalloc(A, &P.att_n_work, 2 + 2 * (size_t)R * e->sh.n_kv_heads));
      RC(dmalloc(A, &P.att_pool, (size_t)s.n_layers));
    } else {
      const int BG = mla_group_rows(P.BN), n_groups = md.nh * (mla_rows_per_head(P.BN) / BG);
      P.RPH = mla_rows_per_head(P.BN);
      const size_t hr = (size_t)md.nh * P.RPH;      // rows of the head-major matrices
      RC(dmalloc(A, &P.qn_hi, hr * md.nope));
      RC(dmalloc(A, &P.qn_lo, hr * md.nope));
      RC(dmalloc(A, &P.q_lat, hr * md.rank));
      RC(dmalloc(A, &P.q_rope, (size_t)R * md.nh * md.rope));
      RC(dmalloc(A, &P.ol_hi, hr * md.rank));
      RC(dmalloc(A, &P.ol_lo, hr * md.rank));
      RC(dmalloc(A, &P.uv_out, hr * (md.nope + md.vh)));
      RC(dmalloc(A, &P.mla_ml, (size_t)mla_part_ml_floats(R, md.nh, e->max_ctx) / 2));
      RC(dmalloc(A, &P.mla_po, (size_t)mla_part_o_floats(R, md.nh, md.rank, e->max_ctx)));
      RC(dmalloc(A, &P.tab_uk, (size_t)n_groups * 3 + 1));
      RC(dmalloc(A, &P.tab_uv, (size_t)n_groups * 3 + 1));
      std::vector<int> tk, tv;                      // all groups are in use
      mla_group_table(tk, md.nh, P.RPH, BG, R, md.rank, 3 * n_groups);
      mla_group_table(tv, md.nh, P.RPH, BG, R, md.nope + md.vh, 3 * n_groups);
      CK(cudaMemcpy(P.tab_uk, tk.data(), tk.size() * sizeof(int), cudaMemcpyHostToDevice));
      CK(cudaMemcpy(P.tab_uv, tv.data(), tv.size() * sizeof(int), cudaMemcpyHostToDevice));
      RC(gemm_plan_create_grouped(&P.p_uk, e->w_ukT, (long long)md.nh * md.rank, md.nope, md.rank, md.nope, P.qn_hi, P.qn_lo, n_groups,
                                  BG, P.q_lat, P.tab_uk, e->num_sms));
      RC(gemm_plan_create_grouped(&P.p_uv, e->w0_uv, (long long)md.nh * (md.nope + md.vh), md.rank, md.nope + md.vh, md.rank, P.ol_hi,
                                  P.ol_lo, n_groups, BG, P.uv_out, P.tab_uv, e->num_sms));
      P.p_uk.keep_div = P.p_uv.keep_div = -1;       // the tables are written once, here: the kernels need not wait for them
    }
    RC(dmalloc(A, &P.qkv_out, (size_t)RR * QKVN));
    RC(dmalloc(A, &P.o_out, (size_t)RR * H));
    // expert layers up to 64 rows: all rows with every expert that one of them selected
    const int NBx = e->moe_E + e->moe_S, half_x = e->moe_E ? gemm_swiglu_blocks_half(e->moe_F, NBx, e->num_sms) : 0;
    P.select = fuse_swiglu && e->moe_E && P.BN <= 64 && half_x && H % GEMM_TILE_N == 0 && NBx <= GEMM_MAX_SELECT &&
               !getenv("CORUN_MOE_DECODE_DENSE");
    const bool groups = grouped && e->moe_E && !P.select && (2 * e->moe_F) % GEMM_TILE_N == 0 && H % GEMM_TILE_N == 0;
    const int Fbuf = P.select || groups ? (Fd > 64 ? Fd : 64) : Fmax;   // those forms have buffers of their own
    RC(dmalloc(A, &P.gu_out, (size_t)R * 2 * Fbuf));
    RC(dmalloc(A, &P.down_out, (size_t)RR * H));
    RC(dmalloc(A, &P.ao_hi, (size_t)RB * QD));
    RC(dmalloc(A, &P.ao_lo, (size_t)RB * QD));
    RC(dmalloc(A, &P.ff_hi, (size_t)RB * Fbuf));
    RC(dmalloc(A, &P.ff_lo, (size_t)RB * Fbuf));
    if (e->mla && e->moe_E && e->first_dense > 0) {   // the dense feed-forward layers of a decoder with expert layers
      RC(gemm_plan_create(&P.p_gu_d, e->w0_gu_d, 2 * Fd, H, P.xn_hi, P.xn_lo, R, P.BN, P.gu_out, P.ws, e->num_sms));
      RC(gemm_plan_create(&P.p_down_d, e->w0_down_d, H, Fd, P.ff_hi, P.ff_lo, R, P.BN, P.down_out, P.ws, e->num_sms));
    }
    // the plans carry layer 0's weights; the per-layer tensor maps override them at launch
    if (P.wide) {
      const bool ffn = !e->moe_E;
      size_t part = gemm_pair_part_floats(QKVN, H, 256, e->num_sms, true);
      for (size_t x : {gemm_pair_part_floats(H, QD, 256, e->num_sms, true), ffn ? gemm_pair_part_floats(H, F, 256, e->num_sms, true) : 0,
                       gemm_pair_part_floats(V, H, 256, e->num_sms, true)})
        part = x > part ? x : part;
      RC(dmalloc(A, &P.pair_part, part, false));
      P.pair_part_floats = part;
      if (!P.plain_tiles) RC(dmalloc(A, &P.plain_tiles, (size_t)((QKVN > V ? QKVN : V) / GEMM_TILE_N + 1)));
      RC(gemm_pair_plan_create(&P.b_qkv, QKVN, H, P.xn_hi, P.xn_lo, 256, P.qkv_out, P.pair_part, e->num_sms, true));
      RC(gemm_pair_plan_create(&P.b_o, H, QD, P.ao_hi, P.ao_lo, 256, P.o_out, P.pair_part, e->num_sms, true));
      if (ffn) {
        RC(gemm_pair_plan_create_swiglu(&P.b_gu, F, H, P.xn_hi, P.xn_lo, 256, P.ff_hi, P.ff_lo, e->num_sms, true));
        RC(gemm_pair_plan_create(&P.b_down, H, F, P.ff_hi, P.ff_lo, 256, P.down_out, P.pair_part, e->num_sms, true));
      }
    } else {
      RC(gemm_plan_create(&P.p_qkv, e->w0_qkv, QKVN, H, P.xn_hi, P.xn_lo, R, P.BN, P.qkv_out, P.ws, e->num_sms));
      RC(gemm_plan_create(&P.p_o, e->w0_o, H, QD, P.ao_hi, P.ao_lo, R, P.BN, P.o_out, P.ws, e->num_sms));
    }
    // expert layers without groups: the routing weight and the SwiGLU in the epilogue of the GEMM over all experts'
    // gate / up rows (65..128 rows, where the grouped form below does not apply; up to 64 rows the masked store plus a
    // SwiGLU kernel measured faster: the epilogue would write zeros for every pair that was not selected)
    const bool moe_fused = fuse_swiglu && e->moe_E && P.BN > 64 && P.BN <= 128 &&
                           gemm_swiglu_blocks_half(e->moe_F, e->moe_E + e->moe_S, e->num_sms) > 0;
    if (P.select) {
      const int nb = e->moe_E + e->moe_S, per_row = e->moe_K + e->moe_S, Fm = e->moe_F;
      RC(dmalloc(A, &P.moe_w, (size_t)R * nb));
      RC(dmalloc(A, &P.router_rs.logit, (size_t)R * e->moe_E));
      RC(dmalloc(A, &P.router_rs.count, (size_t)R));
      RC(dmalloc(A, &P.moe_sel, (size_t)R * per_row));
      RC(dmalloc(A, &P.hg_hi, (size_t)nb * P.BN * Fm));
      RC(dmalloc(A, &P.hg_lo, (size_t)nb * P.BN * Fm));
      RC(dmalloc(A, &P.yg_out, (size_t)nb * P.BN * H));
      RC(dmalloc(A, &P.plain_tiles, (size_t)(H / GEMM_TILE_N + 1)));
      RC(gemm_plan_create_select_up(&P.p_gug, e->w0_gu, nb, Fm, H, half_x, P.xn_hi, P.xn_lo, R, P.BN, P.hg_hi, P.hg_lo, P.moe_w, P.moe_sel,
                                    R * per_row, e->num_sms));
      RC(gemm_plan_create_select_down(&P.p_dng, e->w0_down, nb, H, Fm, P.hg_hi, P.hg_lo, R, P.BN, P.yg_out, P.moe_w, P.moe_sel,
                                      R * per_row, e->num_sms));
    } else if (groups || (P.wide && !e->moe_E)) {
      // their GEMMs are made below / above
    } else if (fuse_swiglu && !e->moe_E && P.BN <= 128)
      RC(gemm_plan_create_swiglu(&P.p_gu, e->w0_gu, F, H, P.xn_hi, P.xn_lo, R, P.BN, P.ff_hi, P.ff_lo, e->num_sms));
    else if (!moe_fused)
      RC(gemm_plan_create(&P.p_gu, e->w0_gu, 2 * F, H, P.xn_hi, P.xn_lo, R, P.BN, P.gu_out, P.ws, e->num_sms));
    if (!P.select && !groups && !(P.wide && !e->moe_E)) RC(gemm_plan_create(&P.p_down, e->w0_down, H, F, P.ff_hi, P.ff_lo, R, P.BN, P.down_out, P.ws, e->num_sms));
    if (e->moe_E && !P.select) {
      const int NB = e->moe_E + e->moe_S;
      RC(dmalloc(A, &P.moe_w, (size_t)R * NB));
      RC(dmalloc(A, &P.router_rs.logit, (size_t)R * e->moe_E));
      RC(dmalloc(A, &P.router_rs.count, (size_t)R));
      if (groups) {
      } else if (moe_fused)
        RC(gemm_plan_create_swiglu_blocks(&P.p_gu, e->w0_gu, NB, e->moe_F, H, P.xn_hi, P.xn_lo, R, P.BN, P.ff_hi, P.ff_lo, P.moe_w,
                                          e->num_sms));
      else if ((2 * e->moe_F) % GEMM_TILE_N == 0) {   // a weight tile belongs to one expert: rows that did not
        P.p_gu.row_keep = P.moe_w;                  // select it are not stored (the SwiGLU does not read them)
        P.p_gu.keep_pitch = NB;
        P.p_gu.keep_div = 2 * e->moe_F / GEMM_TILE_N;
      }
      if (groups) {
        // prefill chunks: every row through every expert would be (E + S) / top_k times the MMA work, which a
        // chunk of 256 rows does pay for; the rows of an expert are gathered into blocks of 64 instead
        if (!P.plain_tiles) RC(dmalloc(A, &P.plain_tiles, (size_t)(H / GEMM_TILE_N + 1)));
        RC(program_create_groups(e, P, R, 6));
      }
    }
  }
  if (lm) {
    RC(dmalloc(A, &P.logits, (size_t)RR * V));
    if (P.wide) return gemm_pair_plan_create(&P.b_lm, V, H, P.xn_hi, P.xn_lo, 256, P.logits, P.pair_part, e->num_sms, true);
    RC(gemm_plan_create(&P.p_lm, e->lm_head, V, H, P.xn_hi, P.xn_lo, R, P.BN, P.logits, P.ws, e->num_sms));
  }
  return CORUN_OK;
}

// Group table of the up-projections of a latent attention layer with rows_per_head rows per head, R of them in use:
// group = (head, block of BG rows): its first weight row, its first weight k-block, its rows; at count_at the number of
// groups.
void mla_group_table(std::vector<int> &t, int nh, int rows_per_head, int BG, int R, int w_rows, int count_at) {
  t.assign((size_t)count_at + 1, 0);
  const int per_head = rows_per_head / BG, n = nh * per_head;
  for (int g = 0; g < n; ++g) {
    const int h = g / per_head, rb = g % per_head, left = R - rb * BG;
    t[3 * g] = h * w_rows;
    t[3 * g + 2] = left < 0 ? 0 : left < BG ? left : BG;
  }
  t[count_at] = n;
}

// Slots of the experts' grouped form for up to R rows, and what their gathered rows, hidden activations and results take at `room`
// (the results over the gathered rows, which only the gate / up product reads).
size_t group_slots(const corun_engine *e, int R, int lg_rows) { return (size_t)moe_max_groups(R, e->moe_E, e->moe_S, e->moe_K, lg_rows) << lg_rows; }
size_t group_room(const corun_engine *e, int R, int lg_rows) { return group_slots(e, R, lg_rows) * 4 * (size_t)(e->sh.hidden + e->moe_F); }

// Buffers and plans of the experts' grouped form for up to R rows.
int program_create_groups(corun_engine *e, Program &P, int R, int lg_rows, char *room) {
  const int Fm = e->moe_F, NB = e->moe_E + e->moe_S, H = e->sh.hidden;
  auto &A = P.allocs;
  MoeGroups &g = P.grp;
  g.lg_rows = lg_rows;
  g.n_groups_max = moe_max_groups(R, e->moe_E, e->moe_S, e->moe_K, lg_rows);
  const size_t slots = group_slots(e, R, lg_rows);
  RC(dmalloc(A, &g.tab_up, (size_t)g.n_groups_max * 3 + 1));
  RC(dmalloc(A, &g.tab_down, (size_t)g.n_groups_max * 3 + 1));
  RC(dmalloc(A, &g.group_expert, (size_t)g.n_groups_max));
  RC(dmalloc(A, &g.slot_row, slots));
  RC(dmalloc(A, &g.slot_of, (size_t)R * NB));
  RC(dmalloc(A, &g.slot_w, slots));
  P.grouped = true;
  if (room) {
    P.xg_hi = (bf16 *)room;
    P.xg_lo = P.xg_hi + slots * H;
    P.yg_out = (float *)room;
    P.hg_hi = P.xg_lo + slots * H;
    P.hg_lo = P.hg_hi + slots * Fm;
  } else {
    RC(dmalloc(A, &P.xg_hi, slots * H));
    RC(dmalloc(A, &P.xg_lo, slots * H));
    RC(dmalloc(A, &P.hg_hi, slots * Fm));
    RC(dmalloc(A, &P.hg_lo, slots * Fm));
    RC(dmalloc(A, &P.yg_out, slots * H));
  }
  if (P.pair) {                                     // prompts: on pairs of SMs
    RC(gemm_experts_plan_create_swiglu(&P.x_gu, Fm, H, P.xg_hi, P.xg_lo, g.n_groups_max, P.hg_hi, P.hg_lo, g.slot_w, g.tab_up, e->num_sms));
    return gemm_experts_plan_create(&P.x_down, H, Fm, P.hg_hi, P.hg_lo, g.n_groups_max, P.yg_out, g.tab_down, e->num_sms);
  }
  // gate / up per group with the routing weight and the SwiGLU in the epilogue where a tile width divides the
  // experts' width, else fp32 sums and a kernel of its own
  const int half = gemm_swiglu_blocks_half(Fm, NB, e->num_sms);
  if (half) {
    RC(gemm_plan_create_grouped_swiglu(&P.p_gug, e->w0_gu, (long long)NB * 2 * Fm, Fm, H, half, P.xg_hi, P.xg_lo, g.n_groups_max,
                                       g.rows(), P.hg_hi, P.hg_lo, g.slot_w, g.tab_up, e->num_sms));
  } else {
    RC(dmalloc(A, &P.gug_out, slots * 2 * Fm));
    RC(gemm_plan_create_grouped(&P.p_gug, e->w0_gu, (long long)NB * 2 * Fm, H, 2 * Fm, H, P.xg_hi, P.xg_lo, g.n_groups_max,
                                g.rows(), P.gug_out, g.tab_up, e->num_sms));
  }
  RC(gemm_plan_create_grouped(&P.p_dng, e->w0_down, H, NB * Fm, H, Fm, P.hg_hi, P.hg_lo, g.n_groups_max, g.rows(),
                              P.yg_out, g.tab_down, e->num_sms));
  return CORUN_OK;
}

// The program of long prompts: buffers for `cap` rows.
int program_create_big(corun_engine *e, Program &P, int cap) {
  const corun_shape &s = e->sh;
  const MlaDims &md = e->md;
  const int H = s.hidden, QD = s.n_q_heads * s.head_dim, KD = s.n_kv_heads * s.head_dim;
  const int QKVN = e->mla ? md.nh * (md.nope + md.rope) + md.rank + md.rope : QD + 2 * KD;
  const int F = e->moe_E ? e->dense_ffn : s.ffn;    // width of the dense feed-forward layers, 0: there are none
  P.pair = true;
  P.R = P.cap = P.BN = cap;
  P.has_layers = true;
  auto &A = P.allocs;
  const size_t c = (size_t)cap;
  // One piece of memory for what the attention half of a layer hands on (the projections, queries, latent queries and values) and what
  // the feed-forward half does.  Each is written, for all rows of the chunk, before it is read, so nothing needs clearing.
  const size_t hr = e->mla ? (size_t)md.nh * cap : 0;   // rows of the head-major matrices (cap is a multiple of 64)
  const size_t attn_room = (c * (QKVN + (e->mla ? 0 : QD)) + hr * (md.rank + md.nope + md.vh)) * sizeof(float);
  const size_t room_bytes = std::max(attn_room, std::max(c * F * 4, e->moe_E ? group_room(e, cap, 7) : (size_t)0));
  // partial tiles of an unfilled wave: consumed by the next kernel of the stream, so one buffer serves all
  size_t part = gemm_pair_part_floats(QKVN, H, cap, e->num_sms);
  for (size_t x : {gemm_pair_part_floats(H, QD, cap, e->num_sms), F > 0 ? gemm_pair_part_floats(H, F, cap, e->num_sms) : 0,
                   e->moe_E ? gemm_pair_part_floats(e->moe_E, H, cap, e->num_sms) : 0})
    part = x > part ? x : part;
  // at most one request of a chunk began in an earlier one: the others' tokens are rows of the chunk
  if (e->big_mla_tiles) P.kv_cap = (e->max_ctx + cap + 64 * MLA_MAX_SEGS + 255) / 256 * 256;
  // All of it in one block.  Engines with chunks of 2048 rows / of 4096, every buffer apart and cleared, in blocks of powers of two / so:
  // 12 Qwen3-8B layers, 8 slots 2686 / 3038 / 2546 MiB, 12 Qwen3-30B-A3B layers, 64 slots 3882 / 4778 / 3704, 9 DeepSeek-V2-Lite layers, 128
  // slots 6174 / 7264 / 5746; created in 19 / 20.5 / 18, 15 / 21 / 14.5 and 15.5 / 17.5 / 13.5 ms.
  const int NB = e->moe_E + e->moe_S;
  size_t all = c * 4 * (3 * (size_t)H + QD + 4) + room_bytes + (gemm_ws_floats(e->num_sms, SHORT_ROWS) + part) * sizeof(float) + (1 << 20);
  if (e->mla)
    all += hr * 4 * (size_t)(md.nope + md.rank + md.rope) + (size_t)P.kv_cap * (4 * md.rank + 128 + 1024 * (size_t)md.nh) +
           ((size_t)mla_part_ml_floats(MLA_ROWS, md.nh, e->max_ctx) + mla_part_o_floats(MLA_ROWS, md.nh, md.rank, e->max_ctx)) * sizeof(float);
  if (e->moe_E) all += c * 4 * (size_t)(2 * NB + e->moe_E) + group_slots(e, cap, 7) * 8 + (size_t)NB * (MOE_MANY_ROWS / 8);
  A.reserve(all);
  RC(dmalloc(A, &P.xn_hi, c * H));
  RC(dmalloc(A, &P.xn_lo, c * H));
  RC(dmalloc(A, &P.row_token, 4 * c));              // token | position | active | slot, as many rows as the chunk at hand has
  RC(dmalloc(A, &P.row_blocks, c / SHORT_ROWS));
  RC(dmalloc(A, &P.h, c * H));
  RC(dmalloc(A, &P.down_out, c * H));
  P.o_out = P.down_out;                             // (the residual takes one up before the other is written)
  char *room = nullptr;
  RC(dmalloc(A, &room, room_bytes, false));
  P.qkv_out = (float *)room;
  RC(dmalloc(A, &P.ao_hi, c * QD));
  RC(dmalloc(A, &P.ao_lo, c * QD));
  RC(dmalloc(A, &P.plain_tiles, (size_t)((QKVN > H ? QKVN : H) / GEMM_TILE_N + 1)));
  const int n_blk = cap / SHORT_ROWS;               // cap is a multiple of 256
  RC(dmalloc(A, &P.ws, gemm_ws_floats(e->num_sms, SHORT_ROWS)));
  for (auto *v : {&P.s_qkv, &P.s_o, &P.s_gu, &P.s_down}) v->resize((size_t)n_blk);
  RC(gemm_plan_create(&P.s_qkv[0], e->w0_qkv, QKVN, H, P.xn_hi, P.xn_lo, SHORT_ROWS, SHORT_ROWS, P.qkv_out, P.ws, e->num_sms));
  RC(gemm_plan_create(&P.s_o[0], e->w0_o, H, QD, P.ao_hi, P.ao_lo, SHORT_ROWS, SHORT_ROWS, P.o_out, P.ws, e->num_sms));
  RC(dmalloc(A, &P.pair_part, part, false));
  RC(gemm_pair_plan_create(&P.b_qkv, QKVN, H, P.xn_hi, P.xn_lo, cap, P.qkv_out, P.pair_part, e->num_sms));
  RC(gemm_pair_plan_create(&P.b_o, H, QD, P.ao_hi, P.ao_lo, cap, P.o_out, P.pair_part, e->num_sms));
  if (F > 0) {
    P.ff_hi = (bf16 *)room;
    P.ff_lo = P.ff_hi + c * F;
    RC(gemm_plan_create_swiglu(&P.s_gu[0], e->moe_E ? e->w0_gu_d : e->w0_gu, F, H, P.xn_hi, P.xn_lo, SHORT_ROWS, SHORT_ROWS, P.ff_hi, P.ff_lo,
                               e->num_sms));
    RC(gemm_plan_create(&P.s_down[0], e->moe_E ? e->w0_down_d : e->w0_down, H, F, P.ff_hi, P.ff_lo, SHORT_ROWS, SHORT_ROWS, P.down_out, P.ws,
                        e->num_sms));
    RC(gemm_pair_plan_create_swiglu(&P.b_gu, F, H, P.xn_hi, P.xn_lo, cap, P.ff_hi, P.ff_lo, e->num_sms));
    RC(gemm_pair_plan_create(&P.b_down, H, F, P.ff_hi, P.ff_lo, cap, P.down_out, P.pair_part, e->num_sms));
  }
  for (int b = n_blk - 1; b >= 0; --b) {            // (block 0 last: the others are copies of it)
    const size_t r0 = (size_t)b * SHORT_ROWS;
    const int *rb = P.row_blocks + b;
    RC(gemm_plan_rebase(&P.s_qkv[b], P.s_qkv[0], P.xn_hi + r0 * H, P.xn_lo + r0 * H, P.qkv_out + r0 * QKVN, nullptr, nullptr, rb));
    RC(gemm_plan_rebase(&P.s_o[b], P.s_o[0], P.ao_hi + r0 * QD, P.ao_lo + r0 * QD, P.o_out + r0 * H, nullptr, nullptr, rb));
    if (F > 0) {
      RC(gemm_plan_rebase(&P.s_gu[b], P.s_gu[0], P.xn_hi + r0 * H, P.xn_lo + r0 * H, nullptr, P.ff_hi + r0 * F, P.ff_lo + r0 * F, rb));
      RC(gemm_plan_rebase(&P.s_down[b], P.s_down[0], P.ff_hi + r0 * F, P.ff_lo + r0 * F, P.down_out + r0 * H, nullptr, nullptr, rb));
    }
  }
  if (!e->mla) {
    P.q = P.qkv_out + c * QKVN;
  } else {
    const int n_groups = md.nh * (cap / 64);
    RC(dmalloc(A, &P.qn_hi, hr * md.nope));
    RC(dmalloc(A, &P.qn_lo, hr * md.nope));
    P.q_lat = P.qkv_out + c * QKVN;
    P.uv_out = P.q_lat + hr * md.rank;
    RC(dmalloc(A, &P.q_rope, c * md.nh * md.rope));
    RC(dmalloc(A, &P.ol_hi, hr * md.rank));
    RC(dmalloc(A, &P.ol_lo, hr * md.rank));
    RC(dmalloc(A, &P.mla_ml, (size_t)mla_part_ml_floats(MLA_ROWS, md.nh, e->max_ctx) / 2));
    RC(dmalloc(A, &P.mla_po, (size_t)mla_part_o_floats(MLA_ROWS, md.nh, md.rank, e->max_ctx)));
    RC(dmalloc(A, &P.tab_uk, (size_t)n_groups * 3 + 1));
    RC(dmalloc(A, &P.tab_uv, (size_t)n_groups * 3 + 1));
    RC(gemm_plan_create_grouped(&P.p_uk, e->w_ukT, (long long)md.nh * md.rank, md.nope, md.rank, md.nope, P.qn_hi, P.qn_lo, n_groups,
                                64, P.q_lat, P.tab_uk, e->num_sms));
    RC(gemm_plan_create_grouped(&P.p_uv, e->w0_uv, (long long)md.nh * (md.nope + md.vh), md.rank, md.nope + md.vh, md.rank, P.ol_hi,
                                P.ol_lo, n_groups, 64, P.uv_out, P.tab_uv, e->num_sms));
    if (e->big_mla_tiles) {
      P.mla_tiles = true;
      const size_t kc = (size_t)P.kv_cap;
      RC(dmalloc(A, &P.c_hi, kc * md.rank));
      RC(dmalloc(A, &P.c_lo, kc * md.rank));
      RC(dmalloc(A, &P.kr, kc * 64));               // zeros beyond rope, and finite everywhere: masked keys have weight zero
      RC(dmalloc(A, &P.kvd, 4 * kc * md.nh * 128));
      RC(dmalloc(A, &P.tile_base, (size_t)cap / 128));
      RC(gemm_pair_plan_create_kv(&P.b_kv, md.nh, md.rank, P.c_hi, P.c_lo, P.kv_cap, P.kvd, e->num_sms));
      RC(tma_encode_2d(&P.tm_kvd, P.kvd, 1, 4 * kc * md.nh, 128, 64, 64));
      RC(tma_encode_2d(&P.tm_kr, P.kr, 1, kc, 64, 64, 64));
      if (mla_prefill_prepare() != cudaSuccess) return CORUN_ECUDA;
    }
    P.p_uk.keep_div = P.p_uv.keep_div = -1;         // the tables are copied ahead of a chunk's kernels (set_mla_rows)
  }
  if (e->moe_E) {
    RC(dmalloc(A, &P.moe_w, c * NB));
    RC(dmalloc(A, &P.router_out, c * e->moe_E));
    RC(dmalloc(A, &P.moe_mask, (size_t)NB * (MOE_MANY_ROWS / 32)));
    RC(gemm_pair_plan_create(&P.b_router, e->moe_E, H, P.xn_hi, P.xn_lo, cap, P.router_out, P.pair_part, e->num_sms));
    RC(program_create_groups(e, P, cap, 7, room));  // (groups of 128 rows: an expert with fewer pays for those it has)
  }
  return CORUN_OK;
}

// (prefill) lays the head-major matrices out for a chunk of R rows: whole blocks of 64 per head, one behind the other.
// stage: pinned memory for the two group tables, not touched again before the stream has drained.
int set_mla_rows(corun_engine *e, Program &P, int R, int *stage) {
  const MlaDims &md = e->md;
  const int rph = (R + 63) / 64 * 64, count_at = md.nh * (P.cap / 64) * 3;
  P.RPH = rph;
  std::vector<int> t;
  for (int k = 0; k < 2; ++k) {
    mla_group_table(t, md.nh, rph, 64, R, k == 0 ? md.rank : md.nope + md.vh, count_at);
    memcpy(stage + k * t.size(), t.data(), t.size() * sizeof(int));
    CK(cudaMemcpyAsync(k == 0 ? P.tab_uk : P.tab_uv, stage + k * t.size(), t.size() * sizeof(int), cudaMemcpyHostToDevice, e->st));
  }
  return CORUN_OK;
}

void program_destroy(Program &P) {
  gemm_plan_destroy(&P.p_qkv);
  gemm_plan_destroy(&P.p_o);
  gemm_plan_destroy(&P.p_gu);
  gemm_plan_destroy(&P.p_down);
  gemm_plan_destroy(&P.p_lm);
  gemm_plan_destroy(&P.p_gug);
  gemm_plan_destroy(&P.p_dng);
  gemm_plan_destroy(&P.p_uk);
  gemm_plan_destroy(&P.p_uv);
  gemm_plan_destroy(&P.p_gu_d);
  gemm_plan_destroy(&P.p_down_d);
  for (auto *v : {&P.s_qkv, &P.s_o, &P.s_gu, &P.s_down})
    if (!v->empty()) gemm_plan_destroy(&(*v)[0]);   // the others share its tables
  P.allocs.release();
}

KvLayout kv_layout(const corun_engine *e) {
  return KvLayout{e->kv_pool, e->d_block_table, e->max_blocks, e->sh.n_kv_heads, e->sh.head_dim, e->layer_stride,
                  (long long)e->pool_blocks, e->B};
}

// The result of a layer's feed-forward part as the next kernel reads it: the down GEMM's partials, or (grouped
// Mixture-of-Experts form) the combined plain matrix.
GemmOut plain_out(const Program &P, const float *m, int N) {
  return GemmOut{m, nullptr, P.plain_tiles, P.plain_tiles, N, 0, P.BN, 0, 0, 0};
}

bool dense_layer(const corun_engine *e, int layer) { return e->mla && e->moe_E && layer < e->first_dense; }

GemmOut ffn_out(const corun_engine *e, const Program &P, int layer) {
  if (P.pair) return P.grouped && !dense_layer(e, layer) ? plain_out(P, P.down_out, e->sh.hidden) : gemm_pair_out(P.b_down, P.R, P.plain_tiles);
  if (dense_layer(e, layer)) return P.p_down_d.out();
  if (P.wide && !e->moe_E) return gemm_pair_out(P.b_down, P.R, P.plain_tiles);
  if (P.grouped || P.select) return plain_out(P, P.down_out, e->sh.hidden);
  return P.p_down.out();
}

// Latent attention of a chunk of long prompts: the segments' keys and values, then their tiles of 128 query tokens.
cudaError_t run_mla_tiles(corun_engine *e, Program &P, int l, const Rows &rows) {
  const MlaDims &md = e->md;
  const MlaCache cache{e->kv_pool + (size_t)l * e->layer_stride, e->d_block_table, e->max_blocks, e->B, (long long)e->pool_blocks, e->kv_run};
  cudaError_t ce = launch_mla_gather(P.segs, cache, md.rank, md.rope, P.kv_tokens, P.c_hi, P.c_lo, P.kr, e->st);
  const float2 *scale = e->kv_scale + (size_t)l * md.nh;
  if (ce == cudaSuccess) ce = gemm_pair_launch(P.b_kv, e->tb_uv[l], P.kv_tokens, e->d_status, e->st, nullptr, reinterpret_cast<const float *>(scale));
  if (ce == cudaSuccess)
    ce = launch_mla_prefill(P.tm_kvd, P.tm_kr, P.qn_hi, P.qn_lo, P.q_rope, rows, P.RPH, md, P.kv_cap, P.tile_base,
                            1.0f / sqrtf((float)(md.nope + md.rope)), scale, P.ao_hi, P.ao_lo, e->d_status, e->st);
  return ce;
}

// Enqueues embed -> all layers (ends with the last down GEMM; prefill: with the final norm of every row).  Counts launches.
int run_layers(corun_engine *e, Program &P, int *launches) {
  const corun_shape &s = e->sh;
  const Rows rows{P.row_token, P.row_pos, P.row_active, P.row_slot, P.R};
  const KvLayout kv = kv_layout(e);
  int n = 0;
  if (&P == &e->dec && !e->mla) {                   // the prefill attention kernel needs no item list
    CK(launch_attn_worklist(rows, e->sh.n_kv_heads, P.att_work, P.att_n_work, P.att_pool, s.n_layers, e->whole_pairs, e->st));   // the same items serve every layer
    n += 1;
  }
  // (debug) slice of the step trace for the idx-th GEMM of the decode program: [num_sms][8] stamps
  auto tr = [&](int idx) -> unsigned long long * {
    return (e->step_trace && &P == &e->dec) ? e->step_trace + (size_t)idx * e->num_sms * 8 : nullptr;
  };
  int stage = 0;
  const int stop = (e->eager && &P == &e->dec) ? e->stop_after : -1;
#define STAGE(call)                                   \
  do {                                                \
    if (stop >= 0 && stage >= stop) return CORUN_OK;  \
    CK(call);                                         \
    ++stage;                                          \
  } while (0)
  const bool many = P.pair && !P.shorts;
  bool normed = false;                              // the layer's input has been normalised behind the layer before
  const int QD = s.n_q_heads * s.head_dim;
  // (short prompts) the blocks of the chunk: first row, and the rows of it as token-wise kernels take them
  const int n_blk = P.shorts ? (P.R + SHORT_ROWS - 1) / SHORT_ROWS : 0;
  auto block_rows = [&](int b) {
    const int r0 = b * SHORT_ROWS, left = P.R - r0;
    return Rows{P.row_token + r0, P.row_pos + r0, P.row_active + r0, P.row_slot + r0, left < SHORT_ROWS ? left : SHORT_ROWS};
  };
  for (int l = 0; l < s.n_layers; ++l) {
    GemmOut prev = ffn_out(e, P, l > 0 ? l - 1 : 0);
    if (!normed)
      STAGE(launch_resid_norm(P.h, s.hidden, e->embed, rows, l == 0 ? nullptr : &prev, e->attn_norm[l], s.rms_eps,
                              P.xn_hi, P.xn_lo, e->st, many));
    normed = false;
    if (P.pair) {
      // prefill; long prompts: projections on pairs of SMs, plain results
      if (!P.shorts) STAGE(gemm_pair_launch(P.b_qkv, e->tb_qkv[l], P.R, e->d_status, e->st));
      if (e->mla) {
        const MlaDims &md = e->md;
        const MlaCache cache{e->kv_pool + (size_t)l * e->layer_stride, e->d_block_table, e->max_blocks, e->B, (long long)e->pool_blocks, e->kv_run};
        if (!P.shorts)
          STAGE(launch_mla_post(gemm_pair_out(P.b_qkv, P.R, P.plain_tiles), rows, e->d_rope, md, e->kv_norm[l], s.rms_eps, cache, P.RPH, P.qn_hi,
                                P.qn_lo, P.q_rope, e->d_status, e->st));
        for (int b = 0; b < n_blk; ++b) {
          const size_t r0 = (size_t)b * SHORT_ROWS;
          STAGE(gemm_launch(P.s_qkv[b], &e->tm_qkv[l], e->d_status, e->st, nullptr, true));
          STAGE(launch_mla_post(P.s_qkv[b].out(), block_rows(b), e->d_rope, md, e->kv_norm[l], s.rms_eps, cache, P.RPH, P.qn_hi + r0 * md.nope,
                                P.qn_lo + r0 * md.nope, P.q_rope + r0 * md.nh * md.rope, e->d_status, e->st));
        }
        if (P.mla_tiles && !P.shorts) {
          STAGE(run_mla_tiles(e, P, l, rows));
        } else {
          STAGE(gemm_launch(P.p_uk, &e->tm_uk[l], e->d_status, e->st, nullptr, true));
          for (int r0 = 0; r0 < P.R; r0 += MLA_ROWS) {
            const int nr = P.R - r0 < MLA_ROWS ? P.R - r0 : MLA_ROWS;
            const Rows part{P.row_token + r0, P.row_pos + r0, P.row_active + r0, P.row_slot + r0, nr};
            STAGE(launch_mla_attention(e->tm_c[l], e->tm_cv[l], P.q_lat + (size_t)r0 * md.rank, md.rank, (long long)P.RPH * md.rank,
                                       P.q_rope + (size_t)r0 * md.nh * md.rope, e->d_block_table, e->max_blocks, nullptr, &part, nr, md,
                                       1.0f / sqrtf((float)(md.nope + md.rope)), e->mla_splits, P.mla_ml, P.mla_po, nullptr,
                                       P.ol_hi + (size_t)r0 * md.rank, P.ol_lo + (size_t)r0 * md.rank, P.RPH, e->num_sms, e->d_status, true,
                                       e->st, e->kv_run));
          }
          STAGE(gemm_launch(P.p_uv, &e->tm_uv[l], e->d_status, e->st, nullptr, true));
          STAGE(launch_mla_ao_split(P.uv_out, P.R, P.RPH, md, P.ao_hi, P.ao_lo, e->st));
        }
      } else {
        if (!P.shorts) STAGE(launch_qkv_post(gemm_pair_out(P.b_qkv, P.R, P.plain_tiles), rows, e->d_rope, s.n_q_heads, kv, l, P.q, e->d_status, e->st));
        for (int b = 0; b < n_blk; ++b) {
          STAGE(gemm_launch(P.s_qkv[b], &e->tm_qkv[l], e->d_status, e->st, nullptr, true));
          STAGE(launch_qkv_post(P.s_qkv[b].out(), block_rows(b), e->d_rope, s.n_q_heads, kv, l, P.q + (size_t)b * SHORT_ROWS * QD, e->d_status,
                                e->st));
        }
        STAGE(launch_attention_prefill(e->tm_k4[l], P.q, rows, s.n_q_heads, kv, P.ao_hi, P.ao_lo, e->d_status, e->st));
      }
      if (!P.shorts) {
        STAGE(gemm_pair_launch(P.b_o, e->tb_o[l], P.R, e->d_status, e->st));
        const GemmOut o = gemm_pair_out(P.b_o, P.R, P.plain_tiles);
        STAGE(launch_resid_norm(P.h, s.hidden, nullptr, rows, &o, e->mlp_norm[l], s.rms_eps, P.xn_hi, P.xn_lo, e->st, many));
      }
      const bool experts = e->moe_E && !dense_layer(e, l);
      const bf16 *next_norm = l + 1 < s.n_layers ? e->attn_norm[l + 1] : e->final_norm;
      for (int b = 0; b < n_blk; ++b) {             // (short prompts) the rest of a dense layer, block by block
        const size_t o0 = (size_t)b * SHORT_ROWS * s.hidden;
        const Rows br = block_rows(b);
        STAGE(gemm_launch(P.s_o[b], &e->tm_o[l], e->d_status, e->st, nullptr, true));
        const GemmOut o = P.s_o[b].out();
        STAGE(launch_resid_norm(P.h + o0, s.hidden, nullptr, br, &o, e->mlp_norm[l], s.rms_eps, P.xn_hi + o0, P.xn_lo + o0, e->st));
        if (experts) continue;
        STAGE(gemm_launch(P.s_gu[b], e->moe_E ? &e->tb_gu_half[l] : &e->tm_gu_half[l], e->d_status, e->st, nullptr, true));
        STAGE(gemm_launch(P.s_down[b], e->moe_E ? &e->tm_down_d[l] : &e->tm_down[l], e->d_status, e->st, nullptr, true));
        const GemmOut d = P.s_down[b].out();
        STAGE(launch_resid_norm(P.h + o0, s.hidden, nullptr, br, &d, next_norm, s.rms_eps, P.xn_hi + o0, P.xn_lo + o0, e->st));
      }
      normed = P.shorts && !experts;
      if (experts) {
        const int NB = e->moe_E + e->moe_S;
        STAGE(gemm_pair_launch(P.b_router, e->tb_router[l], P.R, e->d_status, e->st));
        STAGE(launch_moe_route(gemm_pair_out(P.b_router, P.R, P.plain_tiles), P.R, e->moe_E, e->moe_S, e->moe_K, e->moe_renorm, P.moe_w, e->st));
        STAGE(launch_moe_group_many(P.moe_w, P.row_active, P.R, e->moe_E, e->moe_S, e->moe_F, P.moe_mask, P.grp, e->st));
        STAGE(launch_moe_gather(P.xn_hi, P.xn_lo, s.hidden, P.grp, P.xg_hi, P.xg_lo, e->st));
        STAGE(gemm_experts_launch(P.x_gu, e->tm_gu[l], e->d_status, e->st));
        STAGE(gemm_experts_launch(P.x_down, e->tm_down[l], e->d_status, e->st));
        STAGE(launch_moe_combine(P.yg_out, P.row_active, P.R, NB, s.hidden, P.grp, P.down_out, e->st));
      } else if (!P.shorts) {
        STAGE(gemm_pair_launch(P.b_gu, e->tb_gu[l], P.R, e->d_status, e->st, &e->tb_gu96[l]));
        STAGE(gemm_pair_launch(P.b_down, e->tb_down[l], P.R, e->d_status, e->st));
      }
      continue;
    }
    if (P.wide) STAGE(gemm_pair_launch(P.b_qkv, e->tb_qkv[l], P.R, e->d_status, e->st, nullptr, nullptr, tr(4 * l + 0)));
    else STAGE(gemm_launch(P.p_qkv, &e->tm_qkv[l], e->d_status, e->st, tr(4 * l + 0), true));
    const GemmOut qkv = P.wide ? gemm_pair_out(P.b_qkv, P.R, P.plain_tiles) : P.p_qkv.out();
    if (e->mla) {
      // cache append and query parts -> q_lat = W_uk^T q_nope per head -> absorbed attention over the row's latent
      // pages (decode rows and prefill rows alike) -> [. | o] = W_kv_b o_lat per head -> the value part, split
      const MlaDims &md = e->md;
      const MlaCache cache{e->kv_pool + (size_t)l * e->layer_stride, e->d_block_table, e->max_blocks, e->B, (long long)e->pool_blocks, e->kv_run};
      STAGE(launch_mla_post(qkv, rows, e->d_rope, md, e->kv_norm[l], s.rms_eps, cache, P.RPH, P.qn_hi, P.qn_lo, P.q_rope,
                            e->d_status, e->st));
      STAGE(gemm_launch(P.p_uk, &e->tm_uk[l], e->d_status, e->st, nullptr, true));
      STAGE(launch_mla_attention(e->tm_c[l], e->tm_cv[l], P.q_lat, md.rank, (long long)P.RPH * md.rank, P.q_rope, e->d_block_table,
                                 e->max_blocks, nullptr, &rows, P.R, md, 1.0f / sqrtf((float)(md.nope + md.rope)), e->mla_splits,
                                 P.mla_ml, P.mla_po, nullptr, P.ol_hi, P.ol_lo, P.RPH, e->num_sms, e->d_status, true, e->st, e->kv_run));
      STAGE(gemm_launch(P.p_uv, &e->tm_uv[l], e->d_status, e->st, nullptr, true));
      STAGE(launch_mla_ao_split(P.uv_out, P.R, P.RPH, md, P.ao_hi, P.ao_lo, e->st));
      n += 3 + (&P == &e->dec ? 0 : 1);               // beyond the count below: two grouped GEMMs, the split, and in prefill too a second attention kernel
    } else {
    STAGE(launch_qkv_post(qkv, rows, e->d_rope, s.n_q_heads, kv, l, P.q, e->d_status, e->st));
    STAGE(launch_attention(e->tm_k4[l], e->tm_k4[l], P.q, rows, s.n_q_heads, kv, l, e->max_splits, P.att_work, P.att_n_work,
                           e->num_sms, P.part_acc, P.part_ml, P.att_pool + l, P.ao_hi, P.ao_lo, &P == &e->dec ? (e->whole_pairs ? 2 : 0) : 1,
                           e->d_status, e->st));
    }
    if (P.wide) STAGE(gemm_pair_launch(P.b_o, e->tb_o[l], P.R, e->d_status, e->st, nullptr, nullptr, tr(4 * l + 1)));
    else STAGE(gemm_launch(P.p_o, &e->tm_o[l], e->d_status, e->st, tr(4 * l + 1), true));
    GemmOut o = P.wide ? gemm_pair_out(P.b_o, P.R, P.plain_tiles) : P.p_o.out();
    STAGE(launch_resid_norm(P.h, s.hidden, nullptr, rows, &o, e->mlp_norm[l], s.rms_eps, P.xn_hi, P.xn_lo, e->st));
    if (dense_layer(e, l)) {
      STAGE(gemm_launch(P.p_gu_d, &e->tm_gu_d[l], e->d_status, e->st, nullptr, true));
      STAGE(launch_swiglu(P.p_gu_d.out(), P.R, e->dense_ffn, P.ff_hi, P.ff_lo, e->st));
      STAGE(gemm_launch(P.p_down_d, &e->tm_down_d[l], e->d_status, e->st, nullptr, true));
      n += 9 + (&P == &e->dec ? 1 : 0);
      continue;
    } else if (e->moe_E && P.grouped) {
      // router -> top-k weights -> rows grouped by expert -> gate / up, SwiGLU and down per group -> the row's
      // experts summed in ascending expert id
      const int NB = e->moe_E + e->moe_S;
      STAGE(launch_moe_router(P.xn_hi, P.xn_lo, s.hidden, e->router[l], P.R, e->moe_E, e->moe_S, e->moe_K, e->moe_renorm, P.moe_w, nullptr,
                              nullptr, P.router_rs, e->st, P.row_active));
      STAGE(launch_moe_group(P.moe_w, P.row_active, P.R, e->moe_E, e->moe_S, e->moe_F, P.grp, e->st));
      STAGE(launch_moe_gather(P.xn_hi, P.xn_lo, s.hidden, P.grp, P.xg_hi, P.xg_lo, e->st));
      if (P.p_gug.sw_hi) {                            // routing weight and SwiGLU in the GEMM's epilogue
        STAGE(gemm_launch(P.p_gug, &e->tm_gu_half[l], e->d_status, e->st, nullptr, true));
        n -= 1;
      } else {
        STAGE(gemm_launch(P.p_gug, &e->tm_gu[l], e->d_status, e->st, nullptr, true));
        STAGE(launch_moe_swiglu_grouped(P.gug_out, P.moe_w, NB, e->moe_F, P.grp, P.hg_hi, P.hg_lo, e->st));
      }
      STAGE(gemm_launch(P.p_dng, &e->tm_down[l], e->d_status, e->st, nullptr, true));
      STAGE(launch_moe_combine(P.yg_out, P.row_active, P.R, NB, s.hidden, P.grp, P.down_out, e->st));
      n += 13 + (&P == &e->dec ? 1 : 0);
      continue;
    } else if (P.select) {
      // router -> top-k weights and the rows' experts -> gate / up with routing weight and SwiGLU, then down, per selected
      // expert for all rows -> the row's experts summed in ascending expert id
      STAGE(launch_moe_router(P.xn_hi, P.xn_lo, s.hidden, e->router[l], P.R, e->moe_E, e->moe_S, e->moe_K, e->moe_renorm, P.moe_w, nullptr,
                              nullptr, P.router_rs, e->st, P.row_active, P.moe_sel));
      STAGE(gemm_launch(P.p_gug, &e->tm_gu_half[l], e->d_status, e->st, tr(4 * l + 2), true));
      STAGE(gemm_launch(P.p_dng, &e->tm_down[l], e->d_status, e->st, tr(4 * l + 3), true));
      STAGE(launch_moe_combine_select(P.yg_out, P.moe_sel, e->moe_K + e->moe_S, P.BN, P.R, s.hidden, P.down_out, e->st));
      n += 10 + (&P == &e->dec ? 1 : 0);
      continue;
    } else if (e->moe_E) {
      // router -> top-k weights -> all experts' gate / up (rows that did not select a tile's expert are not
      // stored) -> masked, weighted SwiGLU; the down GEMM then sums over the row's experts in its accumulator
      STAGE(launch_moe_router(P.xn_hi, P.xn_lo, s.hidden, e->router[l], P.R, e->moe_E, e->moe_S, e->moe_K, e->moe_renorm, P.moe_w, nullptr,
                              nullptr, P.router_rs, e->st));
      if (P.p_gu.sw_hi) {                             // routing weight and SwiGLU in the GEMM's epilogue
        STAGE(gemm_launch(P.p_gu, &e->tm_gu_half[l], e->d_status, e->st, tr(4 * l + 2), true));
      } else {                                        // (the router is the one kernel beyond the count below)
        STAGE(gemm_launch(P.p_gu, &e->tm_gu[l], e->d_status, e->st, tr(4 * l + 2), true));
        STAGE(launch_moe_swiglu(P.p_gu.out(), P.moe_w, P.R, e->moe_F, e->moe_E + e->moe_S, P.ff_hi, P.ff_lo, e->st));
        n += 1;
      }
    } else if (P.wide) {
      STAGE(gemm_pair_launch(P.b_gu, e->tb_gu[l], P.R, e->d_status, e->st, &e->tb_gu96[l], nullptr, tr(4 * l + 2)));
      STAGE(gemm_pair_launch(P.b_down, e->tb_down[l], P.R, e->d_status, e->st, nullptr, nullptr, tr(4 * l + 3)));
      n += 9;
      continue;
    } else {
      if (P.p_gu.sw_hi) {                             // SwiGLU in the GEMM's epilogue
        STAGE(gemm_launch(P.p_gu, &e->tm_gu_half[l], e->d_status, e->st, tr(4 * l + 2), true));
        n -= 1;
      } else {
        STAGE(gemm_launch(P.p_gu, &e->tm_gu[l], e->d_status, e->st, tr(4 * l + 2), true));
        STAGE(launch_swiglu(P.p_gu.out(), P.R, s.ffn, P.ff_hi, P.ff_lo, e->st));
      }
    }
    STAGE(gemm_launch(P.p_down, &e->tm_down[l], e->d_status, e->st, tr(4 * l + 3), true));
    n += 9 + (&P == &e->dec ? 1 : 0);   // decode attention is two kernels (splits, combine)
  }
  if (&P != &e->dec && !normed) {                   // prefill: the final norm
    const GemmOut last = ffn_out(e, P, s.n_layers - 1);
    STAGE(launch_resid_norm(P.h, s.hidden, nullptr, rows, &last, e->final_norm, s.rms_eps, P.xn_hi, P.xn_lo, e->st, many));
  }
#undef STAGE
  if (launches) *launches += n;
  return CORUN_OK;
}

int launch_lm_head(corun_engine *e, const Program &P) {
  if (P.wide) {
    CK(gemm_pair_launch(P.b_lm, e->tb_lm, P.R, e->d_status, e->st));
    CK(gemm_pair_fixup_launch(P.b_lm, P.R, e->st));
  } else {
    CK(gemm_launch(P.p_lm, nullptr, e->d_status, e->st, nullptr, true));
    CK(gemm_fixup_launch(P.p_lm, e->st, true));
  }
  return CORUN_OK;
}

// One decode iteration on the stream (what the graph captures).
int enqueue_decode_body(corun_engine *e, int *launches) {
  Program &P = e->dec;
  const corun_shape &s = e->sh;
  int n = 0;
  // mask and seeds are read from the pinned staging buffers by the first kernel, tokens and status are written to
  // them by the last one (zero-copy): a copy node in a graph costs several microseconds, these are 836 bytes
  CK(launch_prepare_rows(e->h_active, e->h_seeds, e->d_seeds, e->d_in_use, e->d_ctx, e->d_pending, e->d_temp, e->d_top_p, e->d_step, e->B,
                         P.row_token, P.row_pos, P.row_active, P.row_slot, P.do_sample, P.row_temp, P.row_top_p, P.row_step, P.slot_row,
                         P.row_blocks, e->st));
  n += 1;
  RC(run_layers(e, P, &n));
  if (!(e->eager && e->stop_after >= 0)) {   // (debug) a truncated layer stack skips the tail too
    const Rows rows{P.row_token, P.row_pos, P.row_active, P.row_slot, P.R};
    GemmOut prev = ffn_out(e, P, s.n_layers - 1);
    CK(launch_resid_norm(P.h, s.hidden, nullptr, rows, &prev, e->final_norm, s.rms_eps, P.xn_hi, P.xn_lo, e->st));
    RC(launch_lm_head(e, P));
    SampleArgs sa{P.logits, s.vocab, P.do_sample, P.row_temp, P.row_top_p, e->d_seeds, P.row_step, nullptr, P.sampled};   // all by row
    CK(launch_sampler(sa, P.R, e->st, true));
    CK(launch_advance(P.slot_row, P.row_active, P.sampled, e->B, e->d_ctx, e->d_step, e->d_pending, e->h_out_tokens, e->d_status, e->h_status,
                      e->st));
    n += 4 + (P.wide ? gemm_pair_has_parts(P.b_lm, P.R) : P.p_lm.n_split_tiles ? 1 : 0);
  }
  if (e->eager && e->stop_after >= 0)            // (debug) no last kernel ran: fetch the status word the plain way
    CK(cudaMemcpyAsync(e->h_status, e->d_status, sizeof(int), cudaMemcpyDeviceToHost, e->st));
  if (launches) *launches = n;
  return CORUN_OK;
}

int check_status(corun_engine *e) {
  if (*e->h_status == 4) return CORUN_EINVAL;   // DEV_BAD_INDEX: an index check of a -DCORUN_CHECKED build failed
  if (*e->h_status != 0) return CORUN_ETIMEOUT;
  return CORUN_OK;
}

int sync_stream(corun_engine *e) {
  CK(cudaStreamSynchronize(e->st));
  e->in_flight = false;
  return CORUN_OK;
}

int reserve_blocks(corun_engine *e, int slot, int reserve_len) {
  const int run_tokens = KV_BLOCK * e->kv_run;
  const int need = (reserve_len + run_tokens - 1) / run_tokens;   // runs
  if ((size_t)need > e->free_blocks.size()) return CORUN_ENOSPACE;
  std::vector<int> &mine = e->slot_blocks[slot];
  mine.clear();
  int *row = e->h_table + (size_t)slot * e->max_blocks;   // pinned; the last copy from it has completed: the slot was free
  memset(row, 0, (size_t)e->max_blocks * sizeof(int));
  for (int i = 0; i < need; ++i) {
    mine.push_back(e->free_blocks.back());
    e->free_blocks.pop_back();
    for (int j = 0; j < e->kv_run && i * e->kv_run + j < e->max_blocks; ++j) row[i * e->kv_run + j] = mine.back() * e->kv_run + j;
  }
  CK(cudaMemcpyAsync(e->d_block_table + (size_t)slot * e->max_blocks, row, e->max_blocks * sizeof(int), cudaMemcpyHostToDevice, e->st));
  return CORUN_OK;
}

int set_slot_state(corun_engine *e, int slot, int in_use, int ctx, int step, int pending, float temp, float top_p) {
  CK(launch_set_slot(SlotArrays{e->d_in_use, e->d_ctx, e->d_step, e->d_pending, e->d_temp, e->d_top_p}, slot, in_use, ctx, step, pending,
                     temp, top_p, e->st));
  return CORUN_OK;
}

bool slot_ok(const corun_engine *e, int slot) { return slot >= 0 && slot < e->B; }

}  // namespace

extern "C" {

int corun_last_cuda_error(void) { return g_last_cuda_error; }

const char *corun_strerror(int st) {
  switch (st) {
    case CORUN_OK: return "ok";
    case CORUN_EINVAL: return "invalid argument";
    case CORUN_ESLOT: return "bad slot (out of range, busy, or empty)";
    case CORUN_ENOSPACE: return "KV pool cannot hold the reserved sequence";
    case CORUN_ECTX: return "an active slot is at its reserved length";
    case CORUN_ECUDA: return "CUDA error";
    case CORUN_ETIMEOUT: return "a bounded device-side wait expired";
    case CORUN_ENOMEM: return "out of memory";
    case CORUN_ELIMIT: return "size exceeds the fixed capacity of corun_gemm_static";
    default: return "unknown status";
  }
}

static int engine_create(const corun_shape *shape, const corun_weights *w, const corun_moe_layers *moe,
                         const corun_mla_layers *mla, int32_t B, int32_t max_context, int32_t kv_block,
                         int64_t kv_pool_blocks, void *cuda_stream, corun_engine **out) {
  if (!shape || !w || !out) return CORUN_EINVAL;
  *out = nullptr;
  corun_shape s = *shape;
  if (s.n_layers < 1) return CORUN_EINVAL;
  int first_dense = 0, dense_ffn = 0;                // MLA: layers with a dense feed-forward, and its width
  if (mla) {
    if (s.arch != 0 && s.arch != 1) return CORUN_EINVAL;
    s.arch = 0;
    if ((mla->kv_lora_rank != 256 && mla->kv_lora_rank != 512) || mla->qk_nope < 64 || mla->qk_nope % 64 || mla->qk_rope < 8 ||
        mla->qk_rope > 64 || mla->qk_rope % 8 || mla->v_head < 64 || (mla->qk_nope + mla->v_head) % 256 || s.n_q_heads < 1 ||
        s.n_q_heads > 16 || mla->first_dense < 0 || mla->first_dense > s.n_layers || (!moe && mla->first_dense != s.n_layers) ||
        !mla->kv_norm || !mla->wkv_b)
      return CORUN_EINVAL;
    for (int l = 0; l < s.n_layers; ++l)
      if (!mla->kv_norm[l] || !mla->wkv_b[l]) return CORUN_EINVAL;
    first_dense = mla->first_dense;
    dense_ffn = s.ffn;
    if (first_dense > 0 && (dense_ffn < 64 || dense_ffn % 64 || !w->wgate_up || !w->wdown)) return CORUN_EINVAL;
    for (int l = 0; l < first_dense; ++l)
      if (!w->wgate_up[l] || !w->wdown[l]) return CORUN_EINVAL;
    if (first_dense == s.n_layers) moe = nullptr;   // no expert layer at all
    s.head_dim = mla->v_head;                        // the o-projection's K is n_q_heads * v_head
    s.n_kv_heads = s.n_q_heads;
  }
  if (moe) {
    if (moe->n_experts < 1 || moe->n_experts > 256 || moe->top_k < 1 || moe->top_k > 16 || moe->top_k > moe->n_experts ||
        moe->expert_ffn < 64 || moe->expert_ffn % 64 || moe->n_shared < 0 || !moe->router || !moe->gate_up || !moe->down)
      return CORUN_EINVAL;
    for (int l = first_dense; l < s.n_layers; ++l)
      if (!moe->router[l] || !moe->gate_up[l] || !moe->down[l]) return CORUN_EINVAL;
    s.ffn = (moe->n_experts + moe->n_shared) * moe->expert_ffn;   // the feed-forward width the row program sees
  }
  if (s.arch != 0 || s.n_layers < 1 || s.hidden < 64 || s.hidden % 64 || s.ffn < 64 || s.ffn % 64 || s.vocab < 1)
    return CORUN_EINVAL;
  if (!mla && s.head_dim != 64 && s.head_dim != 128) return CORUN_EINVAL;
  if (s.n_q_heads < 1 || s.n_kv_heads < 1 || s.n_q_heads % s.n_kv_heads) return CORUN_EINVAL;
  const int group = s.n_q_heads / s.n_kv_heads;
  if (group != 1 && group != 2 && group != 4 && group != 8) return CORUN_EINVAL;
  if ((s.n_q_heads * s.head_dim) % 64) return CORUN_EINVAL;
  if (!(s.rms_eps >= 0.f) || !(s.rope_theta > 0.f)) return CORUN_EINVAL;
  // kv_block: 16, or (latent caches only) 64: pages of 16 tokens handed out in aligned runs of four
  if (B < 1 || B > 256 || max_context < 1 || max_context > 256 * ATT_SPLIT || !(kv_block == KV_BLOCK || (mla && kv_block == 4 * KV_BLOCK)) ||
      kv_pool_blocks < 0)
    return CORUN_EINVAL;
  if (!w->embed || !w->lm_head || !w->final_norm || !w->attn_norm || !w->wqkv || !w->wo || !w->mlp_norm ||
      (!moe && (!w->wgate_up || !w->wdown)))
    return CORUN_EINVAL;
  for (int l = 0; l < s.n_layers; ++l)
    if (!w->attn_norm[l] || !w->wqkv[l] || !w->wo[l] || !w->mlp_norm[l] || (!moe && (!w->wgate_up[l] || !w->wdown[l])))
      return CORUN_EINVAL;
  const int Lm = moe ? first_dense : 0;              // the first layer with experts (whose weights the plans are made on)

  int dev = 0;
  CK(cudaGetDevice(&dev));
  cudaDeviceProp prop;
  CK(cudaGetDeviceProperties(&prop, dev));
  if (prop.major != 10) return CORUN_ECUDA;   // tcgen05 / TMEM kernels: sm_100a only

  corun_engine *e = new (std::nothrow) corun_engine();
  if (!e) return CORUN_ENOMEM;
  auto fail = [&](int rc) {
    corun_destroy(e);
    return rc;
  };
  e->sh = s;
  e->B = B;
  e->max_ctx = max_context;
  e->kv_run = kv_block / KV_BLOCK;
  e->max_blocks = (max_context + kv_block - 1) / kv_block * e->kv_run;   // pages of 16 tokens, whole runs
  e->max_splits = (max_context + ATT_SPLIT - 1) / ATT_SPLIT;
  e->num_sms = prop.multiProcessorCount;
  e->st = (cudaStream_t)cuda_stream;
  if (!e->st) {   // the legacy default stream cannot be captured: use a private one
    if (cudaStreamCreateWithFlags(&e->st, cudaStreamNonBlocking) != cudaSuccess) return fail(CORUN_ECUDA);
    e->own_stream = true;
  }
  e->w0_qkv = w->wqkv[0];
  e->w0_o = w->wo[0];
  e->w0_gu = moe ? moe->gate_up[Lm] : w->wgate_up[0];
  e->w0_down = moe ? moe->down[Lm] : w->wdown[0];
  if (mla) {
    e->mla = true;
    e->md = MlaDims{s.n_q_heads, mla->kv_lora_rank, mla->qk_nope, mla->qk_rope, mla->v_head};
    e->first_dense = first_dense;
    e->dense_ffn = moe ? dense_ffn : 0;
    e->mla_splits = mla_max_splits(max_context);
    e->w0_uv = mla->wkv_b[0];
    if (moe && first_dense > 0) { e->w0_gu_d = w->wgate_up[0]; e->w0_down_d = w->wdown[0]; }
  }
  if (moe) {
    e->moe_E = moe->n_experts;
    e->moe_K = moe->top_k;
    e->moe_F = moe->expert_ffn;
    e->moe_S = moe->n_shared;
    e->moe_renorm = moe->renormalize ? 1 : 0;
  }
  e->pool_blocks = kv_pool_blocks ? kv_pool_blocks * e->kv_run : (int64_t)B * e->max_blocks;   // in pages of 16 tokens
  size_t free_before = 0, total_b = 0;
  if (!kv_pool_blocks && cudaMemGetInfo(&free_before, &total_b) != cudaSuccess) return fail(CORUN_ECUDA);
  e->chunk = 256;
  bool one_chunk_size = false;                      // the environment asks for chunks of its own size, for every prompt
  if (const char *c = getenv("CORUN_ATTN_WHOLE_PAIRS")) e->whole_pairs = atoi(c) != 0;   // ablation only
  if (const char *c = getenv("CORUN_PREFILL_CHUNK")) {
    const int v = atoi(c);
    if (v >= 16 && v <= 256 && v % 16 == 0) { e->chunk = v; one_chunk_size = true; }
  }
  e->embed = (const bf16 *)w->embed;
  e->lm_head = (const bf16 *)w->lm_head;
  e->final_norm = (const bf16 *)w->final_norm;
  const int H = s.hidden, QD = s.n_q_heads * s.head_dim, KD = s.n_kv_heads * s.head_dim, F = s.ffn;
  // prefill runs through the program of many rows where their projections and experts have a form for many rows
  const bool big_ok = !one_chunk_size &&
                      (!moe || (moe->n_experts % 8 == 0 && (2 * moe->expert_ffn) % GEMM_TILE_N == 0 && H % GEMM_TILE_N == 0 &&
                                !getenv("CORUN_MOE_PREFILL_DENSE")));
  // rows of a chunk: as many as all slots' longest prompts could fill (pieces start on attention tiles), at most PREFILL_BIG, and more
  // than half of that only where one prompt can be longer: the buffers of twice the rows make an engine's creation longer (8 slots of
  // 1024 tokens, 12 Qwen3-30B-A3B layers: 49 -> 94 ms)
  const long long big_rows = (long long)B * ((max_context + 127) / 128 * 128);
  const int big_most = std::min(PREFILL_BIG, std::max(PREFILL_BIG / 2, (max_context + 255) / 256 * 256));
  int big_cap = !big_ok ? 0 : big_rows < big_most ? (int)((big_rows + 255) / 256 * 256) : big_most;
  const bool wide = e->wide = pad16(B) >= (moe ? 129 : WIDE_ROWS) && s.vocab % 8 == 0;   // (Program::wide)
  if (wide && gemm_encode_map(&e->tb_lm, w->lm_head, s.vocab, H, 128)) return fail(CORUN_EINVAL);
  e->tm_qkv.resize(s.n_layers);
  e->tm_o.resize(s.n_layers);
  e->tm_gu.resize(s.n_layers);
  e->tm_down.resize(s.n_layers);
  const int moe_half = moe ? gemm_swiglu_blocks_half(moe->expert_ffn, moe->n_experts + moe->n_shared, e->num_sms) : 0;
  if (!moe || moe_half) e->tm_gu_half.resize(s.n_layers);
  for (int l = 0; l < s.n_layers; ++l) {
    e->attn_norm.push_back((const bf16 *)w->attn_norm[l]);
    e->mlp_norm.push_back((const bf16 *)w->mlp_norm[l]);
    int rc;
    const int qkv_rows = mla ? s.n_q_heads * (mla->qk_nope + mla->qk_rope) + mla->kv_lora_rank + mla->qk_rope : QD + 2 * KD;
    if ((rc = gemm_encode_map(&e->tm_qkv[l], w->wqkv[l], qkv_rows, H, GEMM_W_BOX))) return fail(rc);
    if ((rc = gemm_encode_map(&e->tm_o[l], w->wo[l], H, QD, GEMM_W_BOX))) return fail(rc);
    if (big_cap || wide) {                          // the programs of many rows
      if (e->tb_qkv.empty())
        for (auto *v : {&e->tb_qkv, &e->tb_o, &e->tb_gu, &e->tb_down, &e->tb_router, &e->tb_gu_half, &e->tb_gu96}) v->resize(s.n_layers);
      const bool experts = moe && l >= first_dense;
      const int Fd = moe ? dense_ffn : F;
      if ((rc = gemm_encode_map(&e->tb_qkv[l], w->wqkv[l], qkv_rows, H, 128)) || (rc = gemm_encode_map(&e->tb_o[l], w->wo[l], H, QD, 128)))
        return fail(rc);
      if (experts ? (rc = gemm_encode_map(&e->tb_router[l], moe->router[l], moe->n_experts, H, 128))
                  : ((moe && (rc = gemm_encode_map(&e->tb_gu_half[l], w->wgate_up[l], 2 * Fd, H, gemm_swiglu_half(Fd, e->num_sms)))) ||
                     (rc = gemm_encode_map(&e->tb_gu96[l], w->wgate_up[l], 2 * Fd, H, 96)) ||
                     (rc = gemm_encode_map(&e->tb_gu[l], w->wgate_up[l], 2 * Fd, H, 128)) || (rc = gemm_encode_map(&e->tb_down[l], w->wdown[l], H, Fd, 128))))
        return fail(rc);
    }
    if (moe && l < first_dense) {                   // a dense feed-forward layer of a decoder with expert layers
      if (e->tm_gu_d.empty()) { e->tm_gu_d.resize(s.n_layers); e->tm_down_d.resize(s.n_layers); }
      if ((rc = gemm_encode_map(&e->tm_gu_d[l], w->wgate_up[l], 2 * dense_ffn, H, GEMM_W_BOX))) return fail(rc);
      if ((rc = gemm_encode_map(&e->tm_down_d[l], w->wdown[l], H, dense_ffn, GEMM_W_BOX))) return fail(rc);
      continue;
    }
    if ((rc = gemm_encode_map(&e->tm_gu[l], moe ? moe->gate_up[l] : w->wgate_up[l], 2 * F, H, GEMM_W_BOX))) return fail(rc);
    if ((rc = gemm_encode_map(&e->tm_down[l], moe ? moe->down[l] : w->wdown[l], H, F, GEMM_W_BOX))) return fail(rc);
    if (!moe && (rc = gemm_encode_map(&e->tm_gu_half[l], w->wgate_up[l], 2 * F, H, gemm_swiglu_half(F, e->num_sms)))) return fail(rc);
    if (moe && moe_half && (rc = gemm_encode_map(&e->tm_gu_half[l], moe->gate_up[l], 2 * F, H, moe_half))) return fail(rc);
  }
  if (mla) {
    // the key up-projections transposed (q_lat = W_uk^T q_nope is a GEMM over rows of W_uk^T), and per layer
    // the maps of the two grouped up-projection GEMMs
    int rc;
    const MlaDims &md = e->md;
    const size_t per_layer = (size_t)md.nh * md.rank * md.nope;
    if ((rc = dmalloc(e->allocs, &e->w_ukT, per_layer * s.n_layers, false))) return fail(rc);
    e->tm_uk.resize(s.n_layers);
    e->tm_uv.resize(s.n_layers);
    // (contexts beyond 16384 would need more than half a GB of decompressed keys and values: the decode form serves them)
    e->big_mla_tiles = big_cap > 0 && md.nope == 128 && md.vh == 128 && max_context <= 16384;
    if (e->big_mla_tiles) {
      e->tb_uv.resize(s.n_layers);
      if ((rc = dmalloc(e->allocs, &e->kv_scale, (size_t)s.n_layers * md.nh, false))) return fail(rc);
    }
    for (int l = 0; l < s.n_layers; ++l) {
      e->kv_norm.push_back((const bf16 *)mla->kv_norm[l]);
      bf16 *dst = e->w_ukT + (size_t)l * per_layer;
      if (launch_mla_transpose_uk((const bf16 *)mla->wkv_b[l], md, dst, 0) != cudaSuccess) return fail(CORUN_ECUDA);
      if ((rc = gemm_encode_map(&e->tm_uk[l], dst, md.nh * md.rank, md.nope, GEMM_W_BOX))) return fail(rc);
      if ((rc = gemm_encode_map(&e->tm_uv[l], mla->wkv_b[l], md.nh * (md.nope + md.vh), md.rank, GEMM_W_BOX))) return fail(rc);
      if (e->big_mla_tiles) {
        if ((rc = gemm_encode_map(&e->tb_uv[l], mla->wkv_b[l], md.nh * 256, md.rank, 128))) return fail(rc);
        if (launch_mla_kv_scale((const bf16 *)mla->wkv_b[l], e->kv_norm[l], md, e->kv_scale + (size_t)l * md.nh, 0) != cudaSuccess)
          return fail(CORUN_ECUDA);
      }
    }
  }
  if (moe) {
    if (H > MOE_MAX_HIDDEN) return fail(CORUN_EINVAL);   // the router kernel keeps a row in shared memory
    if (moe_router_prepare() != cudaSuccess) return fail(CORUN_ECUDA);
    for (int l = 0; l < s.n_layers; ++l) {
      if (l >= first_dense && ((uintptr_t)moe->router[l] & 15u)) return fail(CORUN_EINVAL);
      e->router.push_back(l >= first_dense ? (const bf16 *)moe->router[l] : nullptr);
    }
  }

  auto &A = e->allocs;
  int rc;
  // the pool, and the maps of its layers
  auto make_pool = [&]() -> int {
    int rc;
    e->layer_stride = mla ? (size_t)e->pool_blocks * KV_BLOCK * (size_t)mla_token_halfs(e->md.rank + e->md.rope, e->kv_run)
                          : (size_t)e->pool_blocks * 2 * s.n_kv_heads * KV_BLOCK * s.head_dim;
    // zero-filled: masked positions of a page are multiplied by zero weights, so they must be finite
    if ((rc = dmalloc(A, &e->kv_pool, e->layer_stride * s.n_layers, true))) return rc;
    if (mla) {
      if (mla_attention_prepare() != cudaSuccess) return (int)CORUN_ECUDA;
      // one layer's pages: rows of rank + rope halfs, 16 per page
      e->tm_c.resize(s.n_layers);
      e->tm_cv.resize(s.n_layers);
      for (int l = 0; l < s.n_layers; ++l)
        if ((rc = mla_encode_maps(&e->tm_c[l], &e->tm_cv[l], e->kv_pool + (size_t)l * e->layer_stride, e->pool_blocks, e->md.rank, e->md.rope,
                                  e->kv_run)))
          return rc;
    } else {
      // one layer's pages seen as rows of hd halfs (16 rows per page and head, keys first, then values)
      const unsigned long long halfs = (unsigned long long)e->layer_stride;
      if (halfs / KV_BLOCK >= (1ull << 31)) return (int)CORUN_EINVAL;
      for (int l = 0; l < s.n_layers; ++l) {
        const __half *base = e->kv_pool + (size_t)l * e->layer_stride;
        // keys and values are cached alike, one view serves both: a tile's 16 tokens x head_dim in ONE box, [2 groups of 8 tokens][halves of 64 dims][8][64]
        const unsigned long long row_b = (unsigned long long)s.head_dim * 2;
        const unsigned long long d4[4] = {64, 8, (unsigned long long)(s.head_dim / 64), halfs / s.head_dim / 8};
        const unsigned long long s4[3] = {row_b, 128, 8 * row_b};
        const unsigned b4[4] = {64, 8, (unsigned)(s.head_dim / 64), 2};
        e->tm_k4.emplace_back();
        if ((rc = tma_encode_fp16_4d(&e->tm_k4[l], base, d4, s4, b4))) return rc;
      }
      if (attention_prepare() != cudaSuccess) return (int)CORUN_ECUDA;
    }
    return CORUN_OK;
  };
  if (kv_pool_blocks && (rc = make_pool())) return fail(rc);
  if ((rc = dmalloc(A, &e->d_block_table, (size_t)B * e->max_blocks))) return fail(rc);
  if ((rc = dmalloc(A, &e->d_in_use, B)) || (rc = dmalloc(A, &e->d_ctx, B)) || (rc = dmalloc(A, &e->d_step, B)) ||
      (rc = dmalloc(A, &e->d_pending, B)) || (rc = dmalloc(A, &e->d_temp, B)) || (rc = dmalloc(A, &e->d_top_p, B)) ||
      (rc = dmalloc(A, &e->d_seeds, B)) || (rc = dmalloc(A, &e->d_active, B)) || (rc = dmalloc(A, &e->d_out_tokens, B)) ||
      (rc = dmalloc(A, &e->d_status, 1)) || (rc = dmalloc(A, &e->d_pf_temp, FINISH_ROWS)) ||
      (rc = dmalloc(A, &e->d_pf_top_p, FINISH_ROWS)) || (rc = dmalloc(A, &e->d_pf_seed, FINISH_ROWS)) ||
      (rc = dmalloc(A, &e->d_pf_step, FINISH_ROWS)) || (rc = dmalloc(A, &e->d_pf_one, FINISH_ROWS)) ||
      (rc = dmalloc(A, &e->d_pf_tok, FINISH_ROWS)) || (rc = dmalloc(A, &e->pf_logits, (size_t)B * s.vocab)))
    return fail(rc);
  e->logits_row.assign((size_t)B, -1);
  {
    // cos/sin of pos * theta^(-2i/hd), evaluated in fp64 on the host (hd: the rotated width)
    const int rot = mla ? mla->qk_rope : s.head_dim, half = rot / 2;
    std::vector<float2> tab((size_t)max_context * half);
    std::vector<double> freq((size_t)half);
    for (int i = 0; i < half; ++i) freq[(size_t)i] = std::pow((double)s.rope_theta, -2.0 * (double)i / (double)rot);
    for (int p = 0; p < max_context; ++p)
      for (int i = 0; i < half; ++i) {
        const double ang = (double)p * freq[(size_t)i];
        tab[(size_t)p * half + i] = make_float2((float)std::cos(ang), (float)std::sin(ang));
      }
    if ((rc = dmalloc(A, &e->d_rope, tab.size(), false))) return fail(rc);
    if (cudaMemcpy(e->d_rope, tab.data(), tab.size() * sizeof(float2), cudaMemcpyHostToDevice) != cudaSuccess)
      return fail(CORUN_ECUDA);
    const std::vector<int> ones(FINISH_ROWS, 1);
    if (cudaMemcpy(e->d_pf_one, ones.data(), FINISH_ROWS * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess) return fail(CORUN_ECUDA);
  }
  e->slot_blocks.resize(B);
  e->in_use.assign(B, 0);
  e->ctx.assign(B, 0);
  e->reserve.assign(B, 0);
  e->step.assign(B, 0);
  {
    // all pinned staging in one allocation (each costs milliseconds)
    size_t off = 0;
    auto place = [&](size_t bytes) { const size_t o = off; off += (bytes + 255) / 256 * 256; return o; };
    const size_t o_active = place(B), o_seeds = place(B * sizeof(uint64_t)), o_tok = place(B * sizeof(int)), o_status = place(sizeof(int)),
                 o_first = place(B * sizeof(int)), o_table = place((size_t)B * e->max_blocks * sizeof(int)),
                 o_logits = place((size_t)s.vocab * sizeof(float)),
                 o_rows = place(((size_t)4 * PREFILL_BIG + 64 + 2 * (16 * (PREFILL_BIG / 64) * 3 + 1)) * sizeof(int));
    if (cudaMallocHost(&e->h_pinned, off) != cudaSuccess) return fail(CORUN_ENOMEM);
    char *h = (char *)e->h_pinned;
    e->h_active = (uint8_t *)(h + o_active);
    e->h_seeds = (uint64_t *)(h + o_seeds);
    e->h_out_tokens = (int *)(h + o_tok);
    e->h_status = (int *)(h + o_status);
    e->h_first = (int *)(h + o_first);
    e->h_table = (int *)(h + o_table);
    e->h_rows = (int *)(h + o_rows);
    e->h_logits = (float *)(h + o_logits);
    for (cudaEvent_t &ev : e->ev_logits)
      if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return fail(CORUN_ECUDA);
  }
  memset(e->h_active, 0, B);
  memset(e->h_seeds, 0, B * sizeof(uint64_t));
  *e->h_status = 0;

#ifdef CORUN_BUILD_DEBUG
  if (const char *ts = getenv("CORUN_TRACE_STEP")) {
    if (atoi(ts) != 0 && (rc = dmalloc(A, &e->step_trace, (size_t)4 * s.n_layers * e->num_sms * 8))) return fail(rc);
  }
#endif
  // expert layers of the decode program: above 64 padded rows the grouped form (an expert's rows gathered into blocks of
  // 64, of which as many are multiplied as there are, where every row through every expert keeps the tensor pipe as busy as the
  // weight stream); up to 64 rows the experts that a row selected (Program::select), each for all rows of the step
  const bool dec_grouped = e->moe_E > 0 && pad16(B) > 64 && !getenv("CORUN_MOE_DECODE_DENSE");
  if ((rc = program_create(e, e->dec, B, true, true, dec_grouped, true))) return fail(rc);
  // the decode step's first kernel says which blocks of rows hold a request (64 rows each up to 128 padded rows, 128
  // rows each above); the GEMMs leave the others out (the one-row program has one block)
  for (GemmPairPlan *pl : {&e->dec.b_qkv, &e->dec.b_o, &e->dec.b_gu, &e->dec.b_down, &e->dec.b_lm}) pl->row_blocks = e->dec.row_blocks;
  for (GemmPlan *pl : {&e->dec.p_qkv, &e->dec.p_o, &e->dec.p_gu, &e->dec.p_down, &e->dec.p_lm, &e->dec.p_gu_d, &e->dec.p_down_d})
    pl->row_blocks = e->dec.row_blocks;
  if (e->dec.select) e->dec.p_gug.row_blocks = e->dec.p_dng.row_blocks = e->dec.row_blocks;
  if ((rc = program_create(e, e->lm1, FINISH_ROWS, false, true))) return fail(rc);
  // Prefill: chunks of as many rows as there is room for (a caller's pool may leave little: 128 MiB stay free for the step's
  // graph); no value depends on that.  Where not even 256 rows fit, latent attention does without decompressed keys and values,
  // and at last the chunk program serves: other forms, with other low bits.
  while (big_cap) {
    size_t free_b = 0;
    rc = program_create_big(e, e->big, big_cap);
    if (rc == CORUN_OK && big_cap > 256 && cudaMemGetInfo(&free_b, &total_b) == cudaSuccess && free_b < (size_t)128 << 20) rc = CORUN_ENOMEM;
    if (rc != CORUN_ENOMEM) break;
    program_destroy(e->big);
    e->big = Program();
    if (big_cap > 256) big_cap = (big_cap / 2 + 255) / 256 * 256;
    else if (e->big_mla_tiles) e->big_mla_tiles = false;
    else big_cap = 0;
  }
  if (big_cap && rc) return fail(rc);
  if (!big_cap && (rc = program_create(e, e->pre, e->chunk, true, false, e->moe_E > 0 && !getenv("CORUN_MOE_PREFILL_DENSE")))) return fail(rc);
  // a prefill chunk is filled from row 0: the host says which blocks of rows it reaches (prefill_run)
  for (GemmPlan *pl : {&e->pre.p_qkv, &e->pre.p_o, &e->pre.p_gu, &e->pre.p_down, &e->pre.p_gu_d, &e->pre.p_down_d})
    pl->row_blocks = e->pre.row_blocks;
  if (!kv_pool_blocks) {
    // default size: a full reservation for every slot, or as many pages as fit beside 6 GiB for the engine's other buffers --
    // what is left of them, and 256 MiB, where these are larger --, whichever is less (admission then refuses what does not fit)
    size_t free_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return fail(CORUN_ECUDA);
    const size_t page_b = mla ? (size_t)s.n_layers * KV_BLOCK * (size_t)mla_token_halfs(mla->kv_lora_rank + mla->qk_rope, e->kv_run) * sizeof(__half)
                              : (size_t)s.n_layers * 2 * s.n_kv_heads * KV_BLOCK * s.head_dim * sizeof(__half);
    const size_t have = (size_t)6 << 30, used = free_before > free_b ? free_before - free_b : 0, least = (size_t)256 << 20;
    const size_t keep = used + least < have ? have - used : least;
    const int64_t fit = free_b > keep ? (int64_t)((free_b - keep) / page_b) : 0;
    if (fit < e->pool_blocks) e->pool_blocks = fit / e->kv_run * e->kv_run;
    if (e->pool_blocks < e->kv_run) return fail(CORUN_ENOMEM);
    if ((rc = make_pool())) return fail(rc);
  }
  {
    const int64_t n_runs = e->pool_blocks / e->kv_run;
    e->free_blocks.resize((size_t)n_runs);
    for (int64_t i = 0; i < n_runs; ++i) e->free_blocks[(size_t)i] = (int)(n_runs - 1 - i);
  }

  // the allocations above were cleared and filled through the legacy stream, which the engine's
  // stream does not wait for: drain the device once before the first launch
  if (cudaDeviceSynchronize() != cudaSuccess) return fail(CORUN_ECUDA);
  // eager warm-up on an all-padding batch (also validates every launch), then capture
  if ((rc = enqueue_decode_body(e, &e->decode_launches))) return fail(rc);
  if (cudaStreamSynchronize(e->st) != cudaSuccess) return fail(CORUN_ECUDA);
  if ((rc = check_status(e))) return fail(rc);
  if (cudaStreamBeginCapture(e->st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return fail(CORUN_ECUDA);
  rc = enqueue_decode_body(e, nullptr);
  cudaError_t ce = cudaStreamEndCapture(e->st, &e->graph);
  if (rc) return fail(rc);
  if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; return fail(CORUN_ECUDA); }
  ce = cudaGraphInstantiate(&e->graph_exec, e->graph, 0);
  if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; return fail(CORUN_ECUDA); }
  *out = e;
  return CORUN_OK;
}

int corun_init(const corun_shape *shape, const corun_weights *w, int32_t B, int32_t max_context, int32_t kv_block,
               int64_t kv_pool_blocks, void *cuda_stream, corun_engine **out) {
  return engine_create(shape, w, nullptr, nullptr, B, max_context, kv_block, kv_pool_blocks, cuda_stream, out);
}

int corun_init_moe(const corun_shape *shape, const corun_weights *w, const corun_moe_layers *moe, int32_t B,
                   int32_t max_context, int32_t kv_block, int64_t kv_pool_blocks, void *cuda_stream, corun_engine **out) {
  if (!moe) return CORUN_EINVAL;
  return engine_create(shape, w, moe, nullptr, B, max_context, kv_block, kv_pool_blocks, cuda_stream, out);
}

int corun_init_mla(const corun_shape *shape, const corun_weights *w, const corun_mla_layers *mla, const corun_moe_layers *moe,
                   int32_t B, int32_t max_context, int32_t kv_block, int64_t kv_pool_blocks, void *cuda_stream,
                   corun_engine **out) {
  if (!mla) return CORUN_EINVAL;
  return engine_create(shape, w, moe, mla, B, max_context, kv_block, kv_pool_blocks, cuda_stream, out);
}

void corun_destroy(corun_engine *e) {
  if (!e) return;
  cudaStreamSynchronize(e->st);
  if (e->graph_exec) cudaGraphExecDestroy(e->graph_exec);
  if (e->graph) cudaGraphDestroy(e->graph);
  program_destroy(e->dec);
  program_destroy(e->pre);
  program_destroy(e->big);
  program_destroy(e->lm1);
  e->allocs.release();
  for (cudaEvent_t ev : e->ev_logits)
    if (ev) cudaEventDestroy(ev);
  if (e->h_pinned) cudaFreeHost(e->h_pinned);
  if (e->own_stream) cudaStreamDestroy(e->st);
  delete e;
}

}  // extern "C"

namespace {

struct PfReq {
  int slot;
  const int32_t *tokens;
  int n, reserve;
  corun_sampling smp;
  uint64_t seed;
  int first;
};

// LM head -> sample with R(seed, 0) for up to FINISH_ROWS requests whose last prompt tokens are rows of the chunk that has
// just run (the final norm is in P.xn); the logits go to the slots' places among the prefill logits, the tokens to h_first
// (valid once the stream has drained).  A row's logits do not depend on the other rows of the product.
int prefill_finish(corun_engine *e, const Program &P, const std::pair<int, int> *fins, int n, PfReq *const *reqs) {
  const corun_shape &s = e->sh;
  Program &L = e->lm1;
  FinishRows f{};
  f.n = n;
  for (int i = 0; i < n; ++i) {
    const PfReq &r = *reqs[fins[i].first];
    f.row[i] = fins[i].second;
    f.temp[i] = r.smp.temperature;
    f.top_p[i] = r.smp.top_p;
    f.seed[i] = r.seed;
  }
  CK(launch_finish_rows(f, P.xn_hi, P.xn_lo, s.hidden, L.xn_hi, L.xn_lo, e->d_pf_temp, e->d_pf_top_p, e->d_pf_seed, e->st));
  CK(gemm_launch(L.p_lm, nullptr, e->d_status, e->st));
  CK(gemm_fixup_launch(L.p_lm, e->st, true, n));
  SampleArgs sa{L.logits, s.vocab, e->d_pf_one, e->d_pf_temp, e->d_pf_top_p, e->d_pf_seed, e->d_pf_step, nullptr,
                e->d_pf_tok};
  CK(launch_sampler(sa, n, e->st, true));
  for (int i = 0; i < n; ++i) {
    const PfReq &r = *reqs[fins[i].first];
    CK(cudaMemcpyAsync(e->pf_logits + (size_t)r.slot * s.vocab, L.logits + (size_t)i * s.vocab, (size_t)s.vocab * sizeof(float),
                       cudaMemcpyDeviceToDevice, e->st));
    CK(cudaMemcpyAsync(e->h_first + r.slot, e->d_pf_tok + i, sizeof(int), cudaMemcpyDeviceToHost, e->st));
    e->logits_row[(size_t)r.slot] = -1;            // corun_get_logits: the prefill's logits until the slot decodes
  }
  return CORUN_OK;
}

// Prefill of one or several requests, all short or all long, through the program of many rows (chunks of up to its `cap`
// rows, launched for the rows they hold) or, where an engine has none, the chunk program (chunks of `chunk` rows).  The
// rows of a chunk are dealt in request order; every piece of a request starts on a tile boundary of the
// prefill attention kernel (a tile's rows share one slot), so a chunk may hold pieces of several requests.
// Every kernel of the program treats its rows independently of each other and of where they sit in the
// chunk, and attention reads all keys -- the chunk's own too -- from the cache, so a request's values do not
// depend on how its prompt is cut into pieces nor on what else shares its chunks.
int prefill_run(corun_engine *e, Program &P, PfReq *const *reqs, int n_req);

int prefill_many(corun_engine *e, PfReq *reqs, int n_req) {
  RC(sync_stream(e));
  size_t need = 0;
  for (int i = 0; i < n_req; ++i) need += (size_t)(reqs[i].reserve + KV_BLOCK * e->kv_run - 1) / (KV_BLOCK * e->kv_run);   // runs
  if (need > e->free_blocks.size()) return CORUN_ENOSPACE;
  int rc = CORUN_OK;
  for (int i = 0; i < n_req && rc == CORUN_OK; ++i) rc = reserve_blocks(e, reqs[i].slot, reqs[i].reserve);
  std::vector<PfReq *> part[2];                     // short and long, by the prompt's own length
  for (int i = 0; i < n_req; ++i) part[e->big.pair && reqs[i].n > PREFILL_SMALL ? 1 : 0].push_back(&reqs[i]);
  for (int k = 0; k < 2 && rc == CORUN_OK; ++k) {
    if (part[k].empty()) continue;
    e->big.shorts = k == 0;
    rc = prefill_run(e, e->big.pair ? e->big : e->pre, part[k].data(), (int)part[k].size());   // (the chunk program takes any length)
  }
  for (int i = 0; i < n_req && rc == CORUN_OK; ++i) {
    PfReq &q = reqs[i];
    q.first = e->h_first[q.slot];
    rc = set_slot_state(e, q.slot, 1, q.n, 1, q.first, q.smp.temperature, q.smp.top_p);
    if (rc != CORUN_OK) break;
    e->in_use[q.slot] = 1;
    e->ctx[q.slot] = q.n;
    e->reserve[q.slot] = q.reserve;
    e->step[q.slot] = 1;
  }
  if (rc != CORUN_OK)                               // nothing was admitted: the pages go back to the pool
    for (int i = 0; i < n_req; ++i) {
      std::vector<int> &mine = e->slot_blocks[reqs[i].slot];
      if (e->in_use[reqs[i].slot]) continue;
      for (int b : mine) e->free_blocks.push_back(b);
      mine.clear();
    }
  return rc;
}

int prefill_run(corun_engine *e, Program &P, PfReq *const *reqs, int n_req) {
  const corun_shape &s = e->sh;
  const int CH = P.pair ? P.cap : e->chunk;
  int unit = 128 / (s.n_q_heads / s.n_kv_heads);    // tokens per attention tile
  const bool tiles = P.mla_tiles && !P.shorts;
  if (e->mla) unit = tiles ? 128 : 16;              // (16: no query tiles, every row is on its own)
  if (unit > CH || CH % unit) unit = CH;
  struct Piece { int slot, row0, rows, end; };      // a request's piece of the chunk; end: its tokens cached after it
  std::vector<Piece> pieces;
  std::vector<int> tok((size_t)CH), pos((size_t)CH), act((size_t)CH), slt((size_t)CH);
  std::vector<std::pair<int, int>> fins;           // (request, chunk row of its last prompt token)
  int fill = 0, pad_slot = reqs[0]->slot;
  auto run_chunk = [&]() -> int {
    const int rows_n = P.pair ? fill : CH;
    for (int i = fill; i < rows_n; ++i) { tok[i] = 0; pos[i] = 0; act[i] = 0; slt[i] = pad_slot; }
    int *h = e->h_rows;                             // pinned: token | position | active | slot of the chunk's rows
    const size_t bytes = (size_t)rows_n * sizeof(int);
    memcpy(h, tok.data(), bytes);
    memcpy(h + rows_n, pos.data(), bytes);
    memcpy(h + 2 * rows_n, act.data(), bytes);
    memcpy(h + 3 * rows_n, slt.data(), bytes);
    int *blocks = h + 4 * PREFILL_BIG, *tabs = blocks + 64;
    if (P.pair) {
      P.R = fill;
      P.row_pos = P.row_token + fill;
      P.row_active = P.row_pos + fill;
      P.row_slot = P.row_active + fill;
      CK(cudaMemcpyAsync(P.row_token, h, 4 * bytes, cudaMemcpyHostToDevice, e->st));
      if (e->mla) RC(set_mla_rows(e, P, fill, tabs));
      if (tiles) {                                  // whose tokens are gathered where
        int *tb = blocks + 32, at = 0;
        P.segs.n = (int)pieces.size();
        for (size_t k = 0; k < pieces.size(); ++k) {
          const Piece &pc = pieces[k];
          P.segs.slot[k] = pc.slot;
          P.segs.off[k] = at;
          P.segs.len[k] = pc.end;
          for (int t = pc.row0 / 128; t <= (pc.row0 + pc.rows - 1) / 128; ++t) tb[t] = at;
          at += (pc.end + 63) / 64 * 64;
        }
        P.kv_tokens = at;
        CK(cudaMemcpyAsync(P.tile_base, tb, (size_t)((fill + 127) / 128) * sizeof(int), cudaMemcpyHostToDevice, e->st));
      }
      if (P.shorts) {                               // which blocks of 64 rows exist
        const int nb = (fill + SHORT_ROWS - 1) / SHORT_ROWS;
        for (int b = 0; b < nb; ++b) blocks[b] = gemm_row_blocks(fill - b * SHORT_ROWS < SHORT_ROWS ? fill - b * SHORT_ROWS : SHORT_ROWS, 64);
        CK(cudaMemcpyAsync(P.row_blocks, blocks, nb * sizeof(int), cudaMemcpyHostToDevice, e->st));
      }
    } else {
      CK(cudaMemcpyAsync(P.row_token, h, bytes, cudaMemcpyHostToDevice, e->st));
      CK(cudaMemcpyAsync(P.row_pos, h + rows_n, bytes, cudaMemcpyHostToDevice, e->st));
      CK(cudaMemcpyAsync(P.row_active, h + 2 * rows_n, bytes, cudaMemcpyHostToDevice, e->st));
      CK(cudaMemcpyAsync(P.row_slot, h + 3 * rows_n, bytes, cudaMemcpyHostToDevice, e->st));
      // the chunk's rows are filled from row 0: the GEMMs leave out the blocks of rows behind the last one in use
      // (blocks of 64 rows up to 128 padded rows, of 128 rows above)
      const int blk = P.BN <= 128 ? 64 : 128;
      blocks[0] = gemm_row_blocks(fill, blk);
      CK(cudaMemcpyAsync(P.row_blocks, blocks, sizeof(int), cudaMemcpyHostToDevice, e->st));
    }
    RC(run_layers(e, P, nullptr));
    for (size_t i = 0; i < fins.size(); i += FINISH_ROWS)
      RC(prefill_finish(e, P, &fins[i], (int)(fins.size() - i < FINISH_ROWS ? fins.size() - i : FINISH_ROWS), reqs));
    CK(cudaStreamSynchronize(e->st));   // the staging arrays are reused by the next chunk
    fins.clear();
    pieces.clear();
    fill = 0;
    return CORUN_OK;
  };
  for (int r = 0; r < n_req; ++r) {
    const PfReq &q = *reqs[r];
    for (int done = 0; done < q.n;) {
      while (fill % unit) { tok[fill] = 0; pos[fill] = 0; act[fill] = 0; slt[fill] = pad_slot; ++fill; }   // rest of the tile before
      if (fill == CH) RC(run_chunk());
      const int take = q.n - done < CH - fill ? q.n - done : CH - fill;
      for (int i = 0; i < take; ++i) {
        tok[fill + i] = q.tokens[done + i];
        pos[fill + i] = done + i;
        act[fill + i] = 1;
        slt[fill + i] = q.slot;
      }
      if (take > 0) pieces.push_back(Piece{q.slot, fill, take, done + take});
      fill += take;
      done += take;
      pad_slot = q.slot;                            // padding up to the tile's end belongs to this request's tile
      if (done == q.n) fins.emplace_back(r, fill - 1);
      if (fill == CH) RC(run_chunk());
    }
  }
  if (fill > 0 || !fins.empty()) RC(run_chunk());
  CK(cudaMemcpyAsync(e->h_status, e->d_status, sizeof(int), cudaMemcpyDeviceToHost, e->st));
  CK(cudaStreamSynchronize(e->st));
  return check_status(e);
}

}  // namespace

extern "C" {

int corun_prefill(corun_engine *e, int32_t slot, const int32_t *tokens, int32_t n, int32_t reserve_len,
                  const corun_sampling *sampling, uint64_t seed, int32_t *out_first_token) {
  if (!e || !tokens || !sampling || n < 1 || reserve_len < n || reserve_len > e->max_ctx) return CORUN_EINVAL;
  if (!slot_ok(e, slot) || e->in_use[slot]) return CORUN_ESLOT;
  for (int i = 0; i < n; ++i)
    if (tokens[i] < 0 || tokens[i] >= e->sh.vocab) return CORUN_EINVAL;
  PfReq r{slot, tokens, n, reserve_len, *sampling, seed, -1};
  RC(prefill_many(e, &r, 1));
  if (out_first_token) *out_first_token = r.first;
  return CORUN_OK;
}

int corun_prefill_batch(corun_engine *e, int32_t n_req, const int32_t *slots, const int32_t *tokens,
                        const int32_t *n_tokens, const int32_t *reserve_lens, const corun_sampling *samplings,
                        const uint64_t *seeds, int32_t *out_first_tokens) {
  if (!e || n_req < 1 || !slots || !tokens || !n_tokens || !reserve_lens || !samplings || !seeds) return CORUN_EINVAL;
  std::vector<PfReq> reqs((size_t)n_req);
  size_t off = 0;
  for (int i = 0; i < n_req; ++i) {
    const int n = n_tokens[i];
    if (n < 1 || reserve_lens[i] < n || reserve_lens[i] > e->max_ctx) return CORUN_EINVAL;
    if (!slot_ok(e, slots[i]) || e->in_use[slots[i]]) return CORUN_ESLOT;
    for (int j = 0; j < i; ++j)
      if (slots[j] == slots[i]) return CORUN_ESLOT;
    for (int t = 0; t < n; ++t)
      if (tokens[off + t] < 0 || tokens[off + t] >= e->sh.vocab) return CORUN_EINVAL;
    reqs[i] = PfReq{slots[i], tokens + off, n, reserve_lens[i], samplings[i], seeds[i], -1};
    off += (size_t)n;
  }
  RC(prefill_many(e, reqs.data(), n_req));
  if (out_first_tokens)
    for (int i = 0; i < n_req; ++i) out_first_tokens[i] = reqs[i].first;
  return CORUN_OK;
}

int corun_decode_enqueue(corun_engine *e, const uint8_t *active, const uint64_t *seeds) {
  if (!e || !active || !seeds) return CORUN_EINVAL;
  for (int s = 0; s < e->B; ++s) {
    if (!active[s]) continue;
    if (!e->in_use[s]) return CORUN_ESLOT;
    if (e->ctx[s] + 1 > e->reserve[s]) return CORUN_ECTX;
  }
  bool same = e->staged_valid;
  for (int s = 0; s < e->B && same; ++s) {
    const uint8_t a = active[s] ? 1 : 0;
    if (e->h_active[s] != a || (a && e->h_seeds[s] != seeds[s])) same = false;
  }
  if (!same) {
    if (e->in_flight) RC(sync_stream(e));   // an earlier replay may still read the staging buffers
    for (int s = 0; s < e->B; ++s) {
      e->h_active[s] = active[s] ? 1 : 0;
      e->h_seeds[s] = active[s] ? seeds[s] : 0;
    }
    e->staged_valid = true;
  }
  if (e->eager) {
    RC(enqueue_decode_body(e, nullptr));
  } else {
    CK(cudaGraphLaunch(e->graph_exec, e->st));
  }
  e->in_flight = true;
  int row = 0;                                      // the step's rows: the slots with a request, ascending (prepare_rows)
  for (int s = 0; s < e->B; ++s)
    if (active[s]) {
      e->ctx[s] += 1;
      e->step[s] += 1;
      e->logits_row[(size_t)s] = row++;
    }
  return CORUN_OK;
}

int corun_decode_wait(corun_engine *e, int32_t *out_tokens) {
  if (!e) return CORUN_EINVAL;
  RC(sync_stream(e));
  if (out_tokens) memcpy(out_tokens, e->h_out_tokens, e->B * sizeof(int));
  return check_status(e);
}

int corun_decode_step(corun_engine *e, const uint8_t *active, const uint64_t *seeds, int32_t *out_tokens) {
  if (!out_tokens) return CORUN_EINVAL;
  RC(corun_decode_enqueue(e, active, seeds));
  return corun_decode_wait(e, out_tokens);
}

int corun_release(corun_engine *e, int32_t slot) {
  if (!e) return CORUN_EINVAL;
  if (!slot_ok(e, slot) || !e->in_use[slot]) return CORUN_ESLOT;
  RC(sync_stream(e));
  for (int b : e->slot_blocks[slot]) e->free_blocks.push_back(b);
  e->slot_blocks[slot].clear();
  RC(set_slot_state(e, slot, 0, 0, 0, 0, 0.f, 1.f));
  e->in_use[slot] = 0;
  e->ctx[slot] = 0;
  e->reserve[slot] = 0;
  e->step[slot] = 0;
  return CORUN_OK;
}

int corun_get_logits(corun_engine *e, int32_t slot, float *out) {
  if (!e || !out) return CORUN_EINVAL;
  if (!slot_ok(e, slot) || !e->in_use[slot]) return CORUN_ESLOT;
  // the logits of the slot's newest token: its row of the last decode step it took part in, else its prefill's
  const int row = e->logits_row[(size_t)slot];
  const float *src = row < 0 ? e->pf_logits + (size_t)slot * e->sh.vocab : e->dec.logits + (size_t)row * e->sh.vocab;
  const int vocab = e->sh.vocab, piece = vocab < LOGITS_SPLIT ? vocab : (vocab + LOGITS_PIECES - 1) / LOGITS_PIECES;
  for (int i = 0, at = 0; at < vocab; ++i, at += piece) {
    const int n = std::min(piece, vocab - at);
    CK(cudaMemcpyAsync(e->h_logits + at, src + at, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, e->st));
    CK(cudaEventRecord(e->ev_logits[i], e->st));
  }
  for (int i = 0, at = 0; at < vocab; ++i, at += piece) {
    CK(cudaEventSynchronize(e->ev_logits[i]));
    memcpy(out + at, e->h_logits + at, (size_t)std::min(piece, vocab - at) * sizeof(float));
  }
  e->in_flight = false;             // the last piece was behind all that the stream held
  return CORUN_OK;
}

int corun_force_token(corun_engine *e, int32_t slot, int32_t token) {
  if (!e || token < 0 || token >= e->sh.vocab) return CORUN_EINVAL;
  if (!slot_ok(e, slot) || !e->in_use[slot]) return CORUN_ESLOT;
  RC(sync_stream(e));
  CK(cudaMemcpyAsync(e->d_pending + slot, &token, sizeof(int), cudaMemcpyHostToDevice, e->st));
  CK(cudaStreamSynchronize(e->st));
  return CORUN_OK;
}

int corun_context_len(corun_engine *e, int32_t slot) {
  if (!e) return CORUN_EINVAL;
  if (!slot_ok(e, slot) || !e->in_use[slot]) return CORUN_ESLOT;
  return e->ctx[slot];
}

int64_t corun_free_blocks(corun_engine *e) { return e ? (int64_t)e->free_blocks.size() : (int64_t)CORUN_EINVAL; }

int corun_engine_info(corun_engine *e, int32_t *B, int32_t *max_context, int32_t *kv_block, int64_t *pool_blocks) {
  if (!e) return CORUN_EINVAL;
  if (B) *B = e->B;
  if (max_context) *max_context = e->max_ctx;
  if (kv_block) *kv_block = KV_BLOCK * e->kv_run;   // the unit pages are handed out in (corun_free_blocks counts these)
  if (pool_blocks) *pool_blocks = e->pool_blocks / e->kv_run;
  return CORUN_OK;
}

int corun_prefill_class(corun_engine *e, int32_t n_tokens, int32_t *prefill_class, int32_t *chunk_rows, int32_t *tile_rows) {
  if (!e || n_tokens < 1) return CORUN_EINVAL;
  const int cls = e->big.pair && n_tokens > PREFILL_SMALL ? 1 : 0;   // (as prefill_many divides them)
  int unit = 128 / (e->sh.n_q_heads / e->sh.n_kv_heads);
  if (e->mla) unit = cls && e->big.mla_tiles ? 128 : 16;
  if (unit > e->chunk || e->chunk % unit) unit = e->chunk;
  if (prefill_class) *prefill_class = cls;
  if (chunk_rows) *chunk_rows = e->chunk;
  if (tile_rows) *tile_rows = unit;
  return CORUN_OK;
}

int corun_prefill_geometry(corun_engine *e, int32_t *chunk_rows, int32_t *tile_rows) {
  return corun_prefill_class(e, 1, nullptr, chunk_rows, tile_rows);
}

// MLA engines: k holds the cached rows ([n][rank + rope]), v is not used (may be NULL).
static int latent_io(corun_engine *e, int slot, int layer, int pos0, int n, float *k, int write) {
  const int row = e->md.rank + e->md.rope;
  const size_t elems = (size_t)n * row;
  float *dk = nullptr;
  if (cudaMalloc(&dk, elems * sizeof(float)) != cudaSuccess) return CORUN_ENOMEM;
  const MlaCache cache{e->kv_pool + (size_t)layer * e->layer_stride, e->d_block_table, e->max_blocks, e->B, (long long)e->pool_blocks, e->kv_run};
  cudaError_t ce = cudaSuccess;
  if (write) ce = cudaMemcpyAsync(dk, k, elems * sizeof(float), cudaMemcpyHostToDevice, e->st);
  if (ce == cudaSuccess) ce = launch_mla_copy(cache, row, slot, pos0, n, dk, write, e->st);
  if (ce == cudaSuccess && !write) ce = cudaMemcpyAsync(k, dk, elems * sizeof(float), cudaMemcpyDeviceToHost, e->st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->st);
  cudaFree(dk);
  if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; return CORUN_ECUDA; }
  return CORUN_OK;
}

static int kv_io(corun_engine *e, int slot, int layer, int pos0, int n, float *k, float *v, int write) {
  if (e && e->mla && !v) v = k;                     // the latent cache has no second array
  if (!e || !k || !v || n < 0 || pos0 < 0 || layer < 0 || layer >= e->sh.n_layers) return CORUN_EINVAL;
  if (!slot_ok(e, slot) || !e->in_use[slot]) return CORUN_ESLOT;
  const int limit = write ? e->reserve[slot] : e->ctx[slot];
  if (pos0 + n > limit) return CORUN_EINVAL;
  if (n == 0) return CORUN_OK;
  RC(sync_stream(e));
  if (e->mla) {
    RC(latent_io(e, slot, layer, pos0, n, k, write));
    if (write && pos0 + n > e->ctx[slot]) {
      e->ctx[slot] = pos0 + n;
      const int c = e->ctx[slot];
      CK(cudaMemcpyAsync(e->d_ctx + slot, &c, sizeof(int), cudaMemcpyHostToDevice, e->st));
      CK(cudaStreamSynchronize(e->st));
    }
    return CORUN_OK;
  }
  const size_t elems = (size_t)n * e->sh.n_kv_heads * e->sh.head_dim;
  float *dk = nullptr, *dv = nullptr;
  if (cudaMalloc(&dk, elems * sizeof(float)) != cudaSuccess) return CORUN_ENOMEM;
  if (cudaMalloc(&dv, elems * sizeof(float)) != cudaSuccess) { cudaFree(dk); return CORUN_ENOMEM; }
  int rc = CORUN_OK;
  cudaError_t ce = cudaSuccess;
  // every copy is ordered on the engine's own stream: a host-synchronous cudaMemcpy from pageable
  // memory may return before its DMA has landed, and the engine's stream does not wait for the
  // legacy stream
  if (write) {
    ce = cudaMemcpyAsync(dk, k, elems * sizeof(float), cudaMemcpyHostToDevice, e->st);
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(dv, v, elems * sizeof(float), cudaMemcpyHostToDevice, e->st);
  }
  if (ce == cudaSuccess) ce = launch_kv_copy(kv_layout(e), layer, slot, pos0, n, dk, dv, write, e->st);
  if (ce == cudaSuccess && !write) {
    ce = cudaMemcpyAsync(k, dk, elems * sizeof(float), cudaMemcpyDeviceToHost, e->st);
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(v, dv, elems * sizeof(float), cudaMemcpyDeviceToHost, e->st);
  }
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->st);
  if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; rc = CORUN_ECUDA; }
  cudaFree(dk);
  cudaFree(dv);
  if (rc == CORUN_OK && write && pos0 + n > e->ctx[slot]) {
    e->ctx[slot] = pos0 + n;
    const int c = e->ctx[slot];
    CK(cudaMemcpyAsync(e->d_ctx + slot, &c, sizeof(int), cudaMemcpyHostToDevice, e->st));
    CK(cudaStreamSynchronize(e->st));
  }
  return rc;
}

int corun_debug_kv_read(corun_engine *e, int32_t slot, int32_t layer, int32_t pos0, int32_t n, float *k, float *v) {
  return kv_io(e, slot, layer, pos0, n, k, v, 0);
}
int corun_debug_kv_write(corun_engine *e, int32_t slot, int32_t layer, int32_t pos0, int32_t n, const float *k,
                         const float *v) {
  return kv_io(e, slot, layer, pos0, n, const_cast<float *>(k), const_cast<float *>(v), 1);
}

int corun_debug_adopt(corun_engine *e, int32_t slot, int32_t n_ctx, int32_t reserve_len, int32_t pending_token,
                      const corun_sampling *sampling, int32_t step) {
  if (!e || !sampling || n_ctx < 0 || reserve_len < n_ctx || reserve_len < 1 || reserve_len > e->max_ctx ||
      pending_token < 0 || pending_token >= e->sh.vocab || step < 0)
    return CORUN_EINVAL;
  if (!slot_ok(e, slot) || e->in_use[slot]) return CORUN_ESLOT;
  RC(sync_stream(e));
  RC(reserve_blocks(e, slot, reserve_len));
  RC(set_slot_state(e, slot, 1, n_ctx, step, pending_token, sampling->temperature, sampling->top_p));
  e->in_use[slot] = 1;
  e->ctx[slot] = n_ctx;
  e->reserve[slot] = reserve_len;
  e->step[slot] = step;
  return CORUN_OK;
}

int corun_debug_kv_fill(corun_engine *e, int32_t slot, int32_t n_ctx, float std, uint64_t seed) {
  if (!e || n_ctx < 0 || !(std >= 0.f)) return CORUN_EINVAL;
  if (!slot_ok(e, slot) || !e->in_use[slot]) return CORUN_ESLOT;
  if (n_ctx > e->reserve[slot]) return CORUN_EINVAL;
  RC(sync_stream(e));
  if (e->mla) {
    for (int l = 0; l < e->sh.n_layers; ++l) {
      const MlaCache cache{e->kv_pool + (size_t)l * e->layer_stride, e->d_block_table, e->max_blocks, e->B, (long long)e->pool_blocks, e->kv_run};
      CK(launch_mla_fill(cache, e->md.rank + e->md.rope, l, slot, n_ctx, std, seed, e->st));
    }
  } else {
    CK(launch_kv_fill(kv_layout(e), e->sh.n_layers, slot, n_ctx, std, seed, e->st));
  }
  CK(cudaMemcpyAsync(e->d_ctx + slot, &n_ctx, sizeof(int), cudaMemcpyHostToDevice, e->st));
  CK(cudaStreamSynchronize(e->st));
  e->ctx[slot] = n_ctx;
  return CORUN_OK;
}

int corun_debug_time_kernel(corun_engine *e, int32_t kind, int32_t reps, float *avg_ms) {
  if (!e || !avg_ms || reps < 1 || kind < 0 || kind > 13) return CORUN_EINVAL;
  if ((kind == 10 || kind == 11) && !e->mla) return CORUN_EINVAL;   // the up-projections of an MLA layer
  if (kind == 12 && !e->moe_E) return CORUN_EINVAL;                  // the router of an expert layer
  if (kind == 13 && !(e->moe_E && e->dec.grouped)) return CORUN_EINVAL;   // grouping + gather of the grouped form
  RC(sync_stream(e));
  Program &P = e->dec;
  const corun_shape &s = e->sh;
  const Rows rows{P.row_token, P.row_pos, P.row_active, P.row_slot, P.R};
  const KvLayout kv = kv_layout(e);
  cudaEvent_t a, b;
  CK(cudaEventCreate(&a));
  CK(cudaEventCreate(&b));
  int rc = CORUN_OK;
  for (int pass = 0; pass < 2 && rc == CORUN_OK; ++pass) {   // pass 0 warms up
    const int n = pass == 0 ? (reps < 3 ? reps : 3) : reps;
    cudaError_t ce = cudaEventRecord(a, e->st);
    for (int i = 0; i < n && ce == cudaSuccess; ++i) {
      int l = i % s.n_layers;         // rotate over the layers so that L2 cannot hold the weights
      // feed-forward kinds of a decoder with dense and expert layers: the expert layers
      if (e->mla && e->moe_E && (kind == 2 || kind == 3 || kind == 6 || kind == 8 || kind == 12 || kind == 13))
        l = e->first_dense + i % (s.n_layers - e->first_dense);
      GemmOut prev = ffn_out(e, P, l);
      const MlaCache mcache{e->mla ? e->kv_pool + (size_t)l * e->layer_stride : nullptr, e->d_block_table, e->max_blocks, e->B,
                            (long long)e->pool_blocks, e->kv_run};
      switch (kind) {
        // launched as in the step's graph: with programmatic stream serialization
        case 0: if (P.wide) { ce = gemm_pair_launch(P.b_qkv, e->tb_qkv[l], P.R, e->d_status, e->st); break; }
                ce = gemm_launch(P.p_qkv, &e->tm_qkv[l], e->d_status, e->st, nullptr, true); break;
        case 1: if (P.wide) { ce = gemm_pair_launch(P.b_o, e->tb_o[l], P.R, e->d_status, e->st); break; }
                ce = gemm_launch(P.p_o, &e->tm_o[l], e->d_status, e->st, nullptr, true); break;
        case 2: if ((P.grouped || P.select) && !dense_layer(e, l)) {   // the groups of the last step's last layer
                  ce = gemm_launch(P.p_gug, P.p_gug.sw_hi ? &e->tm_gu_half[l] : &e->tm_gu[l], e->d_status, e->st, nullptr, true);
                  if (ce == cudaSuccess && !P.p_gug.sw_hi)
                    ce = launch_moe_swiglu_grouped(P.gug_out, P.moe_w, e->moe_E + e->moe_S, e->moe_F, P.grp, P.hg_hi, P.hg_lo, e->st);
                  break;
                }
                if (P.wide && !e->moe_E) { ce = gemm_pair_launch(P.b_gu, e->tb_gu[l], P.R, e->d_status, e->st, &e->tb_gu96[l]); break; }
                ce = gemm_launch(P.p_gu, P.p_gu.sw_hi ? &e->tm_gu_half[l] : &e->tm_gu[l], e->d_status, e->st, nullptr, true); break;
        case 3: if (P.select && !dense_layer(e, l)) {    // down GEMM per selected expert + the sum over a row's experts
                  ce = gemm_launch(P.p_dng, &e->tm_down[l], e->d_status, e->st, nullptr, true);
                  if (ce == cudaSuccess) ce = launch_moe_combine_select(P.yg_out, P.moe_sel, e->moe_K + e->moe_S, P.BN, P.R, s.hidden, P.down_out, e->st);
                  break;
                }
                if (P.grouped && !dense_layer(e, l)) {   // per-group down GEMM + the sum over a row's experts
                  ce = gemm_launch(P.p_dng, &e->tm_down[l], e->d_status, e->st, nullptr, true);
                  if (ce == cudaSuccess) ce = launch_moe_combine(P.yg_out, P.row_active, P.R, e->moe_E + e->moe_S, s.hidden, P.grp, P.down_out, e->st);
                  break;
                }
                if (P.wide && !e->moe_E) { ce = gemm_pair_launch(P.b_down, e->tb_down[l], P.R, e->d_status, e->st); break; }
                ce = gemm_launch(P.p_down, &e->tm_down[l], e->d_status, e->st, nullptr, true); break;
        case 4: ce = launch_lm_head(e, P) == CORUN_OK ? cudaSuccess : cudaErrorUnknown;
                break;
        case 5: if (e->mla) {
                  ce = launch_mla_attention(e->tm_c[l], e->tm_cv[l], P.q_lat, e->md.rank, (long long)P.RPH * e->md.rank, P.q_rope,
                                            e->d_block_table, e->max_blocks, nullptr, &rows, P.R, e->md,
                                            1.0f / sqrtf((float)(e->md.nope + e->md.rope)), e->mla_splits, P.mla_ml, P.mla_po, nullptr,
                                            P.ol_hi, P.ol_lo, P.RPH, e->num_sms, e->d_status, true, e->st, e->kv_run);
                  break;
                }
                ce = cudaMemsetAsync(P.att_pool + l, 0, sizeof(int), e->st);   // the launch does not reset its pool counter
                if (ce == cudaSuccess)
                  ce = launch_attention(e->tm_k4[l], e->tm_k4[l], P.q, rows, s.n_q_heads, kv, l, e->max_splits, P.att_work,
                                        P.att_n_work, e->num_sms, P.part_acc, P.part_ml, P.att_pool + l,
                                        P.ao_hi, P.ao_lo, e->whole_pairs ? 2 : 0, e->d_status, e->st);
                break;
        case 6: ce = launch_resid_norm(P.h, s.hidden, nullptr, rows, &prev, e->attn_norm[l], s.rms_eps, P.xn_hi,
                                       P.xn_lo, e->st); break;
        case 7: if (e->mla) {   // (re-appends the rows' current positions: the same values)
                  ce = launch_mla_post(P.wide ? gemm_pair_out(P.b_qkv, P.R, P.plain_tiles) : P.p_qkv.out(), rows, e->d_rope, e->md, e->kv_norm[l], s.rms_eps, mcache, P.RPH, P.qn_hi, P.qn_lo,
                                       P.q_rope, e->d_status, e->st);
                  break;
                }
                ce = launch_qkv_post(P.wide ? gemm_pair_out(P.b_qkv, P.R, P.plain_tiles) : P.p_qkv.out(), rows, e->d_rope, s.n_q_heads, kv, l, P.q, e->d_status, e->st); break;
        case 8: if (P.p_gu.sw_hi || P.grouped || P.select || (P.wide && !e->moe_E)) break;   // no such kernel: the SwiGLU is in the GEMM's epilogue (grouped form: timed with kind 2)
                ce = e->moe_E ? launch_moe_swiglu(P.p_gu.out(), P.moe_w, P.R, e->moe_F, e->moe_E + e->moe_S, P.ff_hi, P.ff_lo, e->st)
                              : launch_swiglu(P.p_gu.out(), P.R, s.ffn, P.ff_hi, P.ff_lo, e->st);
                break;
        case 9: {
          SampleArgs sa{P.logits, s.vocab, P.do_sample, P.row_temp, P.row_top_p, e->d_seeds, P.row_step, nullptr, P.sampled};
          ce = launch_sampler(sa, P.R, e->st);
          break;
        }
        case 10: ce = gemm_launch(P.p_uk, &e->tm_uk[l], e->d_status, e->st, nullptr, true); break;
        case 11: ce = gemm_launch(P.p_uv, &e->tm_uv[l], e->d_status, e->st, nullptr, true);
                 if (ce == cudaSuccess) ce = launch_mla_ao_split(P.uv_out, P.R, P.RPH, e->md, P.ao_hi, P.ao_lo, e->st);
                 break;
        case 13: ce = launch_moe_group(P.moe_w, P.row_active, P.R, e->moe_E, e->moe_S, e->moe_F, P.grp, e->st);
                 if (ce == cudaSuccess) ce = launch_moe_gather(P.xn_hi, P.xn_lo, s.hidden, P.grp, P.xg_hi, P.xg_lo, e->st);
                 break;
        case 12: ce = launch_moe_router(P.xn_hi, P.xn_lo, s.hidden, e->router[l], P.R, e->moe_E, e->moe_S, e->moe_K, e->moe_renorm,
                                        P.moe_w, nullptr, nullptr, P.router_rs, e->st, P.row_active, P.moe_sel);
                 break;
      }
    }
    if (ce == cudaSuccess) ce = cudaEventRecord(b, e->st);
    if (ce == cudaSuccess) ce = cudaEventSynchronize(b);
    float ms = 0.f;
    if (ce == cudaSuccess) ce = cudaEventElapsedTime(&ms, a, b);
    if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; rc = CORUN_ECUDA; }
    *avg_ms = ms / (float)n;
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  return rc;
}

#ifdef CORUN_BUILD_DEBUG   // kernel timelines: not part of the serving build
int corun_debug_gemm_trace(corun_engine *e, int32_t kind, int32_t layer, uint64_t *stamps, int32_t *n_ctas) {
  if (!e || !stamps || !n_ctas || kind < 0 || kind > 4 || layer < 0 || layer >= e->sh.n_layers) return CORUN_EINVAL;
  RC(sync_stream(e));
  Program &P = e->dec;
  const bool ffn = kind == 2 || kind == 3, experts = e->moe_E && !dense_layer(e, layer);
  const bool pairs = P.wide && !(ffn && e->moe_E), selected = ffn && experts && P.select;
  const GemmPairPlan *pp[5] = {&P.b_qkv, &P.b_o, &P.b_gu, &P.b_down, &P.b_lm};
  const GemmPlan *pl[5] = {&P.p_qkv, &P.p_o, selected ? &P.p_gug : &P.p_gu, selected ? &P.p_dng : &P.p_down, &P.p_lm};
  const GemmPlan &p = *pl[kind];
  // expert layers in their grouped form, and dense ones beside expert layers: no such GEMM
  if (pairs ? false : !p.grid || (ffn && dense_layer(e, layer))) return CORUN_EINVAL;
  const size_t n = (size_t)(pairs ? gemm_pair_ctas(*pp[kind], P.R, kind == 2) : p.grid) * 8;
  unsigned long long *d = nullptr;
  if (cudaMalloc(&d, n * sizeof(unsigned long long)) != cudaSuccess) return CORUN_ENOMEM;
  cudaError_t ce = cudaMemsetAsync(d, 0, n * sizeof(unsigned long long), e->st);
  for (int i = 0; i < 3 && ce == cudaSuccess; ++i) {   // last one counts
    if (pairs) {
      const CUtensorMap *tb[5] = {&e->tb_qkv[layer], &e->tb_o[layer], &e->tb_gu[layer], &e->tb_down[layer], &e->tb_lm};
      ce = gemm_pair_launch(*pp[kind], *tb[kind], P.R, e->d_status, e->st, kind == 2 ? &e->tb_gu96[layer] : nullptr, nullptr, d);
    } else {
      const CUtensorMap *tm[5] = {&e->tm_qkv[layer], &e->tm_o[layer], p.sw_hi ? &e->tm_gu_half[layer] : &e->tm_gu[layer], &e->tm_down[layer], nullptr};
      ce = gemm_launch(p, tm[kind], e->d_status, e->st, d);
    }
  }
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(stamps, d, n * sizeof(unsigned long long), cudaMemcpyDeviceToHost, e->st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->st);
  cudaFree(d);
  if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; return CORUN_ECUDA; }
  *n_ctas = (int32_t)(n / 8);
  return CORUN_OK;
}

int corun_debug_attn_trace(corun_engine *e, int32_t layer, uint64_t *stamps, int32_t *n_ctas) {
  if (!e || !stamps || !n_ctas || layer < 0 || layer >= e->sh.n_layers || e->mla) return CORUN_EINVAL;
  RC(sync_stream(e));
  Program &P = e->dec;
  const corun_shape &s = e->sh;
  const Rows rows{P.row_token, P.row_pos, P.row_active, P.row_slot, P.R};
  const size_t n = (size_t)e->num_sms * 64 * 8;
  unsigned long long *d = nullptr;
  if (cudaMalloc(&d, n * sizeof(unsigned long long)) != cudaSuccess) return CORUN_ENOMEM;
  cudaError_t ce = cudaMemsetAsync(d, 0, n * sizeof(unsigned long long), e->st);
  for (int i = 0; i < 2 && ce == cudaSuccess; ++i) {
    ce = cudaMemsetAsync(P.att_pool + layer, 0, sizeof(int), e->st);   // the launch does not reset its pool counter
    if (ce == cudaSuccess)
      ce = launch_attention(e->tm_k4[layer], e->tm_k4[layer], P.q, rows, s.n_q_heads, kv_layout(e), layer, e->max_splits,
                            P.att_work, P.att_n_work, e->num_sms, P.part_acc, P.part_ml, P.att_pool + layer,
                            P.ao_hi, P.ao_lo, e->whole_pairs ? 2 : 0, e->d_status, e->st, i == 1 ? d : nullptr);   // only the second launch is recorded
  }
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(stamps, d, n * sizeof(unsigned long long), cudaMemcpyDeviceToHost, e->st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->st);
  cudaFree(d);
  if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; return CORUN_ECUDA; }
  *n_ctas = e->num_sms;
  return CORUN_OK;
}

int corun_debug_step_trace(corun_engine *e, uint64_t *stamps, int64_t n) {
  if (!e || !stamps) return CORUN_EINVAL;
  if (!e->step_trace) return CORUN_EINVAL;    // the engine was not created with CORUN_TRACE_STEP=1
  const int64_t have = (int64_t)4 * e->sh.n_layers * e->num_sms * 8;
  if (n != have) return CORUN_EINVAL;
  RC(sync_stream(e));
  CK(cudaMemcpyAsync(stamps, e->step_trace, (size_t)n * sizeof(uint64_t), cudaMemcpyDeviceToHost, e->st));
  CK(cudaStreamSynchronize(e->st));
  return CORUN_OK;
}

#endif  // CORUN_BUILD_DEBUG

int corun_debug_read(corun_engine *e, int32_t which, float *out, int64_t n) {
  if (!e || !out || n < 0) return CORUN_EINVAL;
  RC(sync_stream(e));
  Program &P = e->dec;
  const corun_shape &s = e->sh;
  const size_t QD = (size_t)s.n_q_heads * s.head_dim;
  const float *src = nullptr;
  size_t have = 0;
  switch (which) {
    case 0: src = P.q; have = (size_t)P.R * QD; break;
    case 1: src = P.part_acc; have = (size_t)P.R * s.n_q_heads * e->max_splits * s.head_dim; break;
    case 2: src = P.part_ml; have = (size_t)P.R * s.n_q_heads * e->max_splits * 2; break;
    case 3: src = P.h; have = (size_t)P.R * s.hidden; break;
    case 4: src = (const float *)P.ao_hi; have = (size_t)P.BN * QD / 2; break;
    case 5: src = (const float *)P.ao_lo; have = (size_t)P.BN * QD / 2; break;
    case 6: src = P.o_out; have = (size_t)P.R * s.hidden; break;
    case 7: src = P.ws ? P.ws : P.pair_part; have = P.ws ? gemm_ws_floats(e->num_sms, P.BN) : P.pair_part_floats; break;
    default: return CORUN_EINVAL;
  }
  if (!src || (size_t)n > have) return CORUN_EINVAL;
  CK(cudaMemcpyAsync(out, src, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, e->st));
  CK(cudaStreamSynchronize(e->st));
  return CORUN_OK;
}

int corun_debug_set_eager(corun_engine *e, int32_t eager) {
  if (!e) return CORUN_EINVAL;
  RC(sync_stream(e));
  e->eager = eager != 0;
  e->stop_after = eager > 1 ? eager - 2 : -1;   // eager = 2 + k: stop the layer stack after k stages
  return CORUN_OK;
}

int corun_decode_launches(corun_engine *e) { return e ? e->decode_launches : CORUN_EINVAL; }

int corun_debug_gemm(const void *W, int32_t N, int32_t K, const float *X, int32_t R, float *out, void *cuda_stream) {
  if (!W || !X || !out || N < 1 || K < 64 || K % 64 || R < 1 || R > 256) return CORUN_EINVAL;
  // 16-byte stores of the output, tensor-map loads of W: misaligned buffers are refused before any launch
  if (((uintptr_t)out & 15u) || ((uintptr_t)W & 15u) || ((uintptr_t)X & 3u)) return CORUN_EINVAL;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int dev = 0, sms = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int BN = pad16(R);
  std::vector<void *> keep;
  bf16 *hi = nullptr, *lo = nullptr;
  float *ws = nullptr;
  int *status = nullptr;
  int rc = CORUN_OK;
  GemmPlan p;
  if ((rc = dmalloc(keep, &hi, (size_t)BN * K)) == 0 && (rc = dmalloc(keep, &lo, (size_t)BN * K)) == 0 &&
      (rc = dmalloc(keep, &ws, gemm_ws_floats(sms, BN))) == 0 && (rc = dmalloc(keep, &status, 1)) == 0 &&
      (rc = gemm_plan_create(&p, W, N, K, hi, lo, R, BN, out, ws, sms)) == 0) {
    cudaError_t ce = cudaDeviceSynchronize();   // allocations were cleared through the legacy stream
    if (ce == cudaSuccess) ce = launch_split(X, R, K, hi, lo, st);
    if (ce == cudaSuccess) ce = gemm_launch(p, nullptr, status, st);
    if (ce == cudaSuccess) ce = gemm_fixup_launch(p, st);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
    int hs = 0;
    if (ce == cudaSuccess) ce = cudaMemcpy(&hs, status, sizeof(int), cudaMemcpyDeviceToHost);
    if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; rc = CORUN_ECUDA; }
    else if (hs != 0) rc = CORUN_ETIMEOUT;
  }
  gemm_plan_destroy(&p);
  for (void *q : keep) cudaFree(q);
  return rc;
}

int corun_debug_gemm_pair(int32_t form, const void *W, int32_t N, int32_t K, const float *X, int32_t R, float *out,
                          void *cuda_stream) {
  const bool decode = form >= 3;
  if (decode) form -= 3;
  if (form < 0 || form > 2 || (decode && form > 1) || !W || !X || !out || N < 8 || K < 64 || K % 64 || R < 1 || R > (decode ? 256 : PREFILL_BIG))
    return CORUN_EINVAL;
  if (form == 0 ? N % 8 : form == 1 ? N % 128 : N % GEMM_TILE_N) return CORUN_EINVAL;
  if (((uintptr_t)out & 15u) || ((uintptr_t)W & 15u) || ((uintptr_t)X & 3u)) return CORUN_EINVAL;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int dev = 0, sms = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int cap = (R + 255) / 256 * 256, F = N / 2, nh = N / GEMM_TILE_N;
  const size_t c = (size_t)cap;
  std::vector<void *> keep;
  bf16 *hi = nullptr, *lo = nullptr, *ohi = nullptr, *olo = nullptr;
  __half *kv = nullptr;
  float *part = nullptr, *full = nullptr, *ones = nullptr;   // ones: form 2's scales
  int *status = nullptr, rc = CORUN_OK;              // status word | row_blocks
  GemmPairPlan p;
  CUtensorMap tw, tw96;
  auto ok = [&](int r) { return (rc = r) == CORUN_OK; };
  if (ok(dmalloc(keep, &hi, c * K)) && ok(dmalloc(keep, &lo, c * K)) && ok(dmalloc(keep, &status, 2)) &&
      ok(gemm_encode_map(&tw, W, N, K, 128)) && ok(gemm_encode_map(&tw96, W, N, K, 96))) {
    if (form == 0)
      ok(dmalloc(keep, &part, gemm_pair_part_floats(N, K, cap, sms, decode))) && ok(dmalloc(keep, &full, c * N)) &&
          ok(gemm_pair_plan_create(&p, N, K, hi, lo, cap, full, part, sms, decode));
    else if (form == 1)
      ok(dmalloc(keep, &ohi, c * F)) && ok(dmalloc(keep, &olo, c * F)) && ok(gemm_pair_plan_create_swiglu(&p, F, K, hi, lo, cap, ohi, olo, sms, decode));
    else
      ok(dmalloc(keep, &kv, 4 * c * nh * 128)) && ok(dmalloc(keep, &ones, (size_t)2 * nh)) && ok(gemm_pair_plan_create_kv(&p, nh, K, hi, lo, cap, kv, sms));
  }
  if (rc == CORUN_OK) {
    cudaError_t ce = cudaDeviceSynchronize();       // allocations were cleared through the legacy stream
    const int blocks = R > 128 ? 3 : 1;
    if (ce == cudaSuccess && decode) ce = cudaMemcpy(status + 1, &blocks, sizeof(int), cudaMemcpyHostToDevice);
    if (decode) p.row_blocks = status + 1;
    if (ce == cudaSuccess && form == 2) ce = cudaMemcpy(ones, std::vector<float>((size_t)2 * nh, 1.f).data(), (size_t)2 * nh * sizeof(float), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = launch_split(X, R, K, hi, lo, st);
    if (ce == cudaSuccess) ce = gemm_pair_launch(p, tw, decode ? 256 : R, status, st, form == 1 ? &tw96 : nullptr, ones);
    if (ce == cudaSuccess && form == 0) ce = gemm_pair_fixup_launch(p, decode ? 256 : R, st);
    if (ce == cudaSuccess && form == 0) ce = cudaMemcpyAsync(out, full, (size_t)R * N * sizeof(float), cudaMemcpyDeviceToDevice, st);
    if (ce == cudaSuccess && form == 1) ce = launch_join(ohi, olo, false, R, F, out, F, st);
    for (int i = 0; form == 2 && i < 2 * nh && ce == cudaSuccess; ++i) {   // head i / 2: its keys, its values
      const __half *a = kv + ((size_t)(2 * (i & 1)) * nh + i / 2) * c * 128;
      ce = launch_join(a, a + c * nh * 128, true, R, 128, out + i * 128, N, st);
    }
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
    int hs = 0;
    if (ce == cudaSuccess) ce = cudaMemcpy(&hs, status, sizeof(int), cudaMemcpyDeviceToHost);
    if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; rc = CORUN_ECUDA; }
    else if (hs != 0) rc = CORUN_ETIMEOUT;
  }
  for (void *q : keep) cudaFree(q);
  return rc;
}

int corun_debug_gemm_experts(int32_t form, const void *W, int32_t n_experts, int32_t N, int32_t K, const int32_t *rows, const float *X,
                             const float *row_w, float *out, void *cuda_stream) {
  if (form < 0 || form > 1 || !W || n_experts < 1 || n_experts > 256 || N < 128 || N % (form ? 16 : 128) || K < 64 || K % 64 || !rows || !X || !out ||
      (form && !row_w))
    return CORUN_EINVAL;
  if (((uintptr_t)W & 15u) || ((uintptr_t)X & 3u) || ((uintptr_t)out & 3u) || ((uintptr_t)row_w & 3u)) return CORUN_EINVAL;
  std::vector<int> tab;                              // per group: first weight row, first weight k-block, rows
  for (int x = 0; x < n_experts; ++x) {
    if (rows[x] < 0 || rows[x] > PREFILL_BIG) return CORUN_EINVAL;
    for (int r = 0; r < rows[x]; r += 128)
      for (int v : {form ? x * N : 0, form ? 0 : x * (K / GEMM_BLOCK_K), std::min(128, rows[x] - r)}) tab.push_back(v);
  }
  const int used = (int)tab.size() / 3, n_groups = used + 1, F = N / 2;   // (one group more than there are)
  if (!used) return CORUN_EINVAL;
  tab.insert(tab.end(), {0, 0, 0, used});
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int dev = 0, sms = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const size_t slots = (size_t)n_groups * 128;
  std::vector<void *> keep;
  bf16 *hi = nullptr, *lo = nullptr, *ohi = nullptr, *olo = nullptr;
  float *full = nullptr, *w = nullptr;
  int *status = nullptr, *d_tab = nullptr, rc = CORUN_OK;
  GemmExpertsPlan p;
  CUtensorMap tw;
  auto ok = [&](int r) { return (rc = r) == CORUN_OK; };
  if (ok(dmalloc(keep, &hi, slots * K, false)) && ok(dmalloc(keep, &lo, slots * K, false)) && ok(dmalloc(keep, &w, slots, false)) &&
      ok(dmalloc(keep, &d_tab, tab.size(), false)) && ok(dmalloc(keep, &status, 1)) &&
      ok(tma_encode_2d(&tw, W, 0, (unsigned long long)(form ? (long long)n_experts * N : N), form ? K : n_experts * K, GEMM_W_BOX, GEMM_BLOCK_K))) {
    if (form)
      ok(dmalloc(keep, &ohi, slots * F)) && ok(dmalloc(keep, &olo, slots * F)) &&
          ok(gemm_experts_plan_create_swiglu(&p, F, K, hi, lo, n_groups, ohi, olo, w, d_tab, sms));
    else
      ok(dmalloc(keep, &full, slots * N)) && ok(gemm_experts_plan_create(&p, N, K, hi, lo, n_groups, full, d_tab, sms));
  }
  if (rc == CORUN_OK) {
    // what a group has no row for is never more than its own column of a product: NaN here
    cudaError_t ce = cudaMemset(hi, 0xff, slots * K * sizeof(bf16));
    if (ce == cudaSuccess) ce = cudaMemset(lo, 0xff, slots * K * sizeof(bf16));
    if (ce == cudaSuccess) ce = cudaMemset(w, 0xff, slots * sizeof(float));
    if (ce == cudaSuccess) ce = cudaMemcpy(d_tab, tab.data(), tab.size() * sizeof(int), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaDeviceSynchronize();   // (all of it through the legacy stream)
    size_t at = 0;
    for (int g = 0; g < used && ce == cudaSuccess; at += tab[3 * g++ + 2]) {
      const int n = tab[3 * g + 2];
      ce = launch_split(X + at * K, n, K, hi + (size_t)g * 128 * K, lo + (size_t)g * 128 * K, st);
      if (ce == cudaSuccess && form) ce = cudaMemcpyAsync(w + (size_t)g * 128, row_w + at, (size_t)n * sizeof(float), cudaMemcpyDeviceToDevice, st);
    }
    if (ce == cudaSuccess) ce = gemm_experts_launch(p, tw, status, st);
    at = 0;
    for (int g = 0; g < used && ce == cudaSuccess; at += tab[3 * g++ + 2]) {
      const int n = tab[3 * g + 2];
      ce = form ? launch_join(ohi + (size_t)g * 128 * F, olo + (size_t)g * 128 * F, false, n, F, out + at * F, F, st)
                : cudaMemcpyAsync(out + at * N, full + (size_t)g * 128 * N, (size_t)n * N * sizeof(float), cudaMemcpyDeviceToDevice, st);
    }
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
    int hs = 0;
    if (ce == cudaSuccess) ce = cudaMemcpy(&hs, status, sizeof(int), cudaMemcpyDeviceToHost);
    if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; rc = CORUN_ECUDA; }
    else if (hs != 0) rc = CORUN_ETIMEOUT;
  }
  for (void *q : keep) cudaFree(q);
  return rc;
}

int corun_debug_prefill_attention(corun_engine *e, int32_t slot, int32_t layer, int32_t pos0, int32_t n, const float *q, float *out) {
  if (!e || !q || !out || pos0 < 0 || n < 1 || layer < 0 || layer >= e->sh.n_layers) return CORUN_EINVAL;
  if (!slot_ok(e, slot) || !e->in_use[slot]) return CORUN_ESLOT;
  Program &P = e->big;
  if (!P.pair || n > P.cap || pos0 + n > e->ctx[slot] || (e->mla && !P.mla_tiles)) return CORUN_EINVAL;
  RC(sync_stream(e));
  const corun_shape &s = e->sh;
  const MlaDims &md = e->md;
  std::vector<int> rows((size_t)4 * n, 0);           // token | position | active | slot
  for (int i = 0; i < n; ++i) { rows[(size_t)n + i] = pos0 + i; rows[(size_t)2 * n + i] = 1; rows[(size_t)3 * n + i] = slot; }
  P.R = n;
  P.row_pos = P.row_token + n;
  P.row_active = P.row_pos + n;
  P.row_slot = P.row_active + n;
  const Rows r{P.row_token, P.row_pos, P.row_active, P.row_slot, n};
  cudaError_t ce = cudaMemcpyAsync(P.row_token, rows.data(), rows.size() * sizeof(int), cudaMemcpyHostToDevice, e->st);
  const int width = e->mla ? md.nh * md.vh : s.n_q_heads * s.head_dim;
  float *tmp = nullptr;
  if (cudaMalloc(&tmp, (size_t)n * (e->mla ? md.nh * (md.nope + md.rope) : width) * sizeof(float)) != cudaSuccess) return CORUN_ENOMEM;
  std::vector<float> part;
  if (!e->mla) {
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(P.q, q, (size_t)n * width * sizeof(float), cudaMemcpyHostToDevice, e->st);
    if (ce == cudaSuccess) ce = launch_attention_prefill(e->tm_k4[layer], P.q, r, s.n_q_heads, kv_layout(e), P.ao_hi, P.ao_lo, e->d_status, e->st);
  } else {
    const int qw = md.nope + md.rope, rph = (n + 63) / 64 * 64;
    P.RPH = rph;
    part.resize((size_t)n * qw);
    for (int h = 0; h < md.nh && ce == cudaSuccess; ++h) {           // a head's no-rope parts, head-major
      for (int i = 0; i < n; ++i) memcpy(&part[(size_t)i * md.nope], q + ((size_t)i * md.nh + h) * qw, md.nope * sizeof(float));
      const size_t at = (size_t)h * rph * md.nope;
      ce = cudaMemcpyAsync(tmp, part.data(), (size_t)n * md.nope * sizeof(float), cudaMemcpyHostToDevice, e->st);
      if (ce == cudaSuccess) ce = launch_split(tmp, n, md.nope, P.qn_hi + at, P.qn_lo + at, e->st);
      if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->st);
    }
    part.resize((size_t)n * md.nh * md.rope);
    for (int i = 0; i < n * md.nh; ++i) memcpy(&part[(size_t)i * md.rope], q + (size_t)i * qw + md.nope, md.rope * sizeof(float));
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(P.q_rope, part.data(), part.size() * sizeof(float), cudaMemcpyHostToDevice, e->st);
    if (ce == cudaSuccess) ce = cudaMemsetAsync(P.tile_base, 0, (size_t)(P.cap / 128) * sizeof(int), e->st);
    P.segs.n = 1;
    P.segs.slot[0] = slot;
    P.segs.off[0] = 0;
    P.segs.len[0] = pos0 + n;
    P.kv_tokens = (pos0 + n + 63) / 64 * 64;
    if (ce == cudaSuccess) ce = run_mla_tiles(e, P, layer, r);
  }
  if (ce == cudaSuccess) ce = launch_join(P.ao_hi, P.ao_lo, false, n, width, tmp, width, e->st);
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(out, tmp, (size_t)n * width * sizeof(float), cudaMemcpyDeviceToHost, e->st);
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(e->h_status, e->d_status, sizeof(int), cudaMemcpyDeviceToHost, e->st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->st);
  cudaFree(tmp);
  if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; return CORUN_ECUDA; }
  return check_status(e);
}

int corun_debug_variate(uint64_t seed, uint64_t t, uint32_t *out_u24) {
  if (!out_u24) return CORUN_EINVAL;
  uint32_t *d = nullptr;
  if (cudaMalloc(&d, sizeof(uint32_t)) != cudaSuccess) return CORUN_ENOMEM;
  cudaError_t ce = launch_variate(seed, t, d, nullptr);
  if (ce == cudaSuccess) ce = cudaMemcpy(out_u24, d, sizeof(uint32_t), cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; return CORUN_ECUDA; }
  return CORUN_OK;
}

int corun_debug_sample(const float *logits, int32_t n_rows, int32_t vocab, const corun_sampling *sampling,
                       const uint32_t *u24, int32_t *out_tokens) {
  if (!logits || !sampling || !u24 || !out_tokens || n_rows < 1 || vocab < 1) return CORUN_EINVAL;
  std::vector<void *> keep;
  float *dl = nullptr, *dt = nullptr, *dp = nullptr;
  int *dflag = nullptr, *dstep = nullptr, *dtok = nullptr;
  uint32_t *du = nullptr;
  uint64_t *dseed = nullptr;
  int rc;
  if ((rc = dmalloc(keep, &dl, (size_t)n_rows * vocab, false)) == 0 && (rc = dmalloc(keep, &dt, n_rows)) == 0 &&
      (rc = dmalloc(keep, &dp, n_rows)) == 0 && (rc = dmalloc(keep, &dflag, n_rows)) == 0 &&
      (rc = dmalloc(keep, &dstep, n_rows)) == 0 && (rc = dmalloc(keep, &dtok, n_rows)) == 0 &&
      (rc = dmalloc(keep, &du, n_rows)) == 0 && (rc = dmalloc(keep, &dseed, n_rows)) == 0) {
    std::vector<float> t(n_rows, sampling->temperature), p(n_rows, sampling->top_p);
    std::vector<int> ones(n_rows, 1);
    cudaError_t ce = cudaMemcpy(dl, logits, (size_t)n_rows * vocab * sizeof(float), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMemcpy(dt, t.data(), n_rows * sizeof(float), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMemcpy(dp, p.data(), n_rows * sizeof(float), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMemcpy(dflag, ones.data(), n_rows * sizeof(int), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMemcpy(du, u24, n_rows * sizeof(uint32_t), cudaMemcpyHostToDevice);
    SampleArgs sa{dl, vocab, dflag, dt, dp, dseed, dstep, du, dtok};
    if (ce == cudaSuccess) ce = launch_sampler(sa, n_rows, nullptr);
    if (ce == cudaSuccess) ce = cudaMemcpy(out_tokens, dtok, n_rows * sizeof(int), cudaMemcpyDeviceToHost);
    if (ce != cudaSuccess) { g_last_cuda_error = (int)ce; rc = CORUN_ECUDA; }
  }
  for (void *q : keep) cudaFree(q);
  return rc;
}

}  // extern "C"
