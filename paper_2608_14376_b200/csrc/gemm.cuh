// GEMMs of decode steps and prefill chunks  out[r, n] = sum_k W[n, k] * (Xhi[r, k] + Xlo[r, k]).
//
// Up to GEMM_MAX_ROWS padded rows (gemm_rows.cu) a tile of 128 or 256 weight rows is the M operand of the MMAs and the rows there are
// (hi, then lo) the N operand; above (gemm.cu) blocks of 128 rows are the M operand and a tile of 256 weight rows the N operand;
// prompts and decode steps of many slots run on pairs of SMs (gemm_pair.cu, gemm_experts.cu, below).
//
// The flat space of (weight tile, 64-wide k-block) pairs is cut into one contiguous range per CTA.  The cut depends on the shape
// (N, K), on the padded rows by way of the tile's width, and on the SM count, never on which rows are occupied.  A tile
// whose k-blocks all belong to one CTA is written straight to `direct`;
// otherwise each CTA writes a partial to its workspace slot and the consumer
// adds the partials in ascending CTA order (gemm_load).  No atomics anywhere.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace corun {

// Last CUDA runtime error (cudaError_t), or 100000 + CUresult for driver calls.
extern int g_last_cuda_error;

constexpr int GEMM_TILE_N = 256;   // weight rows per tile (up to GEMM_NARROW_ROWS padded rows: or half)
constexpr int GEMM_ROW_BLOCK = 128; // (above GEMM_MAX_ROWS) activation rows per MMA (the MMA's M)
constexpr int GEMM_BLOCK_K = 64;   // bf16 elements per k-block (= one 128-byte swizzle row)
constexpr int GEMM_MAX_SELECT = 288;  // experts of a selected-experts GEMM
constexpr int GEMM_W_BOX = 128;    // weight rows per TMA box
constexpr int GEMM_MAX_ROWS = 128; // padded rows up to which gemm_rows.cu has the kernel
constexpr int GEMM_NARROW_ROWS = 32;  // padded rows up to which a tile may be 128 weight rows
constexpr int GEMM_ROWS_MAX_SMEM = 224 * 1024;
constexpr int GEMM_THREADS = 192;  // (above GEMM_MAX_ROWS) warp 0 TMA producer, warp 1 MMA issuer, warps 2-5 epilogue

// What a consumer kernel needs to read a GEMM result.
struct GemmOut {
  const float *direct;   // [rows, N]; valid for tiles owned by one CTA
  const float *ws;       // [(cta*2 + slot), BN, 1 << tile_shift] partials
  const int *tile_first; // [n_tiles] 2 * (first CTA touching the tile) + (the slot that CTA used for it)
  const int *tile_cend;  // [n_tiles] last CTA touching the tile (every later CTA used slot 0)
  int N, KB, BN;
  // Result of gemm_pair.cu (row_tiles > 0): tiles [256 rows x 256 columns], row tiles fastest; the first `whole` are in
  // `direct`, the others in `ws`, tile after tile as `slices` partial tiles [256][256].
  int row_tiles, whole, slices;
  int tile_shift = 8;    // log2 of the tile's columns
};

// Values of a gemm_pair.cu result, the slices added in ascending order.
__device__ __forceinline__ const float *gemm_pair_at(const GemmOut &g, int tile, int r, int n) {
  return g.ws + ((size_t)(tile - g.whole) * g.slices * 256 + (r & 255)) * GEMM_TILE_N + n % GEMM_TILE_N;
}
__device__ __forceinline__ float gemm_load_pair(const GemmOut &g, int r, int n) {
  const int tile = (n / GEMM_TILE_N) * g.row_tiles + r / 256;
  if (tile < g.whole) return g.direct[(size_t)r * g.N + n];
  const float *p = gemm_pair_at(g, tile, r, n);
  float acc = p[0];
  for (int s = 1; s < g.slices; ++s) acc += p[(size_t)s * 256 * GEMM_TILE_N];
  return acc;
}
__device__ __forceinline__ float4 gemm_load_pair4(const GemmOut &g, int r, int n) {
  const int tile = (n / GEMM_TILE_N) * g.row_tiles + r / 256;
  if (tile < g.whole) return *reinterpret_cast<const float4 *>(g.direct + (size_t)r * g.N + n);
  const float *p = gemm_pair_at(g, tile, r, n);
  float4 v[8];                                      // at most eight slices, all requested together
#pragma unroll
  for (int s = 0; s < 8; ++s)
    if (s < g.slices) v[s] = *reinterpret_cast<const float4 *>(p + (size_t)s * 256 * GEMM_TILE_N);
  float4 acc = v[0];
#pragma unroll
  for (int s = 1; s < 8; ++s)
    if (s < g.slices) { acc.x += v[s].x; acc.y += v[s].y; acc.z += v[s].z; acc.w += v[s].w; }
  return acc;
}

// Values (r, n) and (r, n2) of a GEMM result as gemm_load gives them, both sets of partials requested together.
__device__ __forceinline__ float2 gemm_load_two(const GemmOut &g, int r, int n, int n2) {
  const int t[2] = {n >> g.tile_shift, n2 >> g.tile_shift}, col[2] = {n - (t[0] << g.tile_shift), n2 - (t[1] << g.tile_shift)};
  const int f[2] = {g.tile_first[t[0]], g.tile_first[t[1]]}, c1[2] = {g.tile_cend[t[0]], g.tile_cend[t[1]]};
  const size_t cta_stride = (size_t)2 * g.BN << g.tile_shift;
  float v[2][4], acc[2];
  const float *p[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int c0 = f[i] >> 1;
    p[i] = g.ws + ((size_t)r << g.tile_shift) + col[i];
    acc[i] = c0 == c1[i] ? g.direct[(size_t)r * g.N + (i ? n2 : n)] : p[i][(size_t)f[i] * g.BN << g.tile_shift];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] = c0 + 1 + j <= c1[i] ? p[i][(size_t)(c0 + 1 + j) * cta_stride] : 0.f;
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    acc[i] += 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i] += v[i][j];
    for (int c = (f[i] >> 1) + 5; c <= c1[i]; ++c) acc[i] += p[i][(size_t)c * cta_stride];
  }
  return make_float2(acc[0], acc[1]);
}

// Value (r, n) of a GEMM result, partials added in ascending CTA order.
__device__ __forceinline__ float gemm_load(const GemmOut &g, int r, int n) {
  const int t = n >> g.tile_shift, col = n - (t << g.tile_shift);
  const int f = g.tile_first[t], c0 = f >> 1, c1 = g.tile_cend[t];
  if (c0 == c1) return g.direct[(size_t)r * g.N + n];
  const float *p = g.ws + ((size_t)r << g.tile_shift) + col;
  const size_t cta_stride = (size_t)2 * g.BN << g.tile_shift;
  float acc = 0.f;
  acc += p[(size_t)f * g.BN << g.tile_shift];
  for (int c = c0 + 1; c <= c1; ++c) acc += p[(size_t)c * cta_stride];
  return acc;
}

// Four consecutive values (n % 4 == 0, N % 4 == 0) with the same summation order as gemm_load.
// Loads are issued four partials at a time; an absent partial contributes +0.0f.
__device__ __forceinline__ float4 gemm_load4(const GemmOut &g, int r, int n) {
  if (g.row_tiles) return gemm_load_pair4(g, r, n);
  const int t = n >> g.tile_shift, col = n - (t << g.tile_shift);
  const int f = g.tile_first[t], c0 = f >> 1, c1 = g.tile_cend[t];
  if (c0 == c1) return *reinterpret_cast<const float4 *>(g.direct + (size_t)r * g.N + n);
  const float *p = g.ws + ((size_t)r << g.tile_shift) + col;
  const size_t cta_stride = (size_t)2 * g.BN << g.tile_shift;
  float4 acc = *reinterpret_cast<const float4 *>(p + ((size_t)f * g.BN << g.tile_shift));
  acc.x += 0.f; acc.y += 0.f; acc.z += 0.f; acc.w += 0.f;   // same rounding path as 0 + first partial
  for (int c = c0 + 1; c <= c1; c += 4) {
    float4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      v[j] = (c + j <= c1) ? *reinterpret_cast<const float4 *>(p + (size_t)(c + j) * cta_stride)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc.x += v[j].x; acc.y += v[j].y; acc.z += v[j].z; acc.w += v[j].w;
    }
  }
  return acc;
}

// Tensor maps of the split activations: boxes of 64, 32 and 16 rows (above GEMM_MAX_ROWS: of 128 rows, the first of each).
struct GemmXMaps {
  CUtensorMap hi[3], lo[3];
};

// Static launch description of one GEMM shape (built once at init).
struct GemmPlan {
  CUtensorMap tmW;
  GemmXMaps tmX;
  int N = 0, K = 0, R = 0, BN = 0;   // weight rows, reduction length, real rows, padded rows
  int tile_n = GEMM_TILE_N;          // weight rows per tile (without SwiGLU)
  int n_tiles = 0, KB = 0, grid = 0, stages = 0;
  uint32_t idesc = 0, stage_bytes = 0;
  size_t smem_bytes = 0;
  float *direct = nullptr;           // not owned
  float *ws = nullptr;               // not owned
  int *d_cta_start = nullptr, *d_tile_first = nullptr, *d_tile_cend = nullptr;  // owned (one allocation)
  int *d_split_tiles = nullptr;      // tiles with partials (same allocation)
  int n_split_tiles = 0;
  // Optional store mask (device, not owned): row r of weight tile t is stored only if
  // row_keep[r * keep_pitch + t / keep_div] != 0 (rows that no consumer will read are skipped).
  const float *row_keep = nullptr;
  int keep_pitch = 0, keep_div = 1;
  // Grouped mode (gemm_plan_create_grouped): the CTAs take the (group, weight tile) pairs in turn; see gemm_rows.cu.
  const int *group_tab = nullptr;    // device, not owned: per group (first weight row, first weight k-block, rows),
                                     // then ONE more int: the number of groups in use (the first ones);
                                     // keep_div = -1 tells the kernel that no kernel of the same stream writes it
  int tiles_per_group = 0;
  bool select = false;               // gemm_plan_create_select_*: group_tab holds the rows' experts, keep_div ints
  // Gate / up GEMM with SwiGLU in the epilogue (gemm_plan_create_swiglu): the bf16 hi/lo output [BN, N / 2].
  __nv_bfloat16 *sw_hi = nullptr, *sw_lo = nullptr;
  int sw_half = 0;                   // gate rows (= up rows) per tile
  // Device int, not owned, written by an earlier kernel of the step (null: all rows): how many rows hold a request this step
  // (they are the first ones) at bits 8 .., and bit b set = block b of 128 rows (up to 128 padded rows: of 64) holds one.  Rows
  // behind the padded count, or blocks without a request, are neither loaded nor multiplied nor stored.
  const int *row_blocks = nullptr;
  GemmOut out() const {
    GemmOut g{direct, ws, d_tile_first, d_tile_cend, N, KB, BN, 0, 0, 0};
    g.tile_shift = tile_n == GEMM_TILE_N ? 8 : 7;
    return g;
  }
};

// The value of *row_blocks for n rows with a request, in blocks of `block` rows.
__host__ __device__ inline int gemm_row_blocks(int n, int block) { return (n > 0 ? 1 : 0) | (n > block ? 2 : 0) | n << 8; }

// Workspace floats needed by any plan with this grid and BN.
inline size_t gemm_ws_floats(int grid, int BN) { return (size_t)grid * 2 * BN * GEMM_TILE_N; }

// Builds the plan: tensor maps for W [N, K] bf16 and the split activations
// Xhi / Xlo [BN, K] bf16 (row pitch K), the CTA partition and its tables.
// Returns 0 or a negative corun_status.
int gemm_plan_create(GemmPlan *p, const void *W, int N, int K, const void *Xhi, const void *Xlo, int R, int BN,
                     float *direct, float *ws, int num_sms);
void gemm_plan_destroy(GemmPlan *p);
// Grouped GEMM over at most n_groups groups of up to BN <= 128 rows each: group g multiplies rows g * BN .. of
// Xhi / Xlo ([n_groups * BN, K]) with N weight rows starting at the row, and K elements starting at the k-block,
// that group_tab names for it, into rows g * BN .. of `direct` ([n_groups * BN, N]).  W is [w_rows, w_cols]
// bf16.  group_tab has 3 * n_groups + 1 ints: the last one is the number of groups in use (groups 0 .. that - 1).
// At most num_sms CTAs take the (group, tile of 256 weight rows) pairs of the groups in use in turn, all k-blocks
// of a tile: no partials.  N % 256 == 0.
int gemm_plan_create_grouped(GemmPlan *p, const void *W, long long w_rows, int w_cols, int N, int K, const void *Xhi,
                             const void *Xlo, int n_groups, int BN, float *direct, const int *group_tab, int num_sms);
// The same for gate / up matrices ([2F, K] per group: F gate rows, then F up rows, from the group's first weight row)
// with the SwiGLU in the epilogue: row_scale[g * BN + r] * silu(gate) * up as a bf16 hi/lo pair [n_groups * BN, F].
// Tiles of `half` gate rows and the `half` up rows of the same outputs (F % half == 0, 64 <= half <= 128).
int gemm_plan_create_grouped_swiglu(GemmPlan *p, const void *W, long long w_rows, int F, int K, int half, const void *Xhi,
                                    const void *Xlo, int n_groups, int BN, __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo,
                                    const float *row_scale, const int *group_tab, int num_sms);
// The experts of a Mixture-of-Experts layer for up to BN <= 64 rows, all rows of the step together per expert: only the
// experts that a row selected are loaded and multiplied.  sel: n_sel ints, every row's experts (< 0: none); w: the routing
// weights [R][NB].  up: W [NB * 2F, K] -> out_hi / out_lo [NB * BN, F], row e * BN + r = w[r, e] * silu(gate) * up (tiles
// of `half` gate rows as above).  down: W [N, NB * F] -> direct [NB * BN, N], row e * BN + r.  Rows that did not select
// the expert keep what they held.
int gemm_plan_create_select_up(GemmPlan *p, const void *W, int NB, int F, int K, int half, const void *Xhi, const void *Xlo, int R, int BN,
                               __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, const float *w, const int *sel, int n_sel, int num_sms);
int gemm_plan_create_select_down(GemmPlan *p, const void *W, int NB, int N, int F, const void *Xhi, const void *Xlo, int R, int BN,
                                 float *direct, const float *w, const int *sel, int n_sel, int num_sms);
// Gate / up GEMM with the SwiGLU in its epilogue (BN <= GEMM_MAX_ROWS): W is [2F, K] (F gate rows, then F up rows; F % 8 == 0);
// out_hi / out_lo [BN, F] receive silu(gate) * up of rows 0 .. R-1 as a bf16 hi/lo pair.  A tile is
// gemm_swiglu_half(F, num_sms) gate rows with the up rows of the same outputs, and every CTA owns whole tiles
// (one each when the SMs allow), so there are no partials; a tensor map that overrides the plan's at launch
// must have a box of that many rows (gemm_encode_map(.., box_rows = gemm_swiglu_half(..))).
int gemm_swiglu_half(int F, int num_sms);
int gemm_plan_create_swiglu(GemmPlan *p, const void *W, int F, int K, const void *Xhi, const void *Xlo, int R, int BN,
                            __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, int num_sms);
// The same for a stack of n_blocks gate / up matrices (the experts of a Mixture-of-Experts layer): W is
// [n_blocks * 2 * Fb, K], block e = Fb gate rows then Fb up rows; out_hi / out_lo [BN, n_blocks * Fb] receive
// row_scale[r * n_blocks + e] * silu(gate) * up in columns e * Fb .., exact zeros where the scale is zero (the
// row did not select the expert).  A tile is gemm_swiglu_blocks_half(Fb, n_blocks, num_sms) gate rows of one
// block with their up rows (0: no multiple of 8 in 64..128 divides Fb); whole tiles, no partials.
int gemm_swiglu_blocks_half(int Fb, int n_blocks, int num_sms);
int gemm_plan_create_swiglu_blocks(GemmPlan *p, const void *W, int n_blocks, int Fb, int K, const void *Xhi, const void *Xlo,
                                   int R, int BN, __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, const float *row_scale,
                                   int num_sms);
// The allocation-free half of gemm_plan_create: fills every host-side field and tensor map of the
// plan and writes the partition tables (cta_start, tile_first, tile_cend, split_tiles) to `tab`
// (capacity tab_cap ints; *tab_ints = ints used).  gemm_plan_bind_tables points the plan at a device
// copy of those tables.
int gemm_plan_fill(GemmPlan *p, const void *W, int N, int K, const void *Xhi, const void *Xlo, int R, int BN,
                   float *direct, float *ws, int num_sms, int *tab, int tab_cap, int *tab_ints);
void gemm_plan_bind_tables(GemmPlan *p, int *d_tab);
// Enqueues the GEMM.  `W` may override the weight matrix of the plan (same
// shape) by passing a different tensor map.
cudaError_t gemm_launch(const GemmPlan &p, const CUtensorMap *tmW_override, int *d_status, cudaStream_t st,
                        unsigned long long *trace = nullptr,   // optional [grid][8] globaltimer stamps (debug)
                        bool pdl = false);                     // programmatic dependent launch (row program)
// Encodes a tensor map for a bf16 [rows, K] row-major matrix with a [box_rows, 64] box, 128-byte swizzle.
int gemm_encode_map(CUtensorMap *m, const void *base, int rows, int K, int box_rows);
// Padded rows of a launch (a group) with n <= 128 rows: boxes of 64, 32 and 16 rows, two at most.
__host__ __device__ constexpr int gemm_rows_padded(int n) {
  return n > 96 ? 128 : n > 80 ? 96 : n > 64 ? 80 : n > 48 ? 64 : n > 32 ? 48 : n > 16 ? 32 : 16;
}
// Opts the GEMM kernel into its dynamic shared-memory size (idempotent, allocates nothing).
cudaError_t gemm_prepare_kernel();
// gemm_rows.cu: sets a plan's ring; the activations' maps; the launch.
int gemm_rows_stages(GemmPlan *p);
int gemm_encode_x(GemmXMaps *m, const void *Xhi, const void *Xlo, unsigned long long rows, int K);
cudaError_t gemm_rows_prepare();
cudaError_t gemm_rows_launch(const GemmPlan &p, const CUtensorMap *tmW_override, int *d_status, cudaStream_t st, unsigned long long *trace, bool pdl);
// Tensor map for a 16-bit [rows, cols] row-major matrix with a [box_rows, box_cols] box: 64 columns
// (128 bytes, 128-byte swizzle) or 16 columns (32 bytes, 32-byte swizzle).
int tma_encode_2d(CUtensorMap *m, const void *base, int is_fp16, unsigned long long rows, int cols, int box_rows,
                  int box_cols);
// Tensor map over fp16 data seen as a 4-dimensional array: dims[0] elements are contiguous, strides[i] is the byte
// distance between consecutive indices of dimension i + 1 (a multiple of 16; they need not ascend); the box's
// innermost extent is 64 elements (128 bytes, 128-byte swizzle).  The box lands in shared memory densely,
// dimension 0 fastest.
int tma_encode_fp16_4d(CUtensorMap *m, const void *base, const unsigned long long dims[4], const unsigned long long strides[3],
                       const unsigned box[4]);
// The same with 2 to 5 dimensions (dims / box: nd values, strides: nd - 1 byte strides of dimensions 1 ..).
int tma_encode_fp16_nd(CUtensorMap *m, const void *base, int nd, const unsigned long long *dims, const unsigned long long *strides,
                       const unsigned *box);
// ---- many rows (gemm_pair.cu): tiles of 256 rows x 256 weight rows, one per pair of SMs; K in up to 8 slices, and the tiles of
// an unfilled wave are left as partial matrices, a slice each: `out` alone is not the result (gemm_pair_out) ----
struct GemmPairPlan {
  CUtensorMap tmHi, tmLo, tmOut, tmOut2;
  int N = 0, K = 0, cap = 0, pairs = 0, n_tiles = 0;   // weight rows, reduction length, rows the buffers hold
  int slices = 1, per_unit = 1;      // cuts of K, a function of the matrix and the GPU, never of the rows; slices per unit of work
  bool swiglu = false;
  int kv_heads = 0;                  // gemm_pair_plan_create_kv
  float *out = nullptr, *part = nullptr;   // not owned
  bool decode = false;               // rows of a decode step (cap 256), in two halves that may be without a request
  const int *row_blocks = nullptr;   // (decode) device, not owned: bit 1 = rows 128 .. hold a request
};
// Floats of partial tiles that launches over up to cap rows leave (the next kernel of the stream consumes them, so one
// buffer serves all plans of a program).
size_t gemm_pair_part_floats(int N, int K, int cap, int num_sms, bool decode = false);
// X W^T for activations Xhi / Xlo [cap, K] (N % 8 == 0) -> out [cap, N] fp32 and, for the tiles of an unfilled wave, part
// (gemm_pair_part_floats).  Read through gemm_pair_out(p, R, zeros).
int gemm_pair_plan_create(GemmPairPlan *p, int N, int K, const void *Xhi, const void *Xlo, int cap, float *out, float *part, int num_sms,
                          bool decode = false);
GemmOut gemm_pair_out(const GemmPairPlan &p, int R, const int *zero_tiles);
int gemm_pair_ctas(const GemmPairPlan &p, int R, bool narrow);   // CTAs of a launch (narrow: with a map of 96 rows)
int gemm_pair_has_parts(const GemmPairPlan &p, int R);   // 1 if some of the result of R rows is left in partial matrices
cudaError_t gemm_pair_fixup_launch(const GemmPairPlan &p, int R, cudaStream_t st);   // makes `out` a plain matrix
// W is [2F, K] (F gate rows, then F up rows; F % 8 == 0): out_hi / out_lo [cap, F] = silu(gate) * up as a bf16 hi/lo pair.
int gemm_pair_plan_create_swiglu(GemmPairPlan *p, int F, int K, const void *Xhi, const void *Xlo, int cap, __nv_bfloat16 *out_hi,
                                 __nv_bfloat16 *out_lo, int num_sms, bool decode = false);
// Decompression of latents into keys and values: W is [nh * 256, K] (per head 128 key rows, 128 value rows); the fp16 hi / lo
// pairs of the products, times the launch's kv_scale [nh][2] (keys, values; device), go to kv [key hi | key lo | value hi | value
// lo][nh][cap][128] (cap % 32 == 0).
int gemm_pair_plan_create_kv(GemmPairPlan *p, int nh, int K, const void *Xhi, const void *Xlo, int cap, void *kv, int num_sms);
int gemm_pair_prepare();             // opts the kernels into their shared-memory size (idempotent)
// Rows 0 .. R-1 (R <= cap).  tmW: the weight matrix with a box of 128 rows (gemm_encode_map(.., 128)); tmW96 (swiglu): the
// same with 96 rows, taken where it shortens the waves.
cudaError_t gemm_pair_launch(const GemmPairPlan &p, const CUtensorMap &tmW, int R, int *d_status, cudaStream_t st,
                             const CUtensorMap *tmW96 = nullptr, const float *kv_scale = nullptr,
                             unsigned long long *trace = nullptr);   // (debug) timeline, as gemm_launch's; 2 * pairs CTAs at most
// ---- the experts of a prompt (gemm_experts.cu): groups of up to 128 rows on pairs of SMs; groups and results as
// gemm_plan_create_grouped / _swiglu with BN = 128.  tmW: the matrix with a box of GEMM_W_BOX rows ----
struct GemmExpertsPlan {
  GemmXMaps tmX;
  int N = 0, K = 0, tiles_per_group = 0, n_groups_max = 0, pairs = 0;
  const int *group_tab = nullptr;    // not owned, as are the others
  const float *row_w = nullptr;
  float *direct = nullptr;
  __nv_bfloat16 *sw_hi = nullptr, *sw_lo = nullptr;
};
int gemm_experts_plan_create(GemmExpertsPlan *p, int N, int K, const void *Xhi, const void *Xlo, int n_groups, float *direct, const int *group_tab,
                             int num_sms);
int gemm_experts_plan_create_swiglu(GemmExpertsPlan *p, int F, int K, const void *Xhi, const void *Xlo, int n_groups, __nv_bfloat16 *out_hi,
                                    __nv_bfloat16 *out_lo, const float *row_w, const int *group_tab, int num_sms);
cudaError_t gemm_experts_launch(const GemmExpertsPlan &p, const CUtensorMap &tmW, int *d_status, cudaStream_t st);
// Tensor map for TMA stores of tiles of 32 rows x 32 columns into a [rows, cols] row-major matrix (fp32: 128-byte swizzle; bf16: 64).
int tma_encode_store_2d(CUtensorMap *m, const void *base, int is_fp32, unsigned long long rows, int cols);
// direct[r, n] = gemm_load(r, n) for every tile that has partials (makes `direct` a plain matrix).
cudaError_t gemm_fixup_launch(const GemmPlan &p, cudaStream_t st, bool pdl = false, int rows = 0);   // rows: the first ones (0: p.R)
// *q = p (gemm_plan_create or gemm_plan_create_swiglu, up to GEMM_MAX_ROWS padded rows) over other rows: activations, outputs and
// row_blocks of its own, the tables shared with p (only p is destroyed).
int gemm_plan_rebase(GemmPlan *q, const GemmPlan &p, const void *Xhi, const void *Xlo, float *direct, __nv_bfloat16 *sw_hi,
                     __nv_bfloat16 *sw_lo, const int *row_blocks);

}  // namespace corun
