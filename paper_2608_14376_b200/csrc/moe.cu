// Mixture-of-Experts feed-forward block without groups: two plain decode GEMMs over all experts with a
// masked, probability-weighted SwiGLU between them (see include/corun_moe.h for the formulation and why
// it is position-invariant).  The kernels here are the router's softmax / top-k, the masked SwiGLU and
// the read-out of the second GEMM; the GEMMs are gemm.cu's.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <new>
#include <vector>

#include "../../include/corun_moe.h"
#include "gemm.cuh"
#include "launch.cuh"
#include "moe.cuh"
#include "ops.cuh"
#include "ptx.cuh"

using namespace corun;

namespace {

using bf16 = __nv_bfloat16;
constexpr int MOE_MAX_TOPK = 16;
constexpr int ROUTER_WARPS = 8;
constexpr int MOE_MAX_EXPERTS = 256;

#define MCK(call)                               \
  do {                                          \
    cudaError_t ce_ = (call);                   \
    if (ce_ != cudaSuccess) {                   \
      g_last_cuda_error = (int)ce_;             \
      return CORUN_ECUDA;                       \
    }                                           \
  } while (0)

__device__ __forceinline__ void moe_split(float x, bf16 &hi, bf16 &lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// One warp routes one row: softmax over the E router logits (load(e) gives logit e), then top_k by repeated arg-max
// with ties to the lower id.  Lane l holds experts l, l + 32, ...; the sum of the exponentials is each lane's
// experts in ascending id, then a fixed butterfly over the lanes.  Writes the routing and the row of SwiGLU weights
// w[r, 0 .. E + S): p_e for the selected experts, 0 for the others, 1 for the shared ones.
template <typename LoadLogit>
__device__ __forceinline__ void moe_route_row(LoadLogit load, int r, int lane, int E, int S, int top_k, int renormalize,
                                              float *__restrict__ w, int *__restrict__ experts, float *__restrict__ probs,
                                              int *__restrict__ sel = nullptr, bool on = true) {
  constexpr int PER = MOE_MAX_EXPERTS / 32;
  float z[PER];
  float mx = -CUDART_INF_F;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int e = lane + 32 * j;
    z[j] = e < E ? load(e) : -CUDART_INF_F;
    mx = fmaxf(mx, z[j]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  float sum = 0.f;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int e = lane + 32 * j;
    z[j] = e < E ? expf(z[j] - mx) : -1.f;           // -1: not an expert
    if (e < E) sum += z[j];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  float *wr = w + (size_t)r * (E + S);
  for (int e = lane; e < E; e += 32) wr[e] = 0.f;
  for (int s = lane; s < S; s += 32) wr[E + s] = 1.f;
  __syncwarp();
  int id = 0;                                        // lane k: the k-th selected expert and its probability
  float prob = 0.f, picked = 0.f;                    // picked: sum of the selected probabilities, in selection order
  for (int k = 0; k < top_k; ++k) {
    float bz = -1.f;                                 // this lane's best: largest value, lowest id on ties
    int be = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if (z[j] > bz) { bz = z[j]; be = lane + 32 * j; }
    // the warp's: values are -1 or not below 0, and those order as their bits do
    const int top = __reduce_max_sync(0xffffffffu, __float_as_int(bz));
    be = __reduce_min_sync(0xffffffffu, __float_as_int(bz) == top ? be : 0x7fffffff);
    if (be >= E) be = k;                             // a row of NaNs: any valid id
    const float p = __fdiv_rn(__int_as_float(top), sum);
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if (lane + 32 * j == be) z[j] = -2.f;          // taken
    if (lane == k) { id = be; prob = p; }
    picked += p;
  }
  if (lane < top_k) {
    const float p = renormalize ? __fdiv_rn(prob, picked) : prob;
    wr[id] = p;
    if (experts) experts[(size_t)r * top_k + lane] = id;
    if (probs) probs[(size_t)r * top_k + lane] = p;
  }
  if (sel) {                                         // ascending ids, the shared experts last
    int *out = sel + (size_t)r * (top_k + S);
    int place = 0;
    for (int j = 0; j < top_k; ++j) {
      const int other = __shfl_sync(0xffffffffu, id, j);
      place += other < id || (other == id && j < lane) ? 1 : 0;   // (a row of NaNs may pick an id twice)
    }
    // a probability that has vanished is no selection: the GEMMs neither compute nor store the row for that expert
    if (lane < top_k) out[place] = on && wr[id] != 0.f ? id : -1;
    for (int s = lane; s < S; s += 32) out[top_k + s] = on ? E + s : -1;
  }
}

// Router: logits = Wr x on the CUDA cores (E dot products of H terms a row: far too little for a tensor-core launch of its
// own), then the routing above.  blockIdx.y: NR rows, as their bf16 hi + lo pairs (exactly what the GEMMs of the block
// see); blockIdx.x: ROUTER_WARPS experts, one per warp.  A lane adds its terms in ascending order (8 consecutive terms per
// step, the weights of eight steps requested together, the first ones ahead of the wait for the predecessor), then a fixed
// butterfly over the lanes: a row's routing depends on the row alone.  The CTA that finishes its rows last routes them.
template <int NR>
__global__ void __launch_bounds__(32 * ROUTER_WARPS) moe_router_kernel(const bf16 *__restrict__ x_hi, const bf16 *__restrict__ x_lo, int H,
                                                                       const bf16 *__restrict__ Wr, int R, int E, int S, int top_k,
                                                                       int renormalize, float *__restrict__ w,
                                                                       int *__restrict__ experts, float *__restrict__ probs,
                                                                       const int *active, int *__restrict__ sel, RouterScratch rs) {
  griddep_launch_dependents();
  extern __shared__ float xs[];                      // the rows as fp32 [NR][H]
  __shared__ int last;
  constexpr int U = 8;
  const int r0 = (int)blockIdx.y * NR, nr = R - r0 < NR ? R - r0 : NR, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int e = (int)blockIdx.x * ROUTER_WARPS + warp;
  uint4 raw[U];
  auto request = [&](int i0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * 8 * 32;
      raw[u] = i < H ? __ldg(reinterpret_cast<const uint4 *>(Wr + (size_t)e * H + i)) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  if (e < E) request(8 * lane);
  griddep_wait();
  x_hi = after_wait(x_hi);
  x_lo = after_wait(x_lo);
  bool any = !active;
  if (active)
    for (int q = 0; q < nr; ++q) any |= after_wait(active)[r0 + q] != 0;
  if (!any && blockIdx.x) return;                    // rows without a request need no logits; the first CTA writes their -1s
  if (any) {
    for (int i = 4 * tid; i < H; i += 4 * 32 * ROUTER_WARPS) {
      uint2 rh[NR], rl[NR];
#pragma unroll
      for (int q = 0; q < NR; ++q) {
        const size_t o = (size_t)(r0 + (q < nr ? q : 0)) * H + i;
        rh[q] = *reinterpret_cast<const uint2 *>(x_hi + o);
        rl[q] = *reinterpret_cast<const uint2 *>(x_lo + o);
      }
#pragma unroll
      for (int q = 0; q < NR; ++q) {
        const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&rh[q]), *l2 = reinterpret_cast<const __nv_bfloat162 *>(&rl[q]);
        const float2 h0 = __bfloat1622float2(h2[0]), h1 = __bfloat1622float2(h2[1]), l0 = __bfloat1622float2(l2[0]), l1 = __bfloat1622float2(l2[1]);
        *reinterpret_cast<float4 *>(xs + (size_t)q * H + i) = make_float4(h0.x + l0.x, h0.y + l0.y, h1.x + l1.x, h1.y + l1.y);
      }
    }
    __syncthreads();
    if (e < E) {
      float acc[NR] = {};
      for (int i0 = 8 * lane; i0 < H; i0 += U * 8 * 32) {
        if (i0 >= U * 8 * 32) request(i0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u * 8 * 32;
          if (i >= H) break;
          const __nv_bfloat162 *w2 = reinterpret_cast<const __nv_bfloat162 *>(&raw[u]);
          const float2 w0 = __bfloat1622float2(w2[0]), w1 = __bfloat1622float2(w2[1]), w2f = __bfloat1622float2(w2[2]), w3 = __bfloat1622float2(w2[3]);
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            const float4 xa = *reinterpret_cast<const float4 *>(xs + (size_t)q * H + i), xb = *reinterpret_cast<const float4 *>(xs + (size_t)q * H + i + 4);
            float a = acc[q];
            a = fmaf(w0.x, xa.x, a); a = fmaf(w0.y, xa.y, a); a = fmaf(w1.x, xa.z, a); a = fmaf(w1.y, xa.w, a);
            a = fmaf(w2f.x, xb.x, a); a = fmaf(w2f.y, xb.y, a); a = fmaf(w3.x, xb.z, a); a = fmaf(w3.y, xb.w, a);
            acc[q] = a;
          }
        }
      }
#pragma unroll
      for (int q = 0; q < NR; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
        if (lane == 0 && q < nr) rs.logit[(size_t)(r0 + q) * E + e] = acc[q];
      }
      if (lane == 0) __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
      last = gridDim.x == 1 || atomicAdd(rs.count + blockIdx.y, 1) == (int)gridDim.x - 1;
      __threadfence();
    }
    __syncthreads();
    if (!last) return;
    if (tid == 0) rs.count[blockIdx.y] = 0;          // for the next launch
  }
  if (warp < nr) {
    const int r = r0 + warp;
    moe_route_row([&](int e) { return any ? __ldcg(rs.logit + (size_t)r * E + e) : 0.f; }, r, lane, E, S, top_k, renormalize, w, experts,
                  probs, sel, !active || after_wait(active)[r] != 0);
  }
}

// h[r, e*F + f] = w[r, e] * silu(gate) * up as a bf16 hi/lo pair; zeros where w[r, e] == 0 (nothing is read
// there).  gate = GEMM-1 column e*2F + f, up = column e*2F + F + f.  Four f per thread.
__global__ void __launch_bounds__(256) moe_swiglu_kernel(GemmOut gu, const float *__restrict__ w, int F, int n_blocks,
                                                         bf16 *__restrict__ out_hi, bf16 *__restrict__ out_lo) {
  griddep_launch_dependents();
  griddep_wait();
  const int r = blockIdx.y;
  const int per_block = F / 4;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= per_block * n_blocks) return;
  const int e = idx / per_block, f = (idx - e * per_block) * 4;
  const float we = w[(size_t)r * n_blocks + e];
  float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
  if (we != 0.f) {
    const float4 g = gemm_load4(gu, r, e * 2 * F + f), u = gemm_load4(gu, r, e * 2 * F + F + f);
    y = make_float4(we * (g.x / (1.f + expf(-g.x)) * u.x), we * (g.y / (1.f + expf(-g.y)) * u.y),
                    we * (g.z / (1.f + expf(-g.z)) * u.z), we * (g.w / (1.f + expf(-g.w)) * u.w));
  }
  bf16 a[4], b[4];
  moe_split(y.x, a[0], b[0]);
  moe_split(y.y, a[1], b[1]);
  moe_split(y.z, a[2], b[2]);
  moe_split(y.w, a[3], b[3]);
  const size_t o = (size_t)r * n_blocks * F + (size_t)e * F + f;
  *reinterpret_cast<uint2 *>(out_hi + o) = *reinterpret_cast<const uint2 *>(a);
  *reinterpret_cast<uint2 *>(out_lo + o) = *reinterpret_cast<const uint2 *>(b);
}

// y[r, :] = the second GEMM's result (partials of a tile added in ascending CTA order).
__global__ void __launch_bounds__(256) moe_readout_kernel(GemmOut d, int H, float *__restrict__ y) {
  griddep_launch_dependents();
  griddep_wait();
  const int r = blockIdx.y;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (i >= H) return;
  *reinterpret_cast<float4 *>(y + (size_t)r * H + i) = gemm_load4(d, r, i);
}

// ---------------------------------------------------------------- grouped form
// One CTA per expert (routed experts, then the shared ones).  Every CTA counts the rows of ALL experts (the table
// w[r, e] != 0 is small and comes from L2), so that it knows where its own expert's groups begin (experts ascending,
// g.rows() rows per group) without a second kernel; it then writes its groups' table entries and hands its rows, in
// ascending row order, consecutive slots (slot_of is expert-major: [E + S][R]).  CTA 0 also clears the entries of
// the groups nobody needs and publishes the number of groups in use.
constexpr int MOE_GROUP_THREADS = 512;
__global__ void __launch_bounds__(MOE_GROUP_THREADS) moe_group_kernel(const float *__restrict__ w, const int *__restrict__ active, int R,
                                                       int NB, int E, int F, MoeGroups g) {
  griddep_launch_dependents();
  __shared__ int cnt[MOE_MAX_EXPERTS + 8];
  __shared__ float wsel[256];                        // the own expert's weight per row, 0 = not selected
  __shared__ unsigned char act[256];
  __shared__ int first_s, total_s;
  const int e = (int)blockIdx.x, tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < NB; i += MOE_GROUP_THREADS) cnt[i] = 0;
  griddep_wait();
  w = after_wait(w); active = after_wait(active);    // no load through them may move up across the wait
  for (int r = tid; r < R; r += MOE_GROUP_THREADS) { act[r] = active[r] != 0; wsel[r] = 0.f; }
  __syncthreads();
  {
    // sixteen independent loads per thread in flight
    const int total = R * NB;
    for (int i0 = tid; i0 < total; i0 += MOE_GROUP_THREADS * 16) {
      float v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = i0 + MOE_GROUP_THREADS * k < total ? w[i0 + MOE_GROUP_THREADS * k] : 0.f;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int i = i0 + MOE_GROUP_THREADS * k;
        if (i < total && v[k] != 0.f) {
          const int r = i / NB, ee = i - r * NB;
          if (act[r]) {
            atomicAdd(&cnt[ee], 1);                  // integer counts: the order of the additions does not matter
            if (ee == e) wsel[r] = v[k];
          }
        }
      }
    }
  }
  __syncthreads();
  if (warp == 0) {
    // groups before this expert, and in all: lanes take experts lane, lane + 32, ...
    int before = 0, all = 0;
    for (int ee = lane; ee < NB; ee += 32) {
      const int n = (cnt[ee] + g.rows() - 1) >> g.lg_rows;
      all += n;
      if (ee < e) before += n;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      before += __shfl_xor_sync(0xffffffffu, before, o);
      all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    if (lane == 0) { first_s = before; total_s = all < g.n_groups_max ? all : g.n_groups_max; }
  }
  __syncthreads();
  const int first = first_s, used = total_s;
  if (e == 0) {
    for (int u = used + tid; u < g.n_groups_max; u += MOE_GROUP_THREADS) {   // groups nobody needs
      g.tab_up[3 * u] = 0; g.tab_up[3 * u + 1] = 0; g.tab_up[3 * u + 2] = 0;
      g.tab_down[3 * u] = 0; g.tab_down[3 * u + 1] = 0; g.tab_down[3 * u + 2] = 0;
      g.group_expert[u] = -1;
    }
    if (tid == 0) g.tab_up[3 * g.n_groups_max] = g.tab_down[3 * g.n_groups_max] = used;   // what the GEMMs walk
  }
  const int n_groups = (cnt[e] + g.rows() - 1) >> g.lg_rows;
  for (int k = tid; k < n_groups; k += MOE_GROUP_THREADS) {
    const int u = first + k;
    if (u >= g.n_groups_max) break;                 // cannot happen: n_groups_max bounds the sum
    const int rows = min(g.rows(), cnt[e] - (k << g.lg_rows));
    g.tab_up[3 * u] = e * 2 * F; g.tab_up[3 * u + 1] = 0; g.tab_up[3 * u + 2] = rows;
    g.tab_down[3 * u] = 0; g.tab_down[3 * u + 1] = e * F / GEMM_BLOCK_K; g.tab_down[3 * u + 2] = rows;
    g.group_expert[u] = e;
  }
  if (warp == 0) {
    int base = (first << g.lg_rows);               // slot of the expert's next row
    for (int r0 = 0; r0 < R; r0 += 32) {
      const int r = r0 + lane;
      const float wv = r < R ? wsel[r] : 0.f;
      const bool on = wv != 0.f;
      const unsigned m = __ballot_sync(0xffffffffu, on);
      int slot = -1;
      if (on) {
        slot = base + __popc(m & ((1u << lane) - 1u));
        g.slot_row[slot] = r;
        g.slot_w[slot] = wv;
      }
      if (r < R) g.slot_of[(size_t)e * R + r] = slot;
      base += __popc(m);
    }
  }
}

// ---- many rows (up to MOE_MANY_ROWS): the kernel above reads the whole table w[r, e] in every CTA, 1 MB at 2048 rows and
// 128 experts.  Here a first kernel turns it into one bit per (expert, row), 64 KB in all, which every CTA of the second
// reads, and the second hands out the slots of all its rows at once.
constexpr int MOE_MASK_WORDS = MOE_MANY_ROWS / 32;

__global__ void __launch_bounds__(256) moe_mask_kernel(const float *__restrict__ w, const int *__restrict__ active, int R, int NB,
                                                       uint32_t *__restrict__ mask) {
  griddep_launch_dependents();
  griddep_wait();
  w = after_wait(w); active = after_wait(active);
  const int r0 = (int)blockIdx.x * 32, lane = (int)threadIdx.x & 31;
  const uint32_t on = __ballot_sync(0xffffffffu, r0 + lane < R && active[r0 + lane] != 0);   // the rows with a token
  for (int e = (int)threadIdx.x; e < NB; e += 256) {
    float v[32];                                     // all of the expert's loads in flight
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = r0 + i < R ? w[(size_t)(r0 + i) * NB + e] : 0.f;
    uint32_t m = 0u;
#pragma unroll
    for (int i = 0; i < 32; ++i) m |= v[i] != 0.f ? 1u << i : 0u;
    mask[e * MOE_MASK_WORDS + (int)blockIdx.x] = m & on;
  }
}

__global__ void __launch_bounds__(MOE_GROUP_THREADS) moe_group_many_kernel(const float *__restrict__ w, const uint32_t *__restrict__ mask, int R,
                                                                           int NB, int E, int F, MoeGroups g) {
  griddep_launch_dependents();
  __shared__ int cnt[MOE_MAX_EXPERTS + 8];
  __shared__ uint32_t own[MOE_MASK_WORDS];
  __shared__ int own_before[MOE_MASK_WORDS];         // the expert's rows before a word
  __shared__ int first_s, total_s;
  const int e = (int)blockIdx.x, tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int words = (R + 31) / 32;
  griddep_wait();
  w = after_wait(w); mask = after_wait(mask);
  for (int ee = warp; ee < NB; ee += MOE_GROUP_THREADS / 32) {
    uint32_t m[MOE_MASK_WORDS / 32];                 // word lane + 32 k
    int n[MOE_MASK_WORDS / 32], inc[MOE_MASK_WORDS / 32], all = 0;   // rows of a word, inclusive sums over the lanes
#pragma unroll
    for (int k = 0; k < MOE_MASK_WORDS / 32; ++k) {
      m[k] = lane + 32 * k < words ? mask[ee * MOE_MASK_WORDS + lane + 32 * k] : 0u;
      n[k] = inc[k] = __popc(m[k]);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int k = 0; k < MOE_MASK_WORDS / 32; ++k) {
        const int x = __shfl_up_sync(0xffffffffu, inc[k], o);
        if (lane >= o) inc[k] += x;
      }
#pragma unroll
    for (int k = 0; k < MOE_MASK_WORDS / 32; ++k) {
      if (ee == e) {
        own[lane + 32 * k] = m[k];
        own_before[lane + 32 * k] = all + inc[k] - n[k];
      }
      all += __shfl_sync(0xffffffffu, inc[k], 31);
    }
    if (lane == 0) cnt[ee] = all;
  }
  __syncthreads();
  if (warp == 0) {
    int before = 0, all = 0;
    for (int ee = lane; ee < NB; ee += 32) {
      const int n = (cnt[ee] + g.rows() - 1) >> g.lg_rows;
      all += n;
      if (ee < e) before += n;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      before += __shfl_xor_sync(0xffffffffu, before, o);
      all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    if (lane == 0) { first_s = before; total_s = all < g.n_groups_max ? all : g.n_groups_max; }
  }
  __syncthreads();
  const int first = first_s, used = total_s;
  if (e == 0) {
    for (int u = used + tid; u < g.n_groups_max; u += MOE_GROUP_THREADS) {   // groups nobody needs
      g.tab_up[3 * u + 2] = 0;
      g.tab_down[3 * u + 2] = 0;
    }
    if (tid == 0) g.tab_up[3 * g.n_groups_max] = g.tab_down[3 * g.n_groups_max] = used;   // what the GEMMs walk
  }
  const int n_groups = (cnt[e] + g.rows() - 1) >> g.lg_rows;
  for (int k = tid; k < n_groups; k += MOE_GROUP_THREADS) {
    const int u = first + k;
    if (u >= g.n_groups_max) break;                 // cannot happen: n_groups_max bounds the sum
    const int rows = min(g.rows(), cnt[e] - (k << g.lg_rows));
    g.tab_up[3 * u] = e * 2 * F; g.tab_up[3 * u + 1] = 0; g.tab_up[3 * u + 2] = rows;
    g.tab_down[3 * u] = 0; g.tab_down[3 * u + 1] = e * F / GEMM_BLOCK_K; g.tab_down[3 * u + 2] = rows;
    g.group_expert[u] = e;
  }
  for (int r = tid; r < R; r += MOE_GROUP_THREADS) {
    const uint32_t m = own[r >> 5], bit = 1u << (r & 31);
    int slot = -1;
    if (m & bit) {
      slot = (first << g.lg_rows) + own_before[r >> 5] + __popc(m & (bit - 1u));
      g.slot_row[slot] = r;
      g.slot_w[slot] = w[(size_t)r * NB + e];
    }
    g.slot_of[(size_t)e * R + r] = slot;
  }
}

// Routing of many rows: one warp per row.
__global__ void __launch_bounds__(256) moe_route_kernel(GemmOut logits, int R, int E, int S, int top_k, int renormalize,
                                                        float *__restrict__ w) {
  griddep_launch_dependents();
  griddep_wait();
  logits.direct = after_wait(logits.direct);
  logits.ws = after_wait(logits.ws);
  const int r = (int)blockIdx.x * 8 + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= R) return;
  moe_route_row([&](int e) { return gemm_load_pair(logits, r, e); }, r, lane, E, S, top_k, renormalize, w, nullptr, nullptr);
}

// The gathered activation rows: one warp per slot of the groups in use (all of a row's loads requested before the
// first store).  H % 256 == 0 up to 4096, else eight 16-byte pieces per lane at a time.
__global__ void __launch_bounds__(256) moe_gather_kernel(const bf16 *__restrict__ x_hi, const bf16 *__restrict__ x_lo, int H,
                                                         MoeGroups g, bf16 *__restrict__ xg_hi, bf16 *__restrict__ xg_lo) {
  griddep_launch_dependents();
  griddep_wait();
  x_hi = after_wait(x_hi); x_lo = after_wait(x_lo);
  const int lane = threadIdx.x & 31;
  const int n_slots = g.tab_up[3 * g.n_groups_max] << g.lg_rows;
  const int n_warps = (int)(gridDim.x * (blockDim.x >> 5));
  for (int slot = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); slot < n_slots; slot += n_warps) {
    if ((slot & (g.rows() - 1)) >= g.tab_up[3 * (slot >> g.lg_rows) + 2]) continue;   // no row in this slot
    const int r = g.slot_row[slot];
    const uint4 *sh = reinterpret_cast<const uint4 *>(x_hi + (size_t)r * H), *sl = reinterpret_cast<const uint4 *>(x_lo + (size_t)r * H);
    uint4 *dh = reinterpret_cast<uint4 *>(xg_hi + (size_t)slot * H), *dl = reinterpret_cast<uint4 *>(xg_lo + (size_t)slot * H);
    for (int i0 = lane; i0 < H / 8; i0 += 32 * 8) {
      uint4 a[8], b[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (i0 + 32 * k < H / 8) { a[k] = sh[i0 + 32 * k]; b[k] = sl[i0 + 32 * k]; }
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (i0 + 32 * k < H / 8) { dh[i0 + 32 * k] = a[k]; dl[i0 + 32 * k] = b[k]; }
    }
  }
}

__global__ void __launch_bounds__(256) moe_swiglu_grouped_kernel(const float *__restrict__ gu, const float *__restrict__ w,
                                                                 int NB, int F, MoeGroups g, bf16 *__restrict__ hg_hi,
                                                                 bf16 *__restrict__ hg_lo) {
  griddep_launch_dependents();
  griddep_wait();
  const int slot = blockIdx.x;
  if ((slot & (g.rows() - 1)) >= g.tab_up[3 * (slot >> g.lg_rows) + 2]) return;   // no row in this slot
  const int r = g.slot_row[slot];
  const int e = g.group_expert[slot >> g.lg_rows];
  const float we = w[(size_t)r * NB + e];
  const float *row = gu + (size_t)slot * 2 * F;
  for (int f = threadIdx.x * 4; f < F; f += blockDim.x * 4) {
    const float4 a = *reinterpret_cast<const float4 *>(row + f), u = *reinterpret_cast<const float4 *>(row + F + f);
    const float4 y = make_float4(we * (a.x / (1.f + expf(-a.x)) * u.x), we * (a.y / (1.f + expf(-a.y)) * u.y),
                                 we * (a.z / (1.f + expf(-a.z)) * u.z), we * (a.w / (1.f + expf(-a.w)) * u.w));
    bf16 p[4], q[4];
    moe_split(y.x, p[0], q[0]);
    moe_split(y.y, p[1], q[1]);
    moe_split(y.z, p[2], q[2]);
    moe_split(y.w, p[3], q[3]);
    *reinterpret_cast<uint2 *>(hg_hi + (size_t)slot * F + f) = *reinterpret_cast<const uint2 *>(p);
    *reinterpret_cast<uint2 *>(hg_lo + (size_t)slot * F + f) = *reinterpret_cast<const uint2 *>(q);
  }
}

// Selected-experts form: y[r, :] = the sum of the row's experts in ascending id; their rows sit at e * BN + r.  Negative
// entries (a vanished weight, a row without a request) have no such row: what is there belongs to other rows and steps.
__global__ void __launch_bounds__(256) moe_combine_select_kernel(const float *__restrict__ yg, const int *__restrict__ sel, int n_per_row,
                                                                 int BN, int H, float *__restrict__ y) {
  griddep_launch_dependents();
  griddep_wait();
  yg = after_wait(yg); sel = after_wait(sel);
  const int r = blockIdx.y, i = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
  const int *mine = sel + (size_t)r * n_per_row;
  if (i >= H) return;
  bool any = false;                                  // a row without a request has no entry
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int k0 = 0; k0 < n_per_row; k0 += 8) {        // eight loads in flight; the additions stay in ascending order
    int e[8];
    float4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      e[k] = k0 + k < n_per_row ? mine[k0 + k] : -1;
      if (e[k] >= 0) v[k] = *reinterpret_cast<const float4 *>(yg + ((size_t)e[k] * BN + r) * H + i);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (e[k] >= 0) { acc.x += v[k].x; acc.y += v[k].y; acc.z += v[k].z; acc.w += v[k].w; any = true; }
  }
  if (any) *reinterpret_cast<float4 *>(y + (size_t)r * H + i) = acc;
}

// One CTA per row: every expert's slot of the row is looked up by a thread of its own, then a thread adds four columns, eight experts'
// loads in flight.  Bound by the experts' rows (2505 rows of 2048 columns, 8 experts each: 164 MB).  With 256 threads (two CTAs a row,
// one warp walking the experts) 49.6 us, so 42.0; 1003 rows 18.7 and 16.1.
constexpr int COMBINE_THREADS = 512;
__global__ void __launch_bounds__(COMBINE_THREADS) moe_combine_kernel(const float *__restrict__ yg, const int *__restrict__ active, int NB,
                                                          int H, MoeGroups g, float *__restrict__ y) {
  griddep_launch_dependents();
  griddep_wait();
  yg = after_wait(yg); active = after_wait(active);
  const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (!active[r]) return;
  __shared__ int slots[MOE_MAX_EXPERTS + 8];         // the row's slots, experts ascending (shared experts last), compacted
  __shared__ int cnt[COMBINE_THREADS / 32];
  static_assert(MOE_MAX_EXPERTS + 8 <= COMBINE_THREADS, "a thread per expert");
  const int slot = tid < NB ? g.slot_of[(size_t)tid * gridDim.x + r] : -1;
  const unsigned m = __ballot_sync(0xffffffffu, slot >= 0);
  if (lane == 0) cnt[warp] = __popc(m);
  __syncthreads();
  int before = 0, n = 0;
#pragma unroll
  for (int k = 0; k < COMBINE_THREADS / 32; ++k) {
    const int c = cnt[k];
    if (k < warp) before += c;
    n += c;
  }
  if (slot >= 0) slots[before + __popc(m & ((1u << lane) - 1u))] = slot;
  __syncthreads();
  for (int i = 4 * tid; i < H; i += 4 * COMBINE_THREADS) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < n; k0 += 8) {              // eight loads in flight; the additions stay in ascending order
      float4 v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k0 + k < n) v[k] = *reinterpret_cast<const float4 *>(yg + (size_t)slots[k0 + k] * H + i);
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k0 + k < n) { acc.x += v[k].x; acc.y += v[k].y; acc.z += v[k].z; acc.w += v[k].w; }
    }
    *reinterpret_cast<float4 *>(y + (size_t)r * H + i) = acc;
  }
}

}  // namespace

namespace corun {

cudaError_t launch_moe_group(const float *w, const int *active, int R, int E, int S, int F, const MoeGroups &g,
                             cudaStream_t st) {
  if (E + S > MOE_MAX_EXPERTS + 8 || F % GEMM_BLOCK_K || R > 256) return cudaErrorInvalidValue;
  return launch_k(moe_group_kernel, dim3(E + S), dim3(MOE_GROUP_THREADS), 0, st, true, w, active, R, E + S, E, F, g);
}

cudaError_t launch_moe_group_many(const float *w, const int *active, int R, int E, int S, int F, uint32_t *mask, const MoeGroups &g,
                                  cudaStream_t st) {
  if (E + S > MOE_MAX_EXPERTS + 8 || F % GEMM_BLOCK_K || R > MOE_MANY_ROWS) return cudaErrorInvalidValue;
  cudaError_t e = launch_k(moe_mask_kernel, dim3((R + 31) / 32), dim3(256), 0, st, true, w, active, R, E + S, mask);
  if (e != cudaSuccess) return e;
  return launch_k(moe_group_many_kernel, dim3(E + S), dim3(MOE_GROUP_THREADS), 0, st, true, w, mask, R, E + S, E, F, g);
}

cudaError_t launch_moe_route(const GemmOut &logits, int R, int E, int S, int top_k, int renormalize, float *w, cudaStream_t st) {
  return launch_k(moe_route_kernel, dim3((R + 7) / 8), dim3(256), 0, st, true, logits, R, E, S, top_k, renormalize, w);
}

cudaError_t launch_moe_gather(const __nv_bfloat16 *x_hi, const __nv_bfloat16 *x_lo, int H, const MoeGroups &g,
                              __nv_bfloat16 *xg_hi, __nv_bfloat16 *xg_lo, cudaStream_t st) {
  const int blocks = ((g.n_groups_max << g.lg_rows) + 7) / 8;   // a warp per slot, as far as 1184 CTAs go
  return launch_k(moe_gather_kernel, dim3(blocks < 1184 ? blocks : 1184), dim3(256), 0, st, true, x_hi, x_lo, H, g, xg_hi, xg_lo);
}

cudaError_t launch_moe_swiglu_grouped(const float *gu, const float *w, int n_blocks, int F, const MoeGroups &g,
                                      __nv_bfloat16 *hg_hi, __nv_bfloat16 *hg_lo, cudaStream_t st) {
  return launch_k(moe_swiglu_grouped_kernel, dim3(g.n_groups_max << g.lg_rows), dim3(192), 0, st, true, gu, w, n_blocks, F, g,
                  hg_hi, hg_lo);
}

cudaError_t launch_moe_combine(const float *yg, const int *active, int R, int n_blocks, int H, const MoeGroups &g, float *y,
                               cudaStream_t st) {
  return launch_k(moe_combine_kernel, dim3(R), dim3(COMBINE_THREADS), 0, st, true, yg, active, n_blocks, H, g, y);
}

cudaError_t moe_router_prepare() {
  return cudaFuncSetAttribute(moe_router_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOE_MAX_HIDDEN * (int)sizeof(float));
}

cudaError_t launch_moe_router(const bf16 *x_hi, const bf16 *x_lo, int H, const bf16 *Wr, int R, int E, int S, int top_k,
                              int renormalize, float *w, int *experts, float *probs, const RouterScratch &rs, cudaStream_t st, const int *active,
                              int *sel) {
  const int shares = (E + ROUTER_WARPS - 1) / ROUTER_WARPS;
  auto go = [&](auto kernel, int n) {
    return launch_k(kernel, dim3(shares, (R + n - 1) / n), dim3(32 * ROUTER_WARPS), (size_t)n * H * sizeof(float), st, true, x_hi, x_lo, H, Wr,
                    R, E, S, top_k, renormalize, w, experts, probs, active, sel, rs);
  };
  // Few rows: the latency of one expert's weights bounds it, so a CTA per row and 8 experts (one CTA per row did all experts:
  // steps of 12 layers with 128 experts 1234 -> 1095 us at 1 row, 3890 -> 3770 at 40 of 64 rows; 4 rows a CTA 1139 / 3816).
  // Many rows: the weights from L2 once per row bound it (100 of 128 rows 4670 us, 4 rows a CTA 4609; 200 of 256 rows 5120
  // with one CTA per row, 5065 with 4 rows).  The rows of a CTA have to fit into 48 KB of shared memory.
  return R > 96 && 4 * (size_t)H * sizeof(float) <= 46 * 1024 ? go(moe_router_kernel<4>, 4) : go(moe_router_kernel<1>, 1);
}

cudaError_t launch_moe_combine_select(const float *yg, const int *sel, int n_per_row, int BN, int R, int H, float *y, cudaStream_t st) {
  return launch_k(moe_combine_select_kernel, dim3((H / 4 + 255) / 256, R), dim3(256), 0, st, true, yg, sel, n_per_row, BN, H, y);
}

cudaError_t launch_moe_swiglu(const GemmOut &gu, const float *w, int R, int F, int n_blocks, __nv_bfloat16 *out_hi,
                              __nv_bfloat16 *out_lo, cudaStream_t st) {
  return launch_k(moe_swiglu_kernel, dim3((n_blocks * (F / 4) + 255) / 256, R), dim3(256), 0, st, true, gu, w, F, n_blocks,
                  out_hi, out_lo);
}

}  // namespace corun

struct corun_moe {
  corun_moe_shape sh{};
  int B = 0, BN = 0, num_sms = 0;
  cudaStream_t st = nullptr;
  std::vector<void *> allocs;
  const bf16 *router = nullptr;                     // [E, H], borrowed
  bf16 *x_hi = nullptr, *x_lo = nullptr, *h_hi = nullptr, *h_lo = nullptr;
  float *out_gu = nullptr, *out_d = nullptr, *ws = nullptr, *w = nullptr;
  int *d_status = nullptr;
  GemmPlan p_gu, p_d;
  // grouped form (more than 64 padded rows): an expert's rows gathered into blocks of 64
  RouterScratch rs{};
  bool grouped = false;
  MoeGroups grp{};
  bf16 *xg_hi = nullptr, *xg_lo = nullptr, *hg_hi = nullptr, *hg_lo = nullptr;
  float *yg = nullptr;
  int *d_active = nullptr;
  GemmPlan p_gug, p_dng;
  int64_t weight_bytes = 0;
};

namespace {

template <typename T>
int moe_alloc(corun_moe *m, T **p, size_t n) {
  void *q = nullptr;
  if (cudaMalloc(&q, n * sizeof(T)) != cudaSuccess) return CORUN_ENOMEM;
  m->allocs.push_back(q);
  if (cudaMemset(q, 0, n * sizeof(T)) != cudaSuccess) return CORUN_ECUDA;
  *p = (T *)q;
  return CORUN_OK;
}

}  // namespace

extern "C" {

int corun_moe_create(const corun_moe_shape *shape, const void *router, const void *gate_up, const void *down,
                     int32_t B, void *cuda_stream, corun_moe **out) {
  if (!shape || !router || !gate_up || !down || !out || B < 1 || B > 256) return CORUN_EINVAL;
  const corun_moe_shape &s = *shape;
  if (s.hidden < 64 || s.hidden % 64 || s.hidden > MOE_MAX_HIDDEN || s.n_experts < 1 || s.n_experts > MOE_MAX_EXPERTS || s.top_k < 1 ||
      s.top_k > MOE_MAX_TOPK || s.top_k > s.n_experts || s.expert_ffn < 64 || s.expert_ffn % 64 || s.n_shared < 0)
    return CORUN_EINVAL;
  corun_moe *m = new (std::nothrow) corun_moe();
  if (!m) return CORUN_ENOMEM;
  auto fail = [&](int rc) { corun_moe_destroy(m); return rc; };
  m->sh = s;
  m->B = B;
  m->BN = (B + 15) / 16 * 16;
  m->st = (cudaStream_t)cuda_stream;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || moe_router_prepare() != cudaSuccess)
    return fail(CORUN_ECUDA);
  const int H = s.hidden, E = s.n_experts, F = s.expert_ffn, NB = E + s.n_shared;
  const size_t N1 = (size_t)NB * 2 * F, K2 = (size_t)NB * F;
  if (N1 > (size_t)1 << 30 || K2 > (size_t)1 << 30) return fail(CORUN_EINVAL);
  int rc;
  if ((rc = moe_alloc(m, &m->x_hi, (size_t)m->BN * H)) ||
      (rc = moe_alloc(m, &m->x_lo, (size_t)m->BN * H)) || (rc = moe_alloc(m, &m->h_hi, (size_t)m->BN * K2)) ||
      (rc = moe_alloc(m, &m->h_lo, (size_t)m->BN * K2)) ||
      (rc = moe_alloc(m, &m->out_gu, (size_t)m->BN * N1)) || (rc = moe_alloc(m, &m->out_d, (size_t)m->BN * H)) ||
      (rc = moe_alloc(m, &m->ws, gemm_ws_floats(m->num_sms, m->BN))) || (rc = moe_alloc(m, &m->w, (size_t)B * NB)) ||
      (rc = moe_alloc(m, &m->rs.logit, (size_t)B * E)) || (rc = moe_alloc(m, &m->rs.count, (size_t)B)) ||
      (rc = moe_alloc(m, &m->d_status, 1)))
    return fail(rc);
  m->router = (const bf16 *)router;
  // the three GEMMs run one after the other and their results are consumed in between: one workspace serves all
  // the form without groups: from 65 to 128 rows (used there only where the grouped form below does not apply) the
  // first GEMM applies the routing weight and the SwiGLU in its epilogue (where a tile width divides the experts'
  // width); else it stores gate / up sums and a kernel of its own follows (faster up to 64 rows, where the masked
  // store skips most of the output)
  const bool fused = m->BN > 64 && m->BN <= 128 && gemm_swiglu_blocks_half(F, NB, m->num_sms) > 0;
  if ((rc = fused ? gemm_plan_create_swiglu_blocks(&m->p_gu, gate_up, NB, F, H, m->x_hi, m->x_lo, B, m->BN, m->h_hi, m->h_lo, m->w, m->num_sms)
                  : gemm_plan_create(&m->p_gu, gate_up, (int)N1, H, m->x_hi, m->x_lo, B, m->BN, m->out_gu, m->ws, m->num_sms)) ||
      (rc = gemm_plan_create(&m->p_d, down, H, (int)K2, m->h_hi, m->h_lo, B, m->BN, m->out_d, m->ws, m->num_sms)))
    return fail(rc);
  if (!fused && (2 * F) % GEMM_TILE_N == 0) {       // a weight tile then belongs to one expert: skip the rows that
    m->p_gu.row_keep = m->w;                        // did not select it (the SwiGLU kernel does not read them)
    m->p_gu.keep_pitch = NB;
    m->p_gu.keep_div = 2 * F / GEMM_TILE_N;
  }
  // above 64 padded rows: the grouped form (an expert's rows gathered into blocks of 64, of which as many are multiplied as there
  // are; every row through every expert would be (E + S) / (top_k + S) times the MMA work), with the routing weight and the SwiGLU in
  // the per-group gate / up GEMM's epilogue
  const int g_half = gemm_swiglu_blocks_half(F, NB, m->num_sms);
  if (m->BN > 64 && g_half > 0 && H % GEMM_TILE_N == 0 && !getenv("CORUN_MOE_DECODE_DENSE")) {
    MoeGroups &g = m->grp;
    g.lg_rows = 6;
    g.n_groups_max = moe_max_groups(B, E, s.n_shared, s.top_k, g.lg_rows);
    const size_t slots = (size_t)g.n_groups_max << g.lg_rows;
    if ((rc = moe_alloc(m, &g.tab_up, (size_t)g.n_groups_max * 3 + 1)) || (rc = moe_alloc(m, &g.tab_down, (size_t)g.n_groups_max * 3 + 1)) ||
        (rc = moe_alloc(m, &g.group_expert, (size_t)g.n_groups_max)) || (rc = moe_alloc(m, &g.slot_row, slots)) ||
        (rc = moe_alloc(m, &g.slot_of, (size_t)B * NB)) || (rc = moe_alloc(m, &g.slot_w, slots)) ||
        (rc = moe_alloc(m, &m->xg_hi, slots * H)) || (rc = moe_alloc(m, &m->xg_lo, slots * H)) ||
        (rc = moe_alloc(m, &m->hg_hi, slots * F)) || (rc = moe_alloc(m, &m->hg_lo, slots * F)) ||
        (rc = moe_alloc(m, &m->yg, slots * H)) || (rc = moe_alloc(m, &m->d_active, (size_t)B)))
      return fail(rc);
    std::vector<int> ones((size_t)B, 1);
    if (cudaMemcpy(m->d_active, ones.data(), (size_t)B * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess) return fail(CORUN_ECUDA);
    if ((rc = gemm_plan_create_grouped_swiglu(&m->p_gug, gate_up, (long long)NB * 2 * F, F, H, g_half, m->xg_hi, m->xg_lo, g.n_groups_max,
                                              g.rows(), m->hg_hi, m->hg_lo, g.slot_w, g.tab_up, m->num_sms)) ||
        (rc = gemm_plan_create_grouped(&m->p_dng, down, H, NB * F, H, F, m->hg_hi, m->hg_lo, g.n_groups_max, g.rows(), m->yg,
                                       g.tab_down, m->num_sms)))
      return fail(rc);
    m->grouped = true;
  }
  m->weight_bytes = ((int64_t)E * H + (int64_t)N1 * H + (int64_t)H * K2) * 2;
  if (cudaDeviceSynchronize() != cudaSuccess) return fail(CORUN_ECUDA);
  *out = m;
  return CORUN_OK;
}

void corun_moe_destroy(corun_moe *m) {
  if (!m) return;
  cudaStreamSynchronize(m->st);
  gemm_plan_destroy(&m->p_gu);
  gemm_plan_destroy(&m->p_d);
  gemm_plan_destroy(&m->p_gug);
  gemm_plan_destroy(&m->p_dng);
  for (void *p : m->allocs) cudaFree(p);
  delete m;
}

int corun_moe_forward(corun_moe *m, const float *x, float *y, int32_t *experts, float *probs) {
  if (!m || !x || !y || x == y) return CORUN_EINVAL;
  if (((uintptr_t)y & 15u) || ((uintptr_t)x & 3u)) return CORUN_EINVAL;   // y is stored 16 bytes at a time
  const corun_moe_shape &s = m->sh;
  const int H = s.hidden, E = s.n_experts, F = s.expert_ffn, NB = E + s.n_shared;
  MCK(launch_split(x, m->B, H, m->x_hi, m->x_lo, m->st));
  MCK(launch_moe_router(m->x_hi, m->x_lo, H, m->router, m->B, E, s.n_shared, s.top_k, s.renormalize, m->w, experts, probs, m->rs, m->st));
  if (m->grouped) {
    // rows grouped by expert -> gate / up with routing weight and SwiGLU, and down, per group -> the row's experts
    // summed in ascending expert id
    MCK(launch_moe_group(m->w, m->d_active, m->B, E, s.n_shared, F, m->grp, m->st));
    MCK(launch_moe_gather(m->x_hi, m->x_lo, H, m->grp, m->xg_hi, m->xg_lo, m->st));
    MCK(gemm_launch(m->p_gug, nullptr, m->d_status, m->st, nullptr, true));
    MCK(gemm_launch(m->p_dng, nullptr, m->d_status, m->st, nullptr, true));
    MCK(launch_moe_combine(m->yg, m->d_active, m->B, NB, H, m->grp, y, m->st));
    return CORUN_OK;
  }
  MCK(gemm_launch(m->p_gu, nullptr, m->d_status, m->st, nullptr, true));
  if (!m->p_gu.sw_hi) MCK(launch_moe_swiglu(m->p_gu.out(), m->w, m->B, F, NB, m->h_hi, m->h_lo, m->st));
  MCK(gemm_launch(m->p_d, nullptr, m->d_status, m->st, nullptr, true));
  MCK(launch_k(moe_readout_kernel, dim3((H / 4 + 255) / 256, m->B), dim3(256), 0, m->st, true, m->p_d.out(), H, y));
  return CORUN_OK;
}

int corun_moe_sync(corun_moe *m) {
  if (!m) return CORUN_EINVAL;
  int hs = 0;
  MCK(cudaMemcpyAsync(&hs, m->d_status, sizeof(int), cudaMemcpyDeviceToHost, m->st));
  MCK(cudaStreamSynchronize(m->st));
  return hs ? CORUN_ETIMEOUT : CORUN_OK;
}

int64_t corun_moe_weight_bytes(const corun_moe *m) { return m ? m->weight_bytes : 0; }

int corun_moe_launches(const corun_moe *m) { return m ? (m->grouped ? 7 : m->p_gu.sw_hi ? 5 : 6) : CORUN_EINVAL; }

}  // extern "C"
