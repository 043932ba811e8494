// tv_kernels.cu -- CUDA kernels of batched Traversal Verification (sm_103a).
//
// One call verifies B independent trees in three kernels on one stream:
//
//   tv_prep_kernel       one warp per tree: structural checks of the parent
//                        array and the token range, then appends the tree's
//                        internal rows (rows with >= 1 child) to a work list.
//   tv_row_stats_kernel  the row normaliser of every internal row, fully
//                        parallel over B x |I| rows: one streaming pass with an
//                        online max / sum of exp2((l - m) log2(e) / T).  These
//                        are the target distributions M_b(.|X^i) Algorithm 3
//                        initialises its acceptance rates from (§3.1).
//   tv_tree_kernel       (tv_tree.cu) the traversal of Algorithm 3 (Appendix E
//                        order), one cluster per tree, with those normalisers.
//
// This is the path of vocabularies that are not a multiple of 8: rows start
// anywhere, so they are read as whole 8-element blocks of the flat
// [B][N+1][V] arrays (16- or 32-byte loads), the neighbouring rows' elements in
// the first and last block masked.  Measured (32 trees of 60 nodes, V = 32003,
// bf16), against element loads and one CTA per tree: 330.6 -> 149.8 us.
//
// The mutable distributions of Algorithm 3 are never materialised.  After k
// rejections at node i (children tokens t_0..t_{k-1} removed) they are, for
// every token x not yet removed,
//     M_b^(k)(x) = [a_k M_b^(0)(x) - b_k M_s^(0)(x)]_+,   M_s^(k)(x) = M_s^(0)(x) / Z_k,
// with a_0 = 1, b_0 = 0, Z_0 = 1 and, at the rejection with rate p and sum S,
//     a_{k+1} = p a_k / S,   b_{k+1} = (p b_k + 1/Z_k) / S,   Z_{k+1} = Z_k - M_s^(0)(t_k),
// which is Eq. (1) and Eq. (2) applied to that form.  A removed token t keeps
// M_s = 0 and M_b(t) = m_t, stored per removed child and rescaled by p / S at
// each later rejection.  Each rejection therefore streams the ORIGINAL target
// and draft rows of the parent once, with two scalars and the short sorted
// list of removed tokens.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tv_device.cuh"
#include "tv_launch.h"

namespace tvk {

// ------------------------------------------------------------------ prep --

__global__ void __launch_bounds__(256) tv_prep_kernel(const int32_t* __restrict__ parents,
                                                      const int32_t* __restrict__ tokens,
                                                      int B, int R, int V,
                                                      int32_t* __restrict__ row_list,
                                                      int32_t* __restrict__ n_rows) {
  __shared__ uint32_t s_has[8][32];   // one bit per row (R <= 1024), per warp
  const int wl = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int tree = blockIdx.x * 8 + wl;
  s_has[wl][lane] = 0u;
  __syncwarp();
  if (tree >= B) return;
  const int32_t* par = parents + (size_t)tree * R;
  const int32_t* tok = tokens + (size_t)tree * R;
  bool bad = false;
  for (int i = lane; i < R; i += 32) {
    int p = par[i];
    if (i == 0) {
      bad |= (p != -1);
    } else {
      int t = tok[i];
      bad |= (t < 0 || t >= V);
      if (p < 0 || p >= i) bad = true;
      else atomicOr(&s_has[wl][p >> 5], 1u << (p & 31));
    }
  }
  bad = __any_sync(0xffffffffu, bad);
  __syncwarp();
  if (bad) return;   // the traversal kernel reports it; no row work queued
  uint32_t word = s_has[wl][lane];
  int cnt = __popc(word);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  int total = __shfl_sync(0xffffffffu, incl, 31);
  int base = 0;
  if (lane == 31) base = atomicAdd(n_rows, total);
  base = __shfl_sync(0xffffffffu, base, 31);
  int pos = base + incl - cnt;
  while (word) {
    int bit = __ffs(word) - 1;
    word &= word - 1;
    row_list[pos++] = tree * R + lane * 32 + bit;
  }
}

// ------------------------------------------------------------- row stats --

constexpr int kStatsThreads = 256;
constexpr int kStatsUnroll = 4;

// One block's eight logits added to a thread's running (max, sum): `n_all`
// elements in the arrays, [lo, hi) of the block's belong to the row.
template <typename L>
__device__ __forceinline__ void stats_block(const typename L::elem* logits, size_t at,
                                            size_t n_all, int lo, int hi, float v[8]) {
  if (at + 8 <= n_all) {
    L::chunk_vec(logits + at, 0, v);
  } else {                       // the arrays' last, partial block
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = k < hi ? L::at(logits + at, k) : TV_NEG_INF;
  }
  if (lo > 0 || hi < 8) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < lo || k >= hi) v[k] = TV_NEG_INF;
  }
}

template <typename L>
__device__ __forceinline__ void stats_add(const float v[8], int lo, int hi, float c_hi, float c_lo,
                                          float& m, Comp& acc) {
  const float cm = fmaxf(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])),
                         fmaxf(fmaxf(v[4], v[5]), fmaxf(v[6], v[7])));
  if (cm > m) {
    if (m != TV_NEG_INF) {
      const float sc = L::exp_rel(m, cm, c_hi, c_lo);
      acc.s *= sc;
      acc.c *= sc;
    }
    m = cm;
  }
  if (m != TV_NEG_INF) {
    float t[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) t[e] = L::exp_rel(v[e], m, c_hi, c_lo);
    if (lo > 0 || hi < 8) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (e < lo || e >= hi) t[e] = 0.f;
    }
    acc.add(sum8(t));
  }
}

template <typename L>
__global__ void __launch_bounds__(kStatsThreads) tv_row_stats_kernel(
    const typename L::elem* __restrict__ logits, int V, size_t n_all, float c_hi, float c_lo,
    const int32_t* __restrict__ row_list, const int32_t* __restrict__ n_rows,
    float2* __restrict__ stats) {
  __shared__ float s_red[kStatsThreads / 32];
  __shared__ float s_max;
  const int n = *n_rows;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int r = blockIdx.x; r < n; r += gridDim.x) {
    const int g = row_list[r];
    // the row's first 8-element block and its elements of the row before
    const size_t first = (size_t)g * V;
    const int sh = (int)(first & 7u);
    const size_t base = first - (size_t)sh;
    const int end = V + sh;              // the row is [sh, end) from base
    // phase 1: per-thread online max / sum relative to that max
    float m = TV_NEG_INF;
    Comp acc;
    const int step = kStatsThreads * kChunk;
    int x0 = threadIdx.x * kChunk;
    for (; x0 + (kStatsUnroll - 1) * step < end; x0 += kStatsUnroll * step) {
      float v[kStatsUnroll][8];
#pragma unroll
      for (int u = 0; u < kStatsUnroll; ++u)
        stats_block<L>(logits, base + x0 + u * step, n_all, sh - (x0 + u * step),
                       end - (x0 + u * step), v[u]);
#pragma unroll
      for (int u = 0; u < kStatsUnroll; ++u)
        stats_add<L>(v[u], sh - (x0 + u * step), end - (x0 + u * step), c_hi, c_lo, m, acc);
    }
    for (; x0 < end; x0 += step) {
      float v[8];
      stats_block<L>(logits, base + x0, n_all, sh - x0, end - x0, v);
      stats_add<L>(v, sh - x0, end - x0, c_hi, c_lo, m, acc);
    }
    // phase 2: the row max, then every partial rescaled once to it and summed
    float bm = warp_max(m);
    if (lane == 0) s_red[wid] = bm;
    __syncthreads();
    if (wid == 0) {
      float x = (lane < kStatsThreads / 32) ? s_red[lane] : TV_NEG_INF;
      x = warp_max(x);
      if (lane == 0) s_max = x;
    }
    __syncthreads();
    const float M = s_max;
    float part = (m == TV_NEG_INF) ? 0.f : acc.value() * L::exp_rel(m, M, c_hi, c_lo);
    part = warp_sum(part);
    __syncthreads();
    if (lane == 0) s_red[wid] = part;
    __syncthreads();
    if (wid == 0) {
      float x = (lane < kStatsThreads / 32) ? s_red[lane] : 0.f;
      x = warp_sum(x);
      if (lane == 0) stats[g] = make_float2(M, x);
    }
    __syncthreads();
  }
}

}  // namespace tvk

// --------------------------------------------------------------- launchers --

namespace {
int launch_error() {
  return (cudaGetLastError() == cudaSuccess) ? 0 : -5;
}
}  // namespace

// (97 bytes a row and 8 for every 256 tokens: the sizes this path has always
// taken, all of which the cluster kernel's plan covers.)
bool tv_tree_fits(int R, int V, size_t smem_per_block) {
  return (size_t)R * 97 + ((size_t)V + 255) / 256 * 8 + 64 <= smem_per_block;
}

namespace {

template <typename L>
int launch_typed(const TravArgs& a, int logit_is_bf16, int* row_list, int* n_rows, int stats_grid,
                 const FusedPlan& plan, cudaStream_t stream, cudaEvent_t* ev) {
  const int R = a.N + 1;
  const auto* lg = reinterpret_cast<const typename L::elem*>(a.logits);
  if (ev && cudaEventRecord(ev[0], stream) != cudaSuccess) return -5;
  if (cudaMemsetAsync(n_rows, 0, sizeof(int), stream) != cudaSuccess) return -5;
  tvk::tv_prep_kernel<<<(a.B + 7) / 8, 256, 0, stream>>>(a.parents, a.tokens, a.B, R, a.V,
                                                          row_list, n_rows);
  if (launch_error()) return -5;
  if (ev && cudaEventRecord(ev[1], stream) != cudaSuccess) return -5;
  tvk::tv_row_stats_kernel<L><<<stats_grid, tvk::kStatsThreads, 0, stream>>>(
      lg, a.V, (size_t)a.B * R * (size_t)a.V, a.c_hi, a.c_lo, row_list, n_rows, a.stats);
  if (launch_error()) return -5;
  if (ev && cudaEventRecord(ev[2], stream) != cudaSuccess) return -5;
  TravArgs t = a;
  t.row_stats = a.stats;
  t.stats_given = 0;
  t.exact_exp = 1;
  if (tv_launch_tree(t, logit_is_bf16, plan, stream) != 0) return -5;
  if (ev && cudaEventRecord(ev[3], stream) != cudaSuccess) return -5;
  return 0;
}

}  // namespace

int tv_launch_all(const TravArgs& a, int logit_is_bf16, int* row_list, int* n_rows,
                  int stats_grid, const FusedPlan& plan, cudaStream_t stream,
                  cudaEvent_t* events) {
  if (!plan.ok) return -5;
  return logit_is_bf16
             ? launch_typed<tvk::Bf16Logits>(a, 1, row_list, n_rows, stats_grid, plan, stream, events)
             : launch_typed<tvk::F32Logits>(a, 0, row_list, n_rows, stats_grid, plan, stream, events);
}
