// tv_kernels.cu -- CUDA kernels of batched Traversal Verification (sm_103a).
//
// The path with separate row normalisers: one call verifies B independent trees in
// two kernels on one stream:
//
//   tv_row_stats_kernel  the row normaliser of every internal row (a row with at
//                        least one child; the others' blocks leave at once), one
//                        block per row: one streaming pass with an online max /
//                        sum of exp2((l - m) log2(e) / T).  These are the target
//                        distributions M_b(.|X^i) Algorithm 3 initialises its
//                        acceptance rates from (§3.1).
//   tv_tree_kernel       (tv_tree.cu) the traversal of Algorithm 3 (Appendix E
//                        order), one cluster per tree, with those normalisers.
//
// This is the path of vocabularies that are not a multiple of 8: rows start
// anywhere, so they are read as whole 8-element blocks of the flat
// [B][N+1][V] arrays (16- or 32-byte loads), the neighbouring rows' elements in
// the first and last block masked.  Measured (32 trees of 60 nodes, V = 32003,
// bf16), against element loads and one CTA per tree: 330.6 -> 149.8 us; then the
// list of internal rows that a first kernel made (with a cleared counter) left to
// the normalisers' blocks, and their arithmetic as below: -> 119 us.
//
// The normaliser kernel is bound by its arithmetic, a third of the HBM rate: 16
// instructions per logit at 69 % of the issue slots before the maximum of a pair
// of bf16 took one instruction and the logits stayed packed until they are used (48
// registers, five blocks per SM).  With four blocks of logits per thread at a time,
// also at a row's end, and two weights per instruction, against one block at a time
// and scalar arithmetic: 256 trees, V = 32003 270 -> 155 us, 32 trees 45 -> 30 us
// (the bytes alone 92 and 11 us).
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

// ------------------------------------------------------------- row stats --

constexpr int kStatsUnroll = 4;

template <typename L, int kStatsThreads>
__global__ void __launch_bounds__(kStatsThreads, kStatsThreads == 256 ? 6 - L::kBytes / 2 : 1)
    tv_row_stats_kernel(const typename L::elem* __restrict__ logits,
                        const int32_t* __restrict__ parents, int R, int V, float c_hi, float c_lo,
                        float2* __restrict__ stats) {
  __shared__ float s_red[kStatsThreads / 32];
  __shared__ float s_max;
  asm volatile("griddepcontrol.launch_dependents;");   // (the traversal waits for this grid)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int g = blockIdx.x, node = g % R;
  {
    const int32_t* par = parents + (g - node);
    int child = 0;
    for (int i = threadIdx.x; i < R; i += kStatsThreads) child |= i > 0 && par[i] == node;
    if (!__syncthreads_or(child)) return;
  }
  // the row's first 8-element block and its elements of the row before
  const size_t first = (size_t)g * V;
  const int sh = (int)(first & 7u);
  const size_t base = first - (size_t)sh;
  const int end = V + sh;              // the row is [sh, end) from base
  // phase 1: per-thread online max / sum relative to that max
  float m = TV_NEG_INF;
  Comp acc;
  const int step = kStatsThreads * kChunk;
  const float2 ch = make_float2(c_hi, c_hi), cl = make_float2(c_lo, c_lo);
  for (int x0 = threadIdx.x * kChunk; x0 < end; x0 += kStatsUnroll * step) {
    typename L::block v[kStatsUnroll];
    const bool edge = x0 < sh || x0 + (kStatsUnroll - 1) * step + kChunk > end;
    if (!edge) {
#pragma unroll
      for (int u = 0; u < kStatsUnroll; ++u)
        v[u] = L::load_block(logits + base + x0 + u * step);
    } else {
#pragma unroll
      for (int u = 0; u < kStatsUnroll; ++u) {
        const int x = x0 + u * step;
        if (x >= sh && x + kChunk <= end) v[u] = L::load_block(logits + base + x);
        else v[u] = L::make_block(logits + base + x, sh - x, end - x);
      }
    }
    float cm = L::block_max(v[0]);
#pragma unroll
    for (int u = 1; u < kStatsUnroll; ++u) cm = fmaxf(cm, L::block_max(v[u]));
    if (cm > m) {
      if (m != TV_NEG_INF) {
        const float sc = L::exp_rel(m, cm, c_hi, c_lo);
        acc.s *= sc;
        acc.c *= sc;
      }
      m = cm;
    }
    if (m == TV_NEG_INF) continue;
#pragma unroll
    for (int u = 0; u < kStatsUnroll; ++u) {
      const int x = x0 + u * step;
      if (x >= end) break;
      float2 t[4];
      L::block_exp(v[u], m, ch, cl, t);
      const float2 p = __fadd2_rn(__fadd2_rn(t[0], t[1]), __fadd2_rn(t[2], t[3]));
      acc.add(p.x + p.y);
    }
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
    // a finite max has weight 1: no normaliser where there is none
    if (!(x >= 1e-30f) || (L::kBytes == 4 && M == -TV_NEG_INF)) x = 0.f;
    if (lane == 0) stats[g] = make_float2(M, x);
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

template <typename L, int kThreads>
void launch_stats(const TravArgs& a, cudaStream_t stream) {
  const int R = a.N + 1;
  tvk::tv_row_stats_kernel<L, kThreads><<<a.B * R, kThreads, 0, stream>>>(
      reinterpret_cast<const typename L::elem*>(a.logits), a.parents, R, a.V, a.c_hi, a.c_lo,
      a.stats);
}

template <typename L>
int launch_typed(const TravArgs& a, int logit_is_bf16, const FusedPlan& plan, int sm_count,
                 cudaStream_t stream, cudaEvent_t* ev) {
  if (ev && cudaEventRecord(ev[0], stream) != cudaSuccess) return -5;
  if (ev && cudaEventRecord(ev[1], stream) != cudaSuccess) return -5;
  // Few rows: more threads on each, as long as every thread has a block or more.
  // Measured (us; the call with 256 / 512 / 1024 threads; 60-node trees, half of
  // their rows internal): V = 128251 bf16, 61 rows 48 / 41 / 38; V = 151933 fp32, 244
  // rows 136 / 124 / 120; V = 32003, 61 rows 94 / 93 / 93, 488 rows 99 / 97 / 99, 1952
  // rows 119 / 124 / 141; V = 1003, 1952 rows 105 / 109 / 117.
  const long rows = (long)a.B * (a.N + 1);
  if (rows <= 304 && a.V > 32768) launch_stats<L, 1024>(a, stream);
  else if (rows <= 608 && a.V > 8192) launch_stats<L, 512>(a, stream);
  else launch_stats<L, 256>(a, stream);
  if (launch_error()) return -5;
  if (ev && cudaEventRecord(ev[2], stream) != cudaSuccess) return -5;
  TravArgs t = a;
  t.row_stats = a.stats;
  t.stats_given = 0;
  t.exact_exp = 1;
  // The traversal starts while the normalisers' last blocks run (a programmatic
  // dependent launch): 54 -> 48 us at B = 1, V = 128251, 104 -> 99 us at B = 8, V =
  // 32003.  Not where its clusters share SMs: they would then crowd on the SMs that
  // are free first (119 -> 126 us at B = 32, V = 32003, 449 -> 463 us at B = 256);
  // single CTAs do not: 170 -> 165 us at B = 512, V = 4001, 774 -> 767 us at B = 600, V
  // = 32003.
  const bool dependent = ev == nullptr && (plan.C == 1 || (long)a.B * plan.C <= sm_count);
  if (tv_launch_tree(t, logit_is_bf16, plan, stream, dependent) != 0) return -5;
  if (ev && cudaEventRecord(ev[3], stream) != cudaSuccess) return -5;
  return 0;
}

}  // namespace

int tv_launch_all(const TravArgs& a, int logit_is_bf16, const FusedPlan& plan, int sm_count,
                  cudaStream_t stream, cudaEvent_t* events) {
  if (!plan.ok) return -5;
  return logit_is_bf16 ? launch_typed<tvk::Bf16Logits>(a, 1, plan, sm_count, stream, events)
                       : launch_typed<tvk::F32Logits>(a, 0, plan, sm_count, stream, events);
}
