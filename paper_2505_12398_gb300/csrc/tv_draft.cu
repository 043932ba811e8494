// tv_draft.cu -- drafting a token tree's children without replacement
// (Definition 1) from the draft rows (sm_103a).
//
// Every child c of node i takes the pre-drawn uniform u[c] and is drawn by
// inverse CDF, in ascending token order, from M_s(.|X^i) with the tokens of
// i's earlier children removed: the smallest y with u[c] W < CDF'(y), where
// CDF' and W = CDF'(V - 1) are the cumulative sums of the row with those
// tokens zeroed.  Siblings are drawn in child-index order, the order in which
// the verification tests them.
//
// One cluster of S CTAs per (tree, row); rows without children return at
// once.  The CTAs stream the row once: each warp reduces 256-token tiles (8
// tokens a lane, four tiles in flight) to float32 tile sums, which go to the
// first CTA's shared memory.  One warp of that CTA takes the float64 prefix of 32
// runs of tiles, and draws the children in order: the first run, in it the
// first tile, in it the first lane's 8 tokens and in them the first token whose
// prefix, less the masses of the earlier siblings' tokens up to there, exceeds
// u W (a ballot and, below the runs, a warp scan each).  The row is read from HBM
// once; a child costs one tile re-read (from L2).
//
// What bounds it: many trees, HBM; few, a row's latency on one SM (32 KB in
// flight) and the children one after another.  Float64 is scarce (a warp's
// instruction takes the SM's unit for 16 cycles, a dependent one 64), so a child
// is drawn with about 28 of them by one warp, without barriers, its siblings'
// uniforms loaded ahead and its mass taken from the registers that hold it.
// With S > 1 while all rows' CTAs fit the GPU at once (clusters_per_row), against
// one CTA per row and a search of the tiles by all its threads through shared-
// memory atomics (60-node trees): B = 1, V = 128256 30.7 -> 20.5 us, B = 8 47.7 ->
// 39.2, B = 128 343 -> 327 us (7.0 TB/s); B = 64, V = 32000 65.4 -> 53.7 us;
// unaligned rows (element loads before): B = 1, V = 128255 43.3 -> 22.7 us, B =
// 32, V = 32003 59.7 -> 39.6 us.
//
// The cumulative sums are float64 over float32 tile sums, so a draw whose
// u W lies within about 1e-6 W of a step of the exact CDF may land on the
// neighbouring token.  If rounding leaves u W past the scanned tile (or past
// the whole row), the last token of positive mass there is taken.  No mass
// left for a child (more children than tokens of positive draft probability,
// or a row that does not sum to a positive finite value) gives -1 for it and
// its later siblings and raises TV_STATUS_DRAFT_EXHAUSTED.
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/tv.h"
#include "tv_launch.h"
#include "tv_ptx.cuh"

namespace tvk {
namespace draft {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kTile = 256;   // tokens per tile: 32 lanes x 8

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The 8 draft probabilities of tokens x0 .. x0+7 (0 past the end; x0 % 8 == 0).
// Rows that do not start on 16 bytes are read as the three aligned quads the 8
// tokens lie in, except at the row's ends.
template <bool kVec>
__device__ __forceinline__ void load8(const float* __restrict__ q, int x0, int V, float* v) {
  if (kVec && x0 + 8 <= V) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(q + x0));
    const float4 b = __ldg(reinterpret_cast<const float4*>(q + x0 + 4));
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  } else if (!kVec && x0 >= 8 && x0 + 12 <= V) {
    const int sh = (int)((reinterpret_cast<uintptr_t>(q) >> 2) & 3u);   // the same in the row
    const float4* p = reinterpret_cast<const float4*>(q + x0 - sh);
    const float4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
    const float w[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
#pragma unroll
    for (int k = 0; k < 8; ++k)
      v[k] = sh < 2 ? (sh == 0 ? w[k] : w[k + 1]) : (sh == 2 ? w[k + 2] : w[k + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = x0 + k < V ? __ldg(q + x0 + k) : 0.f;
  }
}

__device__ __forceinline__ double warp_inclusive_scan(double v, int lane) {
  double x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Tree blockIdx.x / S, row blockIdx.y, S CTAs (kSplit: S > 1).  Dynamic shared memory
// (draft_smem_bytes): rem_q[R] f64, tsum[n_tiles] f32, par[R], kids[R],
// rem_tok[R] int32.
template <bool kVec, bool kSplit>
__global__ void __launch_bounds__(kThreads)
    tv_draft_kernel(const int32_t* __restrict__ parents, const float* __restrict__ drafts,
                    const float* __restrict__ uniforms, int32_t* __restrict__ tokens, int N,
                    int V, int split, uint32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int n_kids;
  const int S = kSplit ? split : 1;
  const int R = N + 1, b = blockIdx.x / S, i = blockIdx.y;
  const int rank = kSplit ? (int)cluster_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_tiles = (V + kTile - 1) / kTile;
  double* rem_q = reinterpret_cast<double*>(smem);
  float* tsum = reinterpret_cast<float*>(rem_q + R);
  int* par = reinterpret_cast<int*>(tsum + n_tiles);
  int* kids = par + R;
  int* rem_tok = kids + R;
  const int32_t* pb = parents + (size_t)b * R;
  int32_t* tb = tokens + (size_t)b * R;

  // ---- the tree's parents: valid (parents[0] = -1, parents[c] in [0, c))?
  int badl = 0;
  for (int c = tid; c < R; c += kThreads) {
    const int p = pb[c];
    par[c] = p;
    if (c == 0 ? p != -1 : (p < 0 || p >= c)) badl = 1;
  }
  if (__syncthreads_or(badl)) {
    if (i == 0 && rank == 0) {   // one CTA of the tree reports it
      for (int c = tid; c < R; c += kThreads) tb[c] = c == 0 ? 0 : -1;
      if (tid == 0) atomicOr(status, (uint32_t)TV_STATUS_BAD_TREE);
    }
    return;
  }
  if (i == 0 && rank == 0 && tid == 0) tb[0] = 0;

  // ---- the children of row i, in index order (warp 0, 32 candidates a step)
  if (warp == 0) {
    int n = 0;
    for (int c0 = i + 1; c0 < R; c0 += 32) {
      const int c = c0 + lane;
      const bool is_kid = c < R && par[c] == i;
      const unsigned m = __ballot_sync(0xffffffffu, is_kid);
      if (is_kid) kids[n + __popc(m & ((1u << lane) - 1u))] = c;
      n += __popc(m);
    }
    if (lane == 0) n_kids = n;
  }
  __syncthreads();
  const int nk = n_kids;
  if (nk == 0) return;   // (every CTA of the cluster)

  // ---- stream the row once: float32 sums of 256-token tiles
  const float* q = drafts + ((size_t)b * R + i) * (size_t)V;
  // four tiles a warp per step (two of unaligned rows; loads past the end read as
  // zeros), so that enough bytes are in flight to stream at the copy bandwidth
  constexpr int kU = kVec ? 4 : 2;
  const int n_warps = S * kWarps;
  if (kSplit) cluster_sync_all();  // the first CTA has started: its shared memory is there
  for (int t = rank * kWarps + warp; t < n_tiles; t += kU * n_warps) {
    float v[kU][8];
#pragma unroll
    for (int k = 0; k < kU; ++k) load8<kVec>(q, (t + k * n_warps) * kTile + lane * 8, V, v[k]);
#pragma unroll
    for (int k = 0; k < kU; ++k) {
      const float s = ((v[k][0] + v[k][1]) + (v[k][2] + v[k][3])) +
                      ((v[k][4] + v[k][5]) + (v[k][6] + v[k][7]));
      const float ts = warp_sum_f(s);
      if (lane == 0 && t + k * n_warps < n_tiles) {
        if (rank == 0) tsum[t + k * n_warps] = ts;
        else st_cluster_f32(map_shared(&tsum[t + k * n_warps], 0), ts);
      }
    }
  }
  if (kSplit) {
    cluster_sync_all();            // every CTA's sums have arrived
    if (rank != 0) return;
  } else {
    __syncthreads();
  }

  if (warp != 0) return;

  // ---- float64 prefix of the runs of tiles: lane r has tiles [r per, (r + 1) per)
  const int per = (n_tiles + 31) / 32;
  const int t_lo = min(n_tiles, lane * per), t_hi = min(n_tiles, t_lo + per);
  double run = 0.0;
  {
    double odd = 0.0;              // (two chains: half the dependent additions)
    int t = t_lo;
    for (; t + 1 < t_hi; t += 2) {
      run += (double)tsum[t];
      odd += (double)tsum[t + 1];
    }
    if (t < t_hi) run += (double)tsum[t];
    run += odd;
  }
  const double upto = warp_inclusive_scan(run, lane);   // through the lane's run
  const double total = __shfl_sync(0xffffffffu, upto, 31);

  // ---- the children, in order
  double rsum = 0.0;               // mass of the earlier siblings' tokens
  const float* u = uniforms + (size_t)b * R;
  float u_own = lane < nk ? __ldg(u + kids[lane]) : 0.f;
  for (int j = 0; j < nk; ++j) {
    const int c = kids[j];
    if (j > 0 && (j & 31) == 0) u_own = j + lane < nk ? __ldg(u + kids[j + lane]) : 0.f;
    const double W = total - rsum;
    if (!(W > 0.0) || !isfinite(W)) {   // the same decision in every lane
      for (int r = j + lane; r < nk; r += 32) tb[kids[r]] = -1;
      if (lane == 0) atomicOr(status, (uint32_t)TV_STATUS_DRAFT_EXHAUSTED);
      return;
    }
    const double target = (double)__shfl_sync(0xffffffffu, u_own, j & 31) * W;
    // the first run whose prefix, less the earlier siblings' masses up to its
    // end, exceeds u W (none: u W is at or past the end by rounding)
    double incl = upto;
    for (int r = 0; r < j; ++r)
      if (rem_tok[r] / kTile < t_hi) incl -= rem_q[r];
    const unsigned in_run = __ballot_sync(0xffffffffu, target < incl);
    int y = -1, ts = n_tiles - 1;
    float qy = 0.f;
    bool take_last = in_run == 0u;
    if (!take_last) {
      const int f = __ffs(in_run) - 1;
      const int r_lo = f * per, r_hi = min(n_tiles, r_lo + per);
      double base = f > 0 ? __shfl_sync(0xffffffffu, incl, f - 1) : 0.0;
      // the first tile of the run, 32 at a time
      ts = -1;
      for (int t0 = r_lo; t0 < r_hi && ts < 0; t0 += 32) {
        const int t = t0 + lane;
        double d = t < r_hi ? (double)tsum[t] : 0.0;
        for (int r = 0; r < j; ++r)
          if (t < r_hi && rem_tok[r] / kTile == t) d -= rem_q[r];
        const double x = base + warp_inclusive_scan(d, lane);
        const unsigned m = __ballot_sync(0xffffffffu, t < r_hi && target < x);
        if (m) {
          const int l = __ffs(m) - 1;
          ts = t0 + l;
          if (l > 0) base = __shfl_sync(0xffffffffu, x, l - 1);
        } else {
          base = __shfl_sync(0xffffffffu, x, 31);
        }
      }
      if (ts < 0) {   // rounding left u W past the run's tiles
        ts = r_hi - 1;
        take_last = true;
      } else {
        // the first lane's 8 tokens of the tile
        const int x0 = ts * kTile + lane * 8;
        float v[8];
        load8<kVec>(q, x0, V, v);
        for (int r = 0; r < j; ++r) {
          const int off = rem_tok[r] - x0;
#pragma unroll
          for (int k = 0; k < 8; ++k) if (k == off) v[k] = 0.f;
        }
        const double ls = (((double)v[0] + (double)v[1]) + ((double)v[2] + (double)v[3])) +
                          (((double)v[4] + (double)v[5]) + ((double)v[6] + (double)v[7]));
        const double x = base + warp_inclusive_scan(ls, lane);
        const unsigned m = __ballot_sync(0xffffffffu, target < x);
        if (m) {
          const int l = __ffs(m) - 1;
          if (l > 0) base = __shfl_sync(0xffffffffu, x, l - 1);
          // those 8 tokens, one a lane: the first whose prefix exceeds u W
          float w = 0.f;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float z = __shfl_sync(0xffffffffu, v[k], l);
            if (lane == k) w = z;
          }
          double p = (double)w;
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) {
            const double z = __shfl_up_sync(0xffffffffu, p, o);
            if (lane >= o) p += z;
          }
          const unsigned hit = __ballot_sync(0xffffffffu, lane < 8 && target < base + p);
          const unsigned pos = __ballot_sync(0xffffffffu, lane < 8 && w > 0.f);
          // (none: the lane's sum crossed u W, its prefixes did not)
          const int k = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : -1);
          if (k >= 0) {
            y = ts * kTile + l * 8 + k;
            qy = __shfl_sync(0xffffffffu, w, k);
          }
        } else {
          take_last = true;   // rounding left u W past this tile
        }
      }
    }
    if (take_last) {
      // the last token of positive mass at or before the tile
      for (int t = ts; t >= 0 && y < 0; --t) {
        const int x0 = t * kTile + lane * 8;
        float v[8];
        load8<kVec>(q, x0, V, v);
        int last = -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          bool rm = false;
          for (int r = 0; r < j; ++r) rm |= rem_tok[r] == x0 + k;
          if (!rm && v[k] > 0.f) last = x0 + k;
        }
        const unsigned m = __ballot_sync(0xffffffffu, last >= 0);
        if (m) y = __shfl_sync(0xffffffffu, last, 31 - __clz(m));
      }
      qy = y >= 0 ? __ldg(q + y) : 0.f;
    }
    rsum += (double)qy;
    if (lane == 0) {
      tb[c] = y;
      rem_tok[j] = y;
      rem_q[j] = (double)qy;
      if (y < 0) atomicOr(status, (uint32_t)TV_STATUS_DRAFT_EXHAUSTED);
    }
    __syncwarp();
  }
}

// CTAs per row: as many as keep the CTAs of all rows (with or without
// children) on the GPU at once, 4 per SM, with at least 4096 tokens each.
int clusters_per_row(int B, int R, int V, int sms) {
  int S = 8;
  while (S > 1 && ((long long)B * R * S > 4LL * sms || V / S < 4096)) S /= 2;
  return S;
}

}  // namespace draft
}  // namespace tvk

namespace {
size_t draft_smem_bytes(int N, int V) {
  const size_t R = (size_t)N + 1, tiles = ((size_t)V + tvk::draft::kTile - 1) / tvk::draft::kTile;
  return tiles * 4 + R * 20;
}
}  // namespace

// (The limit the entry point has always had: 12 bytes a tile, 20 a node, 48 KB.)
bool tv_draft_fits(int N, int V) {
  const size_t tiles = ((size_t)V + tvk::draft::kTile - 1) / tvk::draft::kTile;
  return tiles * 12 + ((size_t)N + 1) * 20 <= 48 * 1024;
}

int tv_launch_draft(const int32_t* parents, const float* drafts, const float* uniforms,
                    int32_t* tokens, int B, int N, int V, int sm_count, uint32_t* status,
                    cudaStream_t stream) {
  using namespace tvk::draft;
  if (B <= 0) return 0;
  const bool vec = (V % 4) == 0 && (reinterpret_cast<uintptr_t>(drafts) & 15u) == 0;
  const int S = clusters_per_row(B, N + 1, V, sm_count);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(B * S), (unsigned)(N + 1), 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = draft_smem_bytes(N, V);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = S > 1 ? 1 : 0;
  auto kernel = vec ? (S > 1 ? tv_draft_kernel<true, true> : tv_draft_kernel<true, false>)
                    : (S > 1 ? tv_draft_kernel<false, true> : tv_draft_kernel<false, false>);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, parents, drafts, uniforms, tokens, N, V,
                                           S, status);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess ? 0 : -5;
}
