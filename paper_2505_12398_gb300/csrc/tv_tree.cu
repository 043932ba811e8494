// tv_tree.cu -- one thread-block cluster per tree: lazy, latency-oriented
// Traversal Verification (sm_103a).
//
// One kernel does all of Algorithm 3 (§3.1) for a batch of trees.  Each tree
// is owned by a cluster of C CTAs (1 to 16): CTA r streams the vocabulary slice
// [v0_r, v1_r) of every row the tree needs, and every CTA runs the same serial
// control on identical data, so their decisions agree without being broadcast;
// only partial results cross the cluster.
//
// What bounds it: a tree is a chain of 10 to 30 dependent vocabulary jobs
// (normalisers of a chain of rows, rejection passes, the bonus draw), each of
// a few microseconds, so the time is the sum of the latencies along that chain,
// not bandwidth.  The kernel is built to keep each link short:
//   * warp-specialised: NCW consumer warps reduce, a producer warp issues the
//     bulk copies (TMA), a control warp runs the serial control.  While a pass
//     runs, the control warp works out the step after it (Ahead), so that one
//     float64 comparison and at most one division stand between a pass's S and
//     the next job;
//   * every consumer warp sends its partial straight to the control warps of
//     all C CTAs (st.async: the store carries its own completion count), with
//     no reduction inside the CTA in between; two exchange buffers alternate;
//   * a normaliser job takes up to kStatRows rows of the chain being entered,
//     each row by a group of warps, with one exchange for all of them; the
//     rows' final sums and their children's float64 masses are spread over the
//     consumer warps;
//   * the consumers take all their tiles of a chunk in one straight line (no
//     test per tile for removed tokens, edges or lengths where a look at the
//     whole chunk rules them out), so that the tiles' chains of dependent
//     operations overlap: one tile at a time a warp took 1160 cycles a tile.
//   * where a slice of a (target, draft) row pair fits the ring, it stays there:
//     the next pass at the same node (about half of all passes) reads no
//     memory, and with room for two the parent's pair is fetched while the
//     node's passes run.
//
// Rows are read lazily.  The target row of a node is streamed (for its
// normaliser) only when the traversal first descends through the node, so
// sub-trees the traversal never enters cost nothing.  Each rejection needs the
// parent's ORIGINAL target and draft rows (the (a, b, Z) closed form of
// Eqs. (1)-(2), see tv_kernels.cu); the bonus draw streams one row (pair).
//
// Rows need no alignment: slices are copied as whole 8-element blocks of the
// flat [B][N+1][V] arrays and the elements of the neighbouring rows in the
// first and last block are masked.  (With V % 8 != 0 the kernel runs as the last
// of the two-kernel path, with the row normalisers that path computes first.)
//
// Every wait is bounded; one that gives up raises TV_STATUS_TIMEOUT, and all
// roles still reach the cluster barrier at the end.
//
// Measured (60-node trees, bf16; 8-token chains, fp32), against one thread of the
// consumers doing the control, a reduction and an exchange per row and no
// resident pairs: V = 32000, B = 64 254 -> 139 us (183 with a row by all warps in turn
// and before the removal of a rate-0 sibling and the descent into a sub-tree were
// worked out ahead, 149 one tile at a time); 16 chains 117 -> 61 us; V = 128256, B =
// 32 368 -> 184 us (213 one tile at a time).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "tv_control.cuh"
#include "tv_device.cuh"
#include "tv_launch.h"
#include "tv_ptx.cuh"

namespace tvk {
namespace fused {

constexpr int kTreeMaxStages = 16;
constexpr int kTreeMaxSlots = 8;     // resident row pairs tracked at most
constexpr int kStatRows = 8;         // rows of one normaliser job at most

// Tiles of 256 tokens one consumer warp takes per ring stage.
__host__ __device__ constexpr int tiles_per_warp(int ncw) { return ncw == 16 ? 1 : 2; }

// One ring stage holds tiles_per_warp tiles per consumer warp of target and
// draft values, or (normalisers, leaf draws) that many bytes of target values.
__host__ __device__ constexpr int tree_stage_bytes(int ncw, int lb) {
  return ncw * tiles_per_warp(ncw) * kTileElems * (lb + 4);
}

// Groups of consumer warps in a normaliser job of n rows: row r is summed by
// group r % groups, so that a warp reduces and sends for few rows; no more
// groups than warps or than rows fit the ring at once (`most`).
__host__ __device__ constexpr int row_groups(int n, int most) {
  int g = 1;
  while (2 * g <= n && 2 * g <= most) g *= 2;
  return g;
}
// Partials of one exchange at most (rows x CTAs x warps per group): a job
// takes up to four rows per group.
__host__ __device__ constexpr int exchange_slots(int C, int ncw) { return 4 * C * ncw; }

// A job as the control warp hands it to the CTA's other warps.
struct TreeJob {
  int kind, node, n_rows, nmask;
  float alpha1, beta, rowmax;
  int total;               // ring chunks the job loads (0: its pair is resident)
  int slot;                // resident slot of a pair (-1: streamed through the ring)
  uint32_t ph;             // parities of the stages' latest fills before the job
  int mbuf;                // which list of removed tokens
  int xb, xph;             // exchange buffer and the parity of its barrier
  int rows[kStatRows];
};

struct TreeShared {
  Ctl ctl;
  Ahead ahead;
  TreeJob job;
  // the resident row pairs, tracked by the control warp: node and last use
  int slot_node[kTreeMaxSlots];
  int slot_used[kTreeMaxSlots];
};

// Sends (x, y) to slot address `dst` of a CTA of the cluster; the store counts
// 8 bytes on that CTA's barrier `bar` (both addresses from map_shared).
__device__ __forceinline__ void st_async_v2(uint32_t dst, float x, float y, uint32_t bar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
          dst),
      "f"(x), "f"(y), "r"(bar)
      : "memory");
}

__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity) ? 1 : 0) != 0;
}

// A row's slice [v0, v1) as whole 8-element blocks of the flat array: first
// element of the first block, elements of the previous row in it, and the
// length from that block's start.
struct Slice {
  size_t base;
  int sh, n;
  __device__ __forceinline__ Slice(size_t row, int V, int v0, int v1) {
    const size_t f = row * (size_t)V + (size_t)v0;
    sh = (int)(f & 7u);
    base = f - (size_t)sh;
    n = v1 > v0 ? v1 - v0 + sh : 0;
  }
};

__device__ __forceinline__ int chunks_of(int n, int per) { return (n + per - 1) / per; }

// Eight logits of one lane: bf16 widened, or fp32.
template <typename L>
__device__ __forceinline__ void lds_logits(const typename L::elem* p, float v[8]) {
  if constexpr (L::kBytes == 2) {
    float2 vp[4];
    bf16x8_pairs(lds128(p), vp);
#pragma unroll
    for (int k = 0; k < 4; ++k) { v[2 * k] = vp[k].x; v[2 * k + 1] = vp[k].y; }
  } else {
    const uint4 a = lds128(p), b = lds128(p + 4);
    v[0] = __uint_as_float(a.x); v[1] = __uint_as_float(a.y);
    v[2] = __uint_as_float(a.z); v[3] = __uint_as_float(a.w);
    v[4] = __uint_as_float(b.x); v[5] = __uint_as_float(b.y);
    v[6] = __uint_as_float(b.z); v[7] = __uint_as_float(b.w);
  }
}

__device__ __forceinline__ float max8(const float v[8]) {
  return fmaxf(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])),
               fmaxf(fmaxf(v[4], v[5]), fmaxf(v[6], v[7])));
}

// e(x) of eight logits relative to m (kPass: the cheaper form of passes and
// draws, which leaves NaN for a weight of 0; see tv_device.cuh).
template <typename L, bool kPass>
__device__ __forceinline__ void exp8(const float v[8], float m, float c_hi, float c_lo,
                                     float e[8]) {
  if constexpr (L::kBytes == 2) {
    const float2 mm = make_float2(-m, -m), ch = make_float2(c_hi, c_hi),
                 cl = make_float2(c_lo, c_lo);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 d = __fadd2_rn(make_float2(v[2 * k], v[2 * k + 1]), mm);
      const float2 r = kPass ? exp2_corrected_x2(d, ch, cl) : exp2_split_zero_x2(d, ch, cl);
      e[2 * k] = r.x;
      e[2 * k + 1] = r.y;
    }
  } else {
    const float2 ch = make_float2(c_hi, c_hi), cl = make_float2(c_lo, c_lo);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 r = L::exp_rel_x2(make_float2(v[2 * k], v[2 * k + 1]), m, ch, cl);
      e[2 * k] = r.x;
      e[2 * k + 1] = r.y;
    }
  }
}

// [alpha e(x) - beta q(x)]_+ of eight tokens.
template <typename L, bool kExact>
__device__ __forceinline__ void residual8(const float v[8], const float* qp, float rowmax,
                                          float alpha, float beta, float c_hi, float c_lo,
                                          float t[8]) {
  const uint4 qa = lds128(qp), qc = lds128(qp + 4);
  const float q[8] = {__uint_as_float(qa.x), __uint_as_float(qa.y), __uint_as_float(qa.z),
                      __uint_as_float(qa.w), __uint_as_float(qc.x), __uint_as_float(qc.y),
                      __uint_as_float(qc.z), __uint_as_float(qc.w)};
  float e[8];
  exp8<L, !kExact>(v, rowmax, c_hi, c_lo, e);
  const float2 al2 = make_float2(alpha, alpha), nb2 = make_float2(-beta, -beta);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 x = __ffma2_rn(al2, make_float2(e[2 * k], e[2 * k + 1]),
                                __fmul2_rn(nb2, make_float2(q[2 * k], q[2 * k + 1])));
    t[2 * k] = fmaxf(x.x, 0.f);
    t[2 * k + 1] = fmaxf(x.y, 0.f);
  }
}

// Up to eight logits / draft probabilities of a block in global memory,
// elements outside [lo, hi) of the block read as -inf / 0.
template <typename L>
__device__ __forceinline__ void block_logits(const typename L::elem* p, int lo, int hi,
                                             float v[8]) {
  if (lo <= 0 && hi >= 8) {
    L::chunk_vec(p, 0, v);
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = (k >= lo && k < hi) ? L::at(p, k) : TV_NEG_INF;
  }
}

__device__ __forceinline__ void block_probs(const float* p, int lo, int hi, float q[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) q[k] = (k >= lo && k < hi) ? __ldg(p + k) : 0.f;
}

// ------------------------------------------------------------- kernel -----

template <typename L, int NCW, bool kExact>
struct TreeCta {
  using E = typename L::elem;
  static constexpr int kLB = L::kBytes;
  static constexpr int kStageBytes = tree_stage_bytes(NCW, kLB);
  static constexpr int kPair = kStageBytes / (kLB + 4);   // tokens of a pair chunk
  static constexpr int kRow = kStageBytes / kLB;          // tokens of a target-only chunk
  static constexpr int kSweep = NCW * kTileElems;
  static constexpr int kTiles = tiles_per_warp(NCW);      // per warp in a pair chunk
  static constexpr int kThreads = NCW * 32 + 64;          // + producer, control warps
  static_assert(kPair % kTileElems == 0, "whole tiles per stage");

  const TravArgs& a;
  TreeSmem s;
  TreeShared& sh;
  char* ring;
  float2* xs;              // [2][exchange_slots] partials of all CTAs
  int* mtok_ahead;         // [2][R] removed tokens of passes worked out ahead
  float* u;                // [R + 1] the tree's uniforms
  uint64_t *full_bar, *empty_bar, *xbar, *job_bar, *ack_bar, *stat_bar, *tile_bar,
      *order_bar;
  int C, n_stages, b, v0, v1;
  int spc;                 // stages a resident pair takes
  int max_groups;          // groups of a normaliser job at most
  uint32_t rank;
  size_t row0;             // the tree's first row in the batch

  __device__ TreeCta(const TravArgs& args, TreeShared& shared) : a(args), sh(shared) {}

  __device__ __forceinline__ void fail() { atomicOr(&sh.ctl.bad, 32u); }
  __device__ __forceinline__ float2* xslots(int buf) const {
    return xs + buf * exchange_slots(C, NCW);
  }
  // Lists of removed tokens: 0 the control's own, 1 and 2 worked out ahead.
  __device__ __forceinline__ int* mtok(int k) const {
    return k == 0 ? s.mask_tok : mtok_ahead + (size_t)(k - 1) * (a.N + 1);
  }
  static __device__ __forceinline__ bool is_pair(int kind) {
    return kind == kJobPass || kind == kJobBonusRes;
  }

  // e(x) in draws and passes: the cheaper form, or (kExact: the two-kernel path,
  // whose normalisers come from exp_rel) that one.
  __device__ __forceinline__ float exp1(float v, float m) const {
    return kExact ? L::exp_rel(v, m, a.c_hi, a.c_lo) : L::exp_pass(v, m, a.c_hi, a.c_lo);
  }

  // ---------------------------------------------------------- producer --
  // Fills stage `st` with the slice's chunk from element x of its first block
  // (n_all: elements of the arrays).
  __device__ void fill(int st, const Slice& sl, int x, bool pair, size_t n_all) {
    const size_t e0 = sl.base + (size_t)x;
    const int n = (min(pair ? kPair : kRow, sl.n - x) + 7) & ~7;   // whole blocks
    char* dst = ring + (size_t)st * kStageBytes;
    int whole = n;
    if (e0 + n > n_all) {
      // the last, partial block of the arrays: its elements one by one
      whole = (int)((n_all - e0) & ~(size_t)7);
      const int tail = (int)(n_all - e0);
      const E* lg = reinterpret_cast<const E*>(a.logits);
      for (int j = whole; j < tail; ++j) {
        reinterpret_cast<E*>(dst)[j] = lg[e0 + j];
        if (pair) reinterpret_cast<float*>(dst + (size_t)kPair * kLB)[j] = a.draft_probs[e0 + j];
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    const uint32_t lbytes = (uint32_t)whole * kLB, qbytes = pair ? (uint32_t)whole * 4u : 0u;
    mbar_arrive_expect_tx(&full_bar[st], lbytes + qbytes);
    if (whole > 0) {
      tma_load_1d(dst, reinterpret_cast<const E*>(a.logits) + e0, lbytes, &full_bar[st]);
      if (pair)
        tma_load_1d(dst + (size_t)kPair * kLB, a.draft_probs + e0, qbytes, &full_bar[st]);
    }
  }
  __device__ size_t elements() const { return (size_t)a.B * (a.N + 1) * (size_t)a.V; }

  // Streams the jobs' rows (one lane).
  __device__ bool produce() {
    const size_t n_all = elements();
    uint32_t jp = 0u, eph = 0u;
    for (;;) {
      if (!mbar_wait(job_bar, jp)) return false;
      jp ^= 1u;
      const TreeJob& t = sh.job;
      const int kind = t.kind, total = t.total, slot = t.slot, n_rows = t.n_rows, node = t.node;
      mbar_arrive(ack_bar);   // (a job that loads is replaced only once its rows are reduced)
      if (kind == kJobDone) return true;
      if (total == 0) continue;
      const bool pair = is_pair(kind);
      const int per = pair ? kPair : kRow;
      int st = slot > 0 ? slot * spc : 0;
      int q = 0;
      uint32_t ph = t.ph, mine = 0u;
      for (int r = 0; r < n_rows; ++r) {
        const Slice sl(row0 + (kind == kJobStats ? sh.job.rows[r] : node), a.V, v0, v1);
        for (int x = 0; x < sl.n; x += per, ++q) {
          if (q >= n_stages) {               // a stage of this job, used again
            if (!mbar_wait(&empty_bar[st], (eph >> st) & 1u)) {
              // (the consumers gave up: the copies under way land first)
              for (; mine != 0u; mine &= mine - 1u) {
                const int k = __ffs(mine) - 1;
                mbar_wait(&full_bar[k], (ph >> k) & 1u);
              }
              return false;
            }
            eph ^= 1u << st;
          }
          fill(st, sl, x, pair, n_all);
          mine |= 1u << st;
          ph ^= 1u << st;
          if (++st == n_stages) st = 0;
        }
      }
    }
  }

  // ---------------------------------------------------------- exchange --
  // A partial to slot `slot` of every CTA.  The exchange's barrier
  // counts the bytes of all CTAs' partials (the control warp arms it); a tree
  // of one CTA is launched without a cluster, so there the warps store to
  // their own slots and arrive once per job (arrive_alone).
  __device__ __forceinline__ void send(int xb, int slot, int lane, float x, float y) {
    if (C == 1) {
      if (lane == 0) xslots(xb)[slot] = make_float2(x, y);
    } else if (lane < C) {
      st_async_v2(map_shared(xslots(xb) + slot, lane), x, y, map_shared(&xbar[xb], lane));
    }
  }
  __device__ __forceinline__ void arrive_alone(int xb, int lane) {
    if (C == 1 && lane == 0) mbar_arrive(&xbar[xb]);
  }
  __device__ __forceinline__ bool exchanged(int xb, uint32_t parity) {   // a whole warp
    if (C == 1) return mbar_wait_warp(&xbar[xb], parity);
    return __all_sync(0xffffffffu, mbar_wait_cluster(&xbar[xb], parity) ? 1 : 0) != 0;
  }

  // --------------------------------------------------------- consumers --

  // The eight logits of the lane's block e0 of a stage, whose elements [lo, hi)
  // belong to the slice (the others read as -inf).
  __device__ __forceinline__ void stage_logits(const E* lb, int e0, bool valid, bool edge, int lo,
                                               int hi, float v[8]) const {
    if (valid) {
      lds_logits<L>(lb + e0, v);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = TV_NEG_INF;
    }
    if (edge) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (e < lo || e >= hi) v[e] = TV_NEG_INF;
    }
  }
  static __device__ __forceinline__ void zero_outside(bool edge, int lo, int hi, float t[8]) {
    if (edge) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (e < lo || e >= hi) t[e] = 0.f;
    }
  }

  // After chunk q of `total` in stage st: releases the stage where the producer
  // waits for it, and moves to the next.
  __device__ __forceinline__ void end_chunk(int q, int total, int& st, int lane) {
    if (q + n_stages < total) {
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty_bar[st]);
    }
    if (++st == n_stages) st = 0;
  }

  // Whether a removed token lies in this warp's tiles of a pair chunk (n tokens
  // from element x of the slice; the same in the whole warp).
  __device__ __forceinline__ bool removed_here(int n, int x, const int* mt, int nmask,
                                               int wid) const {
    const int xs = v0 + x;
    for (int k = 0; k < nmask; ++k) {
      const int off = mt[k] - xs;
      if ((unsigned)off < (unsigned)n && (off / kTileElems) % NCW == wid) return true;
    }
    return false;
  }

  // Row normalisers: this warp's group takes every g-th row.  (Rows of whole blocks:
  // with V % 8 != 0 the normalisers are given and no such job is posted.)
  __device__ bool sum_rows(const TreeJob& job, int wid, int lane) {
    const float c_hi = a.c_hi, c_lo = a.c_lo;
    const int n_rows = job.n_rows, total = job.total, xb = job.xb;
    uint32_t ph = job.ph;
    const int g = row_groups(n_rows, max_groups), group = wid % g, sub = wid / g, nsub = NCW / g;
    const bool reuse = total > n_stages;       // stages are filled more than once
    int st = 0, q = 0;
    for (int r = 0; r < n_rows; ++r) {
      const Slice sl(row0 + job.rows[r], a.V, v0, v1);
      const bool mine = r % g == group;
      float m_run = TV_NEG_INF;
      Comp acc;
      for (int x = 0; x < sl.n; x += kRow, ++q) {
        ph ^= 1u << st;
        if (mine || reuse) {
          if (!mbar_wait_warp(&full_bar[st], (ph >> st) & 1u)) return false;
        }
        if (mine) {
          const E* lb = reinterpret_cast<const E*>(ring + (size_t)st * kStageBytes);
          const int n = min(kRow, sl.n - x);
          const int hop = nsub * kTileElems;
          int t0 = sub * kTileElems;
          // two whole tiles at a time: their chains of dependent operations overlap
          for (; t0 + hop + kTileElems <= n; t0 += 2 * hop) {
            float v[2][8], t[2][8];
            lds_logits<L>(lb + t0 + lane * kChunk, v[0]);
            lds_logits<L>(lb + t0 + hop + lane * kChunk, v[1]);
            const float cm = fmaxf(max8(v[0]), max8(v[1]));
            if (cm > m_run) {
              if (m_run != TV_NEG_INF) {
                const float sc = L::exp_rel(m_run, cm, c_hi, c_lo);
                acc.s *= sc;
                acc.c *= sc;
              }
              m_run = cm;
            }
            exp8<L, false>(v[0], m_run, c_hi, c_lo, t[0]);
            exp8<L, false>(v[1], m_run, c_hi, c_lo, t[1]);
            acc.add(sum8(t[0]));
            acc.add(sum8(t[1]));
          }
          for (; t0 < n; t0 += hop) {
            const int e0 = t0 + lane * kChunk;
            if (e0 >= n) continue;
            float v[8], t[8];
            lds_logits<L>(lb + e0, v);
            const float cm = max8(v);
            if (cm > m_run) {
              if (m_run != TV_NEG_INF) {
                const float sc = L::exp_rel(m_run, cm, c_hi, c_lo);
                acc.s *= sc;
                acc.c *= sc;
              }
              m_run = cm;
            }
            exp8<L, false>(v, m_run, c_hi, c_lo, t);
            acc.add(sum8(t));
          }
        }
        end_chunk(q, total, st, lane);
      }
      if (mine) {
        const float wm = warp_max(m_run);
        const float part =
            (m_run == TV_NEG_INF) ? 0.f : acc.value() * L::exp_rel(m_run, wm, c_hi, c_lo);
        send(xb, (r * C + (int)rank) * nsub + sub, lane, wm, warp_sum(part));
      }
    }
    arrive_alone(xb, lane);
    return true;
  }

  // A rejection pass (kJobPass: the warp's sum, returned) or the tile sums of a
  // bonus draw.
  __device__ bool pair_or_leaf(const TreeJob& job, int wid, int lane, float& sum) {
    const float c_hi = a.c_hi, c_lo = a.c_lo;
    const int kind = job.kind, total = job.total;
    uint32_t ph = job.ph;
    const bool pair = is_pair(kind);
    const int per = pair ? kPair : kRow;
    const int nmask = job.nmask;
    const int* mt = mtok(job.mbuf);
    const float al = job.alpha1, be = job.beta, rm = job.rowmax;
    const Slice sl(row0 + job.node, a.V, v0, v1);
    const bool ragged = (a.V & 7) != 0;
    int st = job.slot > 0 ? job.slot * spc : 0, q = 0, mp = 0;
    Comp acc;
    for (int x = 0; x < sl.n; x += per, ++q) {
      if (total > 0) ph ^= 1u << st;           // filled by this job
      if (!mbar_wait_warp(&full_bar[st], (ph >> st) & 1u)) return false;
      const char* buf = ring + (size_t)st * kStageBytes;
      const E* lb = reinterpret_cast<const E*>(buf);
      const float* qb = reinterpret_cast<const float*>(buf + (size_t)kPair * kLB);
      const int n = min(per, sl.n - x);
      if (kind == kJobPass && !ragged && !removed_here(n, x, mt, nmask, wid)) {
        int t0 = wid * kTileElems;
        if (n >= t0 + (kTiles - 1) * kSweep + kTileElems) {   // all of the warp's tiles, whole
          float v[kTiles][8], t[kTiles][8];
#pragma unroll
          for (int k = 0; k < kTiles; ++k)
            lds_logits<L>(lb + t0 + k * kSweep + lane * kChunk, v[k]);
#pragma unroll
          for (int k = 0; k < kTiles; ++k)
            residual8<L, kExact>(v[k], qb + t0 + k * kSweep + lane * kChunk, rm, al, be, c_hi,
                                 c_lo, t[k]);
#pragma unroll
          for (int k = 0; k < kTiles; ++k) acc.add(sum8(t[k]));
        } else {
          for (; t0 < n; t0 += kSweep) {
            const int e0 = t0 + lane * kChunk;
            if (e0 < n) {
              float v[8], t[8];
              lds_logits<L>(lb + e0, v);
              residual8<L, kExact>(v, qb + e0, rm, al, be, c_hi, c_lo, t);
              acc.add(sum8(t));
            }
          }
        }
        end_chunk(q, total, st, lane);
        continue;
      }
      for (int t0 = wid * kTileElems; t0 < n; t0 += kSweep) {
        const int e0 = t0 + lane * kChunk;
        const bool valid = e0 < n;
        const int xg = v0 - sl.sh + x + e0;    // token of the lane's first element
        const int lo = sl.sh - (x + e0), hi = sl.n - (x + e0);
        const bool edge = ragged && valid && (lo > 0 || hi < 8);
        float v[8], t[8];
        stage_logits(lb, e0, valid, edge, lo, hi, v);
        if (kind == kJobBonusLeaf) {
          const float tm = warp_max(max8(v));
          exp8<L, !kExact>(v, tm, c_hi, c_lo, t);
#pragma unroll
          for (int e = 0; e < 8; ++e) t[e] = fmaxf(t[e], 0.f);
          zero_outside(edge, lo, hi, t);
          const float ts = warp_sum(valid ? sum8(t) : 0.f);
          if (lane == 0) {
            s.tsum[(x + t0) / kTileElems] = ts;
            s.tmax[(x + t0) / kTileElems] = tm;
          }
          continue;
        }
        if (valid) {
          residual8<L, kExact>(v, qb + e0, rm, al, be, c_hi, c_lo, t);
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) t[e] = 0.f;
        }
        zero_outside(edge, lo, hi, t);
        if (nmask > 0) {
          while (mp < nmask && mt[mp] < xg) ++mp;
          for (int mq = mp; mq < nmask && mt[mq] < xg + kChunk; ++mq) {
            const int off = mt[mq] - xg;
            if (!valid || off < lo || off >= hi) continue;   // (another slice's token)
            const float mv = (kind == kJobPass) ? 0.f : s.mask_val[mq];
#pragma unroll
            for (int e = 0; e < 8; ++e) if (e == off) t[e] = mv;
          }
        }
        if (kind == kJobPass) {
          if (valid) acc.add(sum8(t));
        } else {
          const float ts = warp_sum(valid ? sum8(t) : 0.f);
          if (lane == 0) s.tsum[(x + t0) / kTileElems] = ts;
        }
      }
      end_chunk(q, total, st, lane);
    }
    sum = acc.value();
    return true;
  }

  __device__ void consumer(int wid, int lane) {
    uint32_t jp = 0u;
    for (;;) {
      if (!mbar_wait_warp(job_bar, jp)) { fail(); return; }
      jp ^= 1u;
      const TreeJob& job = sh.job;
      const int kind = job.kind;
      if (kind == kJobDone) return;
      if (kind == kJobStats) {
        if (!sum_rows(job, wid, lane) || !finish_rows(job, wid, lane)) { fail(); return; }
        continue;
      }
      float sum;
      if (!pair_or_leaf(job, wid, lane, sum)) { fail(); return; }
      if (kind == kJobPass) {
        const int xb = job.xb;
        // once every CTA's control warp has all partials, the job is replaced:
        // nothing of it is read after this
        send(xb, (int)rank * NCW + wid, lane, warp_sum(sum), 0.f);
        arrive_alone(xb, lane);
        continue;
      }
      if (wid != 0) arrive_alone(job.xb, lane);
      __syncwarp();
      if (lane == 0) mbar_arrive(tile_bar);
      if (wid == 0 && !draw(job, lane)) { fail(); return; }
    }
  }

  // The rows' normalisers from all warps' partials (a row per warp, the same
  // order in every CTA), and M_b^(0) of their children.
  __device__ bool finish_rows(const TreeJob& job, int wid, int lane) {
    const float c_hi = a.c_hi, c_lo = a.c_lo;
    const int n_rows = job.n_rows, n = C * (NCW / row_groups(n_rows, max_groups));
    if (!exchanged(job.xb, job.xph) || !mbar_wait_warp(order_bar, 0u)) return false;
    for (int r = wid; r < n_rows; r += NCW) {
      const float2* x = xslots(job.xb) + r * n;
      float M = TV_NEG_INF;
      for (int k = lane; k < n; k += 32) M = fmaxf(M, x[k].x);
      M = warp_max(M);
      float S = 0.f;
      for (int k = lane; k < n; k += 32) {
        const float2 p = x[k];
        if (p.x != TV_NEG_INF) S += p.y * L::exp_rel(p.x, M, c_hi, c_lo);
      }
      S = warp_sum(S);
      const int node = job.rows[r];
      const double invs = 1.0 / (double)S;
      int j = s.first[node];
      for (int k = 0; k < lane && j >= 0; ++k) j = s.next[j];
      while (j >= 0) {
        set_child_mass(s, j, M, invs, a.c);
        for (int k = 0; k < 32 && j >= 0; ++k) j = s.next[j];
      }
      if (lane == 0) {
        s.rowm[node] = M;
        s.rows[node] = S;
        s.invs[node] = invs;
        if (!(S > 0.f)) atomicOr(&sh.ctl.bad, 64u);   // no finite logit in the row
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(stat_bar);
    return true;
  }

  // The bonus draw (warp 0 of every CTA): slice totals, crossing slice,
  // crossing tile, token.
  __device__ bool draw(const TreeJob& job, int lane) {
    const float c_hi = a.c_hi, c_lo = a.c_lo;
    const bool leaf = (job.kind == kJobBonusLeaf);
    const int node = job.node, R = a.N + 1;
    if (!mbar_wait_warp(tile_bar, 0u)) return false;
    const Slice sl(row0 + node, a.V, v0, v1);
    const int ntl = (sl.n + kTileElems - 1) / kTileElems;
    float Mc = 0.f;
    if (leaf) {
      float lm = TV_NEG_INF;
      for (int k = lane; k < ntl; k += 32) lm = fmaxf(lm, s.tmax[k]);
      Mc = warp_max(lm);
      for (int k = lane; k < ntl; k += 32)
        s.tsum[k] = (s.tmax[k] == TV_NEG_INF)
                        ? 0.f : s.tsum[k] * L::exp_rel(s.tmax[k], Mc, c_hi, c_lo);
      __syncwarp();
    }
    float Wc = 0.f;
    for (int k0 = 0; k0 < ntl; k0 += 32) {
      const float v = (k0 + lane < ntl) ? s.tsum[k0 + lane] : 0.f;
      Wc += warp_sum(v);
    }
    // every CTA learns every slice's (max, total)
    send(job.xb, (int)rank, lane, Mc, Wc);
    arrive_alone(job.xb, lane);
    if (!exchanged(job.xb, job.xph)) return false;
    const float2* x = xslots(job.xb);
    float scale = 1.f, target = 0.f, before = 0.f, W = 0.f;
    int owner = -1;
    float Mg = x[0].x;
    if (leaf)
      for (int rr = 1; rr < C; ++rr) Mg = fmaxf(Mg, x[rr].x);
    auto slice_scale = [&](int rr) -> float {
      return leaf ? ((x[rr].x == TV_NEG_INF) ? 0.f : L::exp_rel(x[rr].x, Mg, c_hi, c_lo)) : 1.f;
    };
    for (int rr = 0; rr < C; ++rr) W += x[rr].y * slice_scale(rr);
    target = u[R] * W;
    float acc0 = 0.f;
    for (int rr = 0; rr < C; ++rr) {
      const float wr = x[rr].y * slice_scale(rr);
      if (owner < 0 && target < acc0 + wr) { owner = rr; before = acc0; }
      acc0 += wr;
    }
    if (owner < 0) {   // rounding: the last slice with weight
      owner = C - 1;
      while (owner > 0 && !(x[owner].y > 0.f)) --owner;
      before = 0.f;
      for (int rr = 0; rr < owner; ++rr) before += x[rr].y * slice_scale(rr);
    }
    if ((uint32_t)owner != rank) return true;
    scale = slice_scale((int)rank);
    // local target in this slice's units
    const float lt = (scale > 0.f) ? (target - before) / scale : 0.f;
    int tile = -1;
    float tbase = 0.f, base = 0.f;
    for (int k0 = 0; k0 < ntl && tile < 0; k0 += 32) {
      float v = (k0 + lane < ntl) ? s.tsum[k0 + lane] : 0.f;
      const float own = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float w2 = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += w2;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, (k0 + lane < ntl) && (lt < base + v));
      if (hit) {
        const int l = __ffs(hit) - 1;
        tile = k0 + l;
        tbase = base + __shfl_sync(0xffffffffu, v - own, l);
      }
      base += __shfl_sync(0xffffffffu, v, 31);
    }
    if (tile < 0) {
      tile = ntl - 1;
      while (tile > 0 && !(s.tsum[tile] > 0.f)) --tile;
      float a0 = 0.f;
      for (int k = 0; k < tile; ++k) a0 += s.tsum[k];
      tbase = a0;
    }
    // element-level rescan of the crossing tile (global loads, L2-hot)
    const int g0 = tile * kTileElems + lane * kChunk;
    const int x0 = v0 - sl.sh + g0;
    const int lo = sl.sh - g0, hi = sl.n - g0;
    const size_t at = sl.base + (size_t)g0;
    float w[8];
    {
      float v[8];
      block_logits<L>(reinterpret_cast<const E*>(a.logits) + at, lo, hi, v);
      if (leaf) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          w[e] = (v[e] == TV_NEG_INF) ? 0.f
                                      : exp1(v[e], Mc);
      } else {
        float qv[8];
        block_probs(a.draft_probs + at, lo, hi, qv);
#pragma unroll
        for (int e = 0; e < 8; ++e)
          w[e] = (v[e] == TV_NEG_INF)
                     ? 0.f
                     : fmaxf(fmaf(job.alpha1,
                                  exp1(v[e], job.rowmax),
                                  -job.beta * qv[e]), 0.f);
        const int* mt = mtok(job.mbuf);
        for (int mq = 0; mq < job.nmask; ++mq) {
          const int off = mt[mq] - x0;
          if (off < lo || off >= hi) continue;
          const float mv = s.mask_val[mq];
#pragma unroll
          for (int e = 0; e < 8; ++e) if (e == off) w[e] = mv;
        }
      }
    }
    float pre[8];
    float run = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) { run += w[e]; pre[e] = run; }
    float v = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float w2 = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += w2;
    }
    const float lbase = tbase + (v - run);
    int found = 8;
#pragma unroll
    for (int e = 7; e >= 0; --e) if (e >= lo && lt < lbase + pre[e]) found = e;
    const unsigned hit = __ballot_sync(0xffffffffu, found < 8);
    // the draw's margin (kernel sums), in this slice's units, then relative to
    // the total
    float clo = lbase, chi = lbase;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (e == found) chi = lbase + pre[e];
      if (e + 1 == found) clo = lbase + pre[e];
    }
    const float my_margin = fminf(lt - clo, chi - lt) * scale / W;
    int yy;
    float bm = 0.f;
    if (hit) {
      const int l = __ffs(hit) - 1;
      yy = x0 - lane * kChunk + l * kChunk + __shfl_sync(0xffffffffu, found, l);
      bm = __shfl_sync(0xffffffffu, my_margin, l);
    } else {
      int last = -1;
#pragma unroll
      for (int e = 0; e < 8; ++e) if (w[e] > 0.f) last = x0 + e;
      const unsigned any = __ballot_sync(0xffffffffu, last >= 0);
      yy = any ? __shfl_sync(0xffffffffu, last, 31 - __clz(any)) : v1 - 1;
    }
    if (lane == 0) {
      a.out_bonus[b] = yy;
      if (a.out_margin) a.out_margin[2 * (size_t)b + 1] = bm;
    }
    return true;
  }

  // ----------------------------------------------------------- control --
  // What lane 0 of the control warp keeps of the ring: the parities of the
  // stages' latest fills, the stages whose latest fill was a fetch ahead that may
  // still be on its way, the resident slots, the node and slot of the latest
  // pair, jobs and exchanges so far.
  struct Ring {
    uint32_t ph = 0xffffffffu, coming = 0u;
    int n_slots = 0, node = -1, slot = 0, jobs = 0, xk = 0;
    __device__ __forceinline__ void took(uint32_t stages) { ph ^= stages; }
    // `total` chunks through a ring of n stages, from stage 0
    __device__ __forceinline__ void streamed(int total, int n) {
      for (; total >= n; total -= n) took((1u << n) - 1u);
      took((1u << total) - 1u);
    }
  };

  // Waits until every fetch ahead has landed: before a stage is filled again,
  // since a wait on a barrier's parity cannot tell the fill before the latest one
  // from it.
  __device__ bool settle(Ring& ring) const {
    for (; ring.coming != 0u; ring.coming &= ring.coming - 1u) {
      const int st = __ffs(ring.coming) - 1;
      if (!mbar_wait(&full_bar[st], (ring.ph >> st) & 1u)) return false;
    }
    return true;
  }

  // The slot of a pair: the one that holds it, or the one used longest ago
  // (other than `keep`).
  __device__ int find_slot(const Ring& ring, int node, int keep, bool& held) const {
    int old = -1;
    for (int k = 0; k < ring.n_slots; ++k) {
      if (sh.slot_node[k] == node) { held = true; return k; }
      if (k != keep && (old < 0 || sh.slot_used[k] < sh.slot_used[old])) old = k;
    }
    held = false;
    return old;
  }

  // Lane 0: completes the job's ring, slot and exchange fields and publishes it.
  // This stands between a pass's result and the next job's start, so the usual
  // case, a pass at the node of the latest one, looks nothing up.
  __device__ bool publish(const Job& j, int mbuf, Ring& ring) {
    TreeJob& t = sh.job;
    // the producer has copied the job before (the consumers have finished it)
    if (ring.jobs > 0 && !mbar_wait(ack_bar, (uint32_t)(ring.jobs - 1) & 1u)) return false;
    t.kind = j.kind;
    if (j.kind != kJobDone) {
      uint32_t bytes;
      int n_rows = 1, total = 0, slot = -1;
      t.ph = ring.ph;
      t.node = j.node;
      t.nmask = j.nmask;
      t.alpha1 = j.alpha1;
      t.beta = j.beta;
      t.rowmax = j.rowmax;
      t.mbuf = mbuf;
      t.xb = ring.xk & 1;
      t.xph = (ring.xk >> 1) & 1;
      if (is_pair(j.kind)) {
        bytes = (j.kind == kJobPass) ? (uint32_t)(C * NCW) * 8u : (uint32_t)C * 8u;
        if (ring.n_slots > 0 && ring.node == j.node) {
          slot = ring.slot;
        } else {
          bool held = false;
          if (ring.n_slots > 0) {
            slot = find_slot(ring, j.node, -1, held);
            sh.slot_node[slot] = j.node;
            sh.slot_used[slot] = ring.jobs + 1;
            ring.node = j.node;
            ring.slot = slot;
          }
          if (!held) {
            if (!settle(ring)) return false;
            total = chunks_of(Slice(row0 + j.node, a.V, v0, v1).n, kPair);
            if (slot >= 0) ring.took(((1u << total) - 1u) << (slot * spc));
            else ring.streamed(total, n_stages);
          }
        }
      } else {
        // target rows only: through the whole ring
        if (!settle(ring)) return false;
        for (int k = 0; k < ring.n_slots; ++k) sh.slot_node[k] = -1;
        ring.node = -1;
        if (j.kind == kJobStats) {
          n_rows = min(j.n_rows, min(kStatRows, 4 * max_groups));
          for (int r = 0; r < n_rows; ++r) {
            t.rows[r] = s.job_rows[r];
            total += chunks_of(Slice(row0 + s.job_rows[r], a.V, v0, v1).n, kRow);
          }
          bytes = (uint32_t)(n_rows * C * (NCW / row_groups(n_rows, max_groups))) * 8u;
        } else {
          total = chunks_of(Slice(row0 + j.node, a.V, v0, v1).n, kRow);
          bytes = (uint32_t)C * 8u;
        }
        ring.streamed(total, n_stages);
      }
      t.total = total;
      t.slot = slot;
      t.n_rows = n_rows;
      if (C > 1) mbar_arrive_expect_tx(&xbar[ring.xk & 1], bytes);
    }
    mbar_arrive(job_bar);
    ++ring.jobs;
    return true;
  }

  // Lane 0, while a pass at node i runs: fetches the pair of i's parent into
  // another slot, for the pass there that a rejection of i leads to.
  __device__ bool fetch_parent(Ring& ring) {
    const int i = ring.node;
    if (ring.n_slots < 2 || i <= 0 || a.token_level) return true;
    const int g = s.par[i];
    bool held;
    const int slot = find_slot(ring, g, ring.slot, held);
    if (held) return true;
    if (!settle(ring)) return false;
    const Slice sl(row0 + g, a.V, v0, v1);
    const int n = chunks_of(sl.n, kPair);
    for (int k = 0; k < n; ++k) fill(slot * spc + k, sl, k * kPair, true, elements());
    ring.coming = ((1u << n) - 1u) << (slot * spc);
    ring.took(ring.coming);
    sh.slot_node[slot] = g;
    sh.slot_used[slot] = ring.jobs + 1;
    return true;
  }

  __device__ void run_tree(int lane, Ring& ring) {
    Ctl& ctl = sh.ctl;
    Ahead& ah = sh.ahead;
    const bool ahead = a.token_level == 0;
    int mnext = 1;                       // next list of removed tokens
    uint32_t stat_ph = 0u;               // parity of stat_bar
    int ok = 1;
    if (lane == 0) {
      if (ctl.job.kind != kJobDone) advance(s, ctl, u, a.token_level != 0);
      ok = publish(ctl.job, 0, ring) ? 1 : 0;
      ah.ok = 0;
      if (ahead) prepare_ahead(s, ctl, ah, mtok(mnext), u);
    }
    if (!a.row_stats) {
      // the first job is a normaliser's (or a leaf's draw): the children's order
      // is needed only once it is done (before the first job: 64.4 -> 62.5 us at 16
      // chains of 8, 113.6 -> 111.8 us at 16 and 142.3 -> 141.2 us at 64 trees of 60
      // nodes, V = 32000)
      __syncwarp();
      if (sh.ctl.job.kind == kJobStats) {
        const int R = a.N + 1;
        for (int i = lane; i < R; i += 32) children_order(s, i);
        __syncwarp();
        for (int i = lane + 1; i < R; i += 32) child_order(s, i);
        __syncwarp();
      }
      if (lane == 0) mbar_arrive(order_bar);
    }
    for (;;) {
      __syncwarp();
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) { fail(); return; }
      const int kind = ctl.job.kind;
      if (kind == kJobDone) return;
      const int xk = ring.xk;            // (the same in every lane)
      const bool got = kind == kJobStats ? mbar_wait_warp(stat_bar, stat_ph)
                                         : exchanged(xk & 1, (uint32_t)(xk >> 1) & 1u);
      if (!got) { fail(); return; }
      float S = 0.f;
      if (kind == kJobPass) {
        const float2* x = xslots(xk & 1);
        for (int k = lane; k < C * NCW; k += 32) S += x[k].x;
        S = warp_sum(S);
      }
      ++ring.xk;
      if (kind == kJobStats) stat_ph ^= 1u;
      if (kind == kJobPass && ah.ok && S > 0.f) {
        // the next step was worked out while the pass ran: decide, publish, then
        // update the state (the same values in every lane)
        const double Sd = (double)S * ctl.s_unit + ah.pm, D = Sd + ah.omp;
        bool accept = false, first = true;
        if (lane == 0) {
          Job jf;
          first = job_ahead(s, ah, Sd, D, jf, accept);
          if (first) ok = publish(jf, mnext, ring) ? 1 : 0;
        }
        __syncwarp();
        // 1 / D, 1 / S and S / D in lanes 0, 1 and 2: a float64 division takes as
        // long for one lane as for three
        const double quot = (lane == 2 ? Sd : 1.0) / (lane == 1 ? Sd : D);
        const double inv_s = __shfl_sync(0xffffffffu, quot, 1);
        const double p_new = __shfl_sync(0xffffffffu, quot, 2);
        if (lane == 0) {
          ctl.S = S;
          control_step_ahead(s, ctl, ah, accept, D, quot, inv_s, p_new);
          if (!first) ok = publish(ctl.job, 0, ring) ? 1 : 0;
          else mnext = 3 - mnext;             // that list is in use now
          prepare_ahead(s, ctl, ah, mtok(mnext), u);
          if (ctl.job.kind == kJobPass && !fetch_parent(ring)) ok = 0;
        }
      } else if (lane == 0) {
        if (kind == kJobBonusLeaf || kind == kJobBonusRes) {
          ctl.job.kind = kJobDone;
        } else {
          if (kind == kJobPass) ctl.S = S;
          if (*(volatile uint32_t*)&ctl.bad & (32u | 64u)) ctl.job.kind = kJobDone;
          else advance(s, ctl, u, a.token_level != 0);
        }
        ok = publish(ctl.job, 0, ring) ? 1 : 0;
        ah.ok = 0;
        if (ahead) prepare_ahead(s, ctl, ah, mtok(mnext), u);
        if (ctl.job.kind == kJobPass && !fetch_parent(ring)) ok = 0;
      }
    }
  }

  __device__ void control(int lane) {
    if (lane < kTreeMaxSlots) { sh.slot_node[lane] = -1; sh.slot_used[lane] = 0; }
    __syncwarp();
    Ring ring;
    // resident row pairs the ring has room for (0: pairs are streamed)
    ring.n_slots = min(n_stages / spc, kTreeMaxSlots);
    run_tree(lane, ring);
    // copies in flight land before the CTA may exit: fetches ahead here, those of
    // a job the consumers gave up on in produce()
    if (lane == 0 && !settle(ring)) fail();
    __syncwarp();
  }

  // Writes the tree's outputs (control warp of rank 0).
  __device__ void outputs(int lane) {
    const int R = a.N + 1, N = a.N;
    const Ctl& ctl = sh.ctl;
    const bool ok = (ctl.bad & (15u | 32u | 64u)) == 0u;
    for (int k = lane; k < N; k += 32) a.out_path[(size_t)b * N + k] = -1;
    if (a.out_node_p)
      for (int i = lane; i < R; i += 32)
        a.out_node_p[row0 + i] = ok ? s.dbgp[i] : __int_as_float(0x7fc00000);
    __syncwarp();
    if (lane != 0) return;
    const int acc_node = ok ? ctl.accepted : -1;
    if (acc_node >= 0) {
      int depth = 0;
      for (int j = acc_node; j != 0; j = s.par[j]) ++depth;
      int k = depth - 1;
      for (int j = acc_node; j != 0; j = s.par[j]) a.out_path[(size_t)b * N + (k--)] = j;
      a.out_accept_len[b] = depth;
    } else {
      a.out_accept_len[b] = -1;
      a.out_bonus[b] = -1;
    }
    if (a.out_stats) {
      int distinct = 0;
      for (int i = 0; i < R; ++i) distinct += (s.npass[i] > 0);
      int normalised = 0;
      for (int i = 0; i < R; ++i) normalised += (s.rows[i] > 0.f);
      int32_t* o = a.out_stats + (size_t)b * 5;
      o[0] = ok ? ctl.n_tests : 0;
      o[1] = ok ? ctl.n_passes : 0;
      o[2] = ok ? distinct : 0;
      o[3] = (acc_node >= 0 && s.first[acc_node] < 0) ? 1 : 0;
      o[4] = (ok && !a.stats_given) ? normalised : 0;   // rows this call streamed
    }
    if (a.out_margin) {
      // the bonus margin was written by the CTA that drew the bonus
      const float nan = __int_as_float(0x7fc00000);
      a.out_margin[2 * (size_t)b] = acc_node >= 0 ? test_margin_serial(s.dbgp, u, R) : nan;
      if (acc_node < 0) a.out_margin[2 * (size_t)b + 1] = nan;
    }
    if (ctl.bad) atomicOr(a.status, ctl.bad);
  }
};

template <typename L, int NCW, bool kExact>
__global__ void __launch_bounds__(TreeCta<L, NCW, kExact>::kThreads, 16 / NCW)
    tv_tree_kernel(const __grid_constant__ TravArgs args, int C, int n_stages) {
  using T = TreeCta<L, NCW, kExact>;
  extern __shared__ __align__(128) char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kTreeMaxStages];
  __shared__ __align__(8) uint64_t empty_bar[kTreeMaxStages];
  __shared__ __align__(8) uint64_t xbar[2];
  __shared__ __align__(8) uint64_t job_bar, ack_bar, stat_bar, tile_bar, order_bar;
  __shared__ TreeShared sh;

  const int R = args.N + 1, V = args.V;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  T t(args, sh);
  t.C = C;
  t.n_stages = n_stages;
  t.rank = (C > 1) ? cluster_rank() : 0u;
  t.b = blockIdx.x / C;
  const int SL = slice_len(V, C);
  t.v0 = min((int)t.rank * SL, V);
  t.v1 = min(t.v0 + SL, V);
  t.row0 = (size_t)t.b * R;
  t.ring = smem_raw;
  t.xs = reinterpret_cast<float2*>(smem_raw + (size_t)n_stages * T::kStageBytes);
  t.spc = max(1, chunks_of(t.v1 - t.v0 + 7, T::kPair));
  t.max_groups = max(1, min(NCW, n_stages / max(1, chunks_of(SL + 7, T::kRow))));
  char* tree_base = reinterpret_cast<char*>(t.xs + 2 * exchange_slots(C, NCW));
  t.s = carve_tree_nt(tree_base, R, tree_tiles(V, C));
  t.mtok_ahead = reinterpret_cast<int*>(
      tree_base + ((tree_smem_bytes_nt(R, tree_tiles(V, C)) + 15) & ~(size_t)15));
  t.u = reinterpret_cast<float*>(t.mtok_ahead + 2 * R);
  t.full_bar = full_bar;
  t.empty_bar = empty_bar;
  t.xbar = xbar;
  t.job_bar = &job_bar;
  t.ack_bar = &ack_bar;
  t.stat_bar = &stat_bar;
  t.tile_bar = &tile_bar;
  t.order_bar = &order_bar;
  const TreeSmem& s = t.s;
  Ctl& ctl = sh.ctl;
  const typename L::elem* logits = reinterpret_cast<const typename L::elem*>(args.logits);

  // ---- set-up: barriers, tree structure, validation, gathers ----
  if (tid == 0) {
    for (int k = 0; k < n_stages; ++k) {
      mbar_init(&full_bar[k], 1);
      mbar_init(&empty_bar[k], NCW);
    }
    mbar_init(&xbar[0], C > 1 ? 1 : NCW);
    mbar_init(&xbar[1], C > 1 ? 1 : NCW);
    mbar_init(&job_bar, 1);
    mbar_init(&ack_bar, 1);
    mbar_init(&stat_bar, NCW);
    mbar_init(&tile_bar, NCW);
    mbar_init(&order_bar, 1);
    fence_mbar_init();
    ctl.bad = 0u;
    ctl.accepted = -1;
    ctl.node = 0;
    ctl.pending = -1;
    ctl.masked_sum = 0.0;
    ctl.s_unit = 1.0;
    ctl.n_tests = ctl.n_passes = 0;
    ctl.job.kind = 0;
  }
  for (int i = tid; i <= R; i += T::kThreads)
    t.u[i] = args.uniforms[t.row0 + t.b + i];
  for (int i = tid; i < R; i += T::kThreads) {
    s.par[i] = args.parents[t.row0 + i];
    s.tok[i] = args.tokens[t.row0 + i];
    s.first[i] = 0x7fffffff;
    s.npass[i] = 0;
    s.state[i] = kAlive;
    s.a[i] = 1.0;
    s.b[i] = 0.0;
    s.m[i] = 0.0;
    s.p[i] = 0.0;
    s.rows[i] = 0.f;
    s.dbgp[i] = __int_as_float(0x7fc00000);
  }
  __syncthreads();
  {
    uint32_t bad = 0u;
    for (int i = tid; i < R; i += T::kThreads) {
      const int p = s.par[i];
      if (i == 0) {
        if (p != -1) bad |= 1u;
      } else {
        if (p < 0 || p >= i) bad |= 1u;
        else atomicMin(&s.first[p], i);
        const int tk = s.tok[i];
        if (tk < 0 || tk >= V) bad |= 2u;
      }
    }
    if (bad) atomicOr(&ctl.bad, bad);
  }
  __syncthreads();
  if (ctl.bad == 0u) {
    uint32_t bad = 0u;
    for (int i = tid; i < R; i += T::kThreads) {
      if (s.first[i] == 0x7fffffff) s.first[i] = -1;
      int nx = -1;
      if (i > 0) {
        const int p = s.par[i], tk = s.tok[i];
        const size_t prow = (t.row0 + p) * (size_t)V;
        const float gl = L::at(logits + prow, tk);      // (in flight during the search)
        const float gq = __ldg(args.draft_probs + prow + tk);
        for (int j = i + 1; j < R; ++j) {
          if (s.par[j] != p) continue;
          if (nx < 0) nx = j;
          if (s.tok[j] == tk) bad |= 4u;
        }
        s.gl[i] = gl;
        s.gq[i] = gq;
        if (!(gq > 0.f)) bad |= 8u;
      }
      s.next[i] = nx;
    }
    if (bad) atomicOr(&ctl.bad, bad);
  }
  __syncthreads();
  if (args.row_stats) {
    // launched as a dependent of the kernel that works them out: it has ended
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // given normalisers (from the LM head's epilogue, or the two-kernel
    // path's): every internal row is normalised up front and no normaliser job
    // is ever posted.  (Otherwise the control warp works out the children's order
    // while the first normaliser job runs.)
    if (ctl.bad == 0u) {
      uint32_t bad = 0u;
      for (int i = tid; i < R; i += T::kThreads) {
        if (s.first[i] < 0) continue;
        children_order(s, i);
        const float2 st = args.row_stats[t.row0 + i];
        s.rowm[i] = st.x;
        s.rows[i] = st.y;
        s.invs[i] = 1.0 / (double)st.y;
        if (!(st.y > 0.f)) bad |= 64u;
      }
      if (bad) atomicOr(&ctl.bad, bad);
    }
    __syncthreads();
    if (ctl.bad == 0u)
      for (int i = tid + 1; i < R; i += T::kThreads) {
        child_order(s, i);
        set_child_mass(s, i, s.rowm[s.par[i]], s.invs[s.par[i]], args.c);
      }
    __syncthreads();
  }
  if (tid == 0) {
    if (ctl.bad == 0u) s.p[0] = 1.0;
    else ctl.job.kind = kJobDone;
  }
  if (C > 1) cluster_sync_all();   // peers' barriers initialised before any remote store
  else __syncthreads();
  if (wid < NCW) {
    t.consumer(wid, lane);
  } else if (wid == NCW) {
    if (lane == 0 && !t.produce()) t.fail();
  } else {
    t.control(lane);
  }
  __syncthreads();                 // (a role that gave up has raised ctl.bad)
  if (t.rank == 0 && wid == NCW + 1) t.outputs(lane);
  if (C > 1) cluster_sync_all();   // no CTA leaves while a peer may still write to it
}

}  // namespace fused
}  // namespace tvk

// --------------------------------------------------------------- launcher --

namespace {

constexpr int kStaticBytes = 1536;   // at least the kernel's static shared memory

size_t tree_cta_bytes(int ncw, int lb, int C, int stages, int R, int V) {
  using namespace tvk::fused;
  return (size_t)stages * tree_stage_bytes(ncw, lb) + (size_t)2 * exchange_slots(C, ncw) * 8 +
         ((tree_smem_bytes_nt(R, tree_tiles(V, C)) + 15) & ~(size_t)15) + (size_t)R * 12 + 4;
}

// Ring stages that fit when `per_sm` CTAs share an SM's shared memory.
int stages_for(int ncw, int lb, int C, int per_sm, int R, int V, int smem_per_sm,
               int smem_per_block) {
  using namespace tvk::fused;
  const long reserve = 1024 + kStaticBytes;   // (1024: the system's own, per CTA)
  long per_cta = (long)smem_per_sm / per_sm - reserve;
  if (per_cta > smem_per_block - kStaticBytes) per_cta = smem_per_block - kStaticBytes;
  const long st = (per_cta - (long)tree_cta_bytes(ncw, lb, C, 0, R, V)) /
                  tree_stage_bytes(ncw, lb);
  return (int)(st > kTreeMaxStages ? kTreeMaxStages : st);
}

}  // namespace

FusedPlan tv_fused_plan(int batch, int R, int V, int logit_bytes, const TreeDevice& dev,
                        int force_ncw, int force_c, int force_stages) {
  using namespace tvk::fused;
  FusedPlan p;
  // (the batches below are those of 152 SMs)
  const long B = (long)batch * 152 / dev.sm_count;
  // Few trees: as many SMs per tree as keep all trees in one wave (152 SMs, two
  // CTAs of 8 consumer warps or one of 16 on each; clusters do not cross a GPC,
  // so about 8 clusters of 16 whole SMs fit), down to slices of 1000 tokens, below
  // which a job is all latency.  Measured (us; 60-node trees; ncw x C):
  //   V = 262144, B = 1: 16x16 71, 8x16 82, 16x8 94, 8x8 109; B = 4: 92, 106, 126, 144
  //   V = 151936, B = 1: 8x16 79, 16x16 80, 16x8 93, 8x8 101
  //   V = 128256, B = 1: 8x16 68, 16x16 70, 16x8 82, 8x8 82; B = 4: 98, 102, 118, 120
  //   V = 128256, B = 16: 8x16 128, 16x8 144, 8x8 147, 4x8 194, 16x16 207
  //   V = 128256, B = 48: 4x8 215, 8x4 218, 16x4 220, 8x8 221; B = 64: 8x4 239, 4x8
  //   240, 8x8 287; B = 128: 8x2 419, 8x4 424, 4x4 429
  //   V = 262144, B = 32: 8x8 255, 4x8 341, 16x4 346, 8x4 364
  //   V = 32000, B = 1: 8x16 56, 8x8 57, 4x8 58; B = 16: 4x8 101, 8x8 102, 8x16 106
  //   V = 32000, B = 64: 8x4 149, 4x8 154, 8x8 160; B = 128: 4x4 191, 8x2 192, 8x4 212
  //   V = 32000, B = 200: 8x2 230, 4x4 255, 4x2 280; B = 256: 4x2 250, 8x1 260, 8x2 261;
  //   B = 512: 4x2 386, 8x1 388, 8x2 399; B = 1024: 4x2 661, 8x1 662, 4x1 727, 8x2 731
  //   V = 16384, B = 300: 4x2 195, 8x1 200, 8x2 232; B = 1024: 8x1 470, 4x1 479
  //   V = 4000, B = 512: 4x1 183, 8x1 235; V = 8000, B = 1024 (26 nodes): 4x1 258, 8x1 308
  // (16 consumer warps pay from between V = 151936 and 262144 on; from 98304, where they
  // are taken, to there they are 1 to 4 % behind)
  int ncw = 8, C = 1;
  if (V > 98304 && B <= 4) ncw = 16, C = 16;
  else if (B <= 8 || (V > 98304 && B <= 16)) C = 16;
  else if (B <= 32) C = 8;
  else if (B <= 76) C = 4;
  else if (B <= 224) C = 2;
  else if (B <= 320 || (B <= 512 && V > 20000)) ncw = 4, C = 2;
  else if (V <= 12288) ncw = 4;
  while (C > 1 && V / C < 1000) C /= 2;
  while (C < 8 && tree_tiles(V, C) * 8 > 32768) C *= 2;   // bonus tiles' shared memory
  C = std::min(C, dev.max_cluster);
  if (force_ncw == 4 || force_ncw == 8 || force_ncw == 16) ncw = force_ncw;
  if (force_c == 1 || force_c == 2 || force_c == 4 || force_c == 8 || force_c == 16)
    C = std::min(force_c, dev.max_cluster);
  auto fit = [&] {
    int st = 0;
    for (int per_sm = 16 / ncw; per_sm > 0 && st < 3; --per_sm)
      st = stages_for(ncw, logit_bytes, C, per_sm, R, V, dev.smem_per_sm, dev.smem_per_block);
    return st;
  };
  int stages = fit();
  // the largest trees of the longest rows (from 1016 nodes of 4.0 million tokens, fp32):
  // shorter slices, whose bonus tiles leave room for the ring
  while (stages < 2 && C < 8 && C < dev.max_cluster) {
    C *= 2;
    stages = fit();
  }
  if (force_stages >= 2 && force_stages <= kTreeMaxStages && force_stages < stages)
    stages = force_stages;
  p.ncw = ncw;
  p.C = C;
  p.stages = stages;
  p.smem = stages >= 0 ? tree_cta_bytes(ncw, logit_bytes, C, stages, R, V) : 0;
  p.smem_most = (size_t)(dev.smem_per_block - kStaticBytes);
  p.ok = stages >= 2 && p.smem <= p.smem_most;
  return p;
}

namespace {

template <typename L, int NCW, bool kExact>
cudaError_t launch_one(const TravArgs& a, const FusedPlan& plan, cudaStream_t stream,
                       bool dependent) {
  auto k = tvk::fused::tv_tree_kernel<L, NCW, kExact>;
  // (the kernel's limit, the same at every launch: another thread may be about to launch
  // with more shared memory than this plan has)
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)plan.smem_most);
  if (e != cudaSuccess) return e;
  if (plan.C > 8) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.B * plan.C), 1, 1);
  cfg.blockDim = dim3(tvk::fused::TreeCta<L, NCW, kExact>::kThreads, 1, 1);
  cfg.dynamicSmemBytes = plan.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  unsigned n = 0;
  if (plan.C > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)plan.C;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  if (dependent) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, k, a, plan.C, plan.stages);
}

template <typename L, bool kExact>
cudaError_t launch_ncw(const TravArgs& a, const FusedPlan& plan, cudaStream_t stream,
                       bool dependent) {
  if (plan.ncw == 16) return launch_one<L, 16, kExact>(a, plan, stream, dependent);
  if (plan.ncw == 8) return launch_one<L, 8, kExact>(a, plan, stream, dependent);
  return launch_one<L, 4, kExact>(a, plan, stream, dependent);
}

}  // namespace

// The largest cluster of CTAs that fill an SM each, so that one of any plan's shape
// fits: 16 CTAs is more than a device has to hold (their SMs must share a GPC), and a
// device with few SMs may not hold 8 either.
bool tv_tree_device(int device, TreeDevice* out) {
  constexpr int kDevices = 64;
  static std::mutex mutex;
  static TreeDevice known[kDevices];
  if (device < 0 || device >= kDevices) return false;
  std::lock_guard<std::mutex> lock(mutex);
  TreeDevice& d = known[device];
  if (d.sm_count == 0) {
    using T = tvk::fused::TreeCta<tvk::Bf16Logits, 16, false>;
    auto k = tvk::fused::tv_tree_kernel<tvk::Bf16Logits, 16, false>;
    TreeDevice q;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaDeviceGetAttribute(&q.smem_per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor,
                               device) != cudaSuccess ||
        cudaDeviceGetAttribute(&q.smem_per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin,
                               device) != cudaSuccess)
      return false;
    const int smem = q.smem_per_block - kStaticBytes;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
      return false;
    for (int C = 16; C > 1; C /= 2) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)C, 1, 1);
      cfg.blockDim = dim3(T::kThreads, 1, 1);
      cfg.dynamicSmemBytes = (size_t)smem;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = (unsigned)C;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int active = 0;
      if (cudaOccupancyMaxActiveClusters(&active, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        active = 0;
      }
      if (active > 0) {
        q.max_cluster = C;
        break;
      }
    }
    q.sm_count = sms;
    d = q;
  }
  *out = d;
  return true;
}

int tv_launch_tree(const TravArgs& a, int logit_is_bf16, const FusedPlan& plan,
                   cudaStream_t stream, bool dependent) {
  // (fp32 logits have one exponential: the two forms are the same kernel)
  const cudaError_t e =
      !logit_is_bf16
          ? launch_ncw<tvk::F32Logits, false>(a, plan, stream, dependent)
          : (a.exact_exp ? launch_ncw<tvk::Bf16Logits, true>(a, plan, stream, dependent)
                         : launch_ncw<tvk::Bf16Logits, false>(a, plan, stream, dependent));
  if (e == cudaSuccess) return 0;
  cudaGetLastError();
  return -5;
}

int tv_launch_fused(const TravArgs& a, int logit_is_bf16, const FusedPlan& plan,
                    cudaStream_t stream, cudaEvent_t* ev) {
  if (!plan.ok) return -3;
  if (ev) {
    for (int k = 0; k < 3; ++k)
      if (cudaEventRecord(ev[k], stream) != cudaSuccess) return -5;
  }
  if (tv_launch_tree(a, logit_is_bf16, plan, stream, false) != 0) return -5;
  if (ev && cudaEventRecord(ev[3], stream) != cudaSuccess) return -5;
  return 0;
}
