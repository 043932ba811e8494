// tv_control.cuh -- per-tree state and the serial control of Algorithm 3
// (§3.1), shared by the fused kernels.
//
// The tree's state lives in the shared memory of the CTA that owns it; thread
// 0 advances the traversal (control_step) until it needs vocabulary-wide work
// and describes that work as a Job: normalisers of a list of rows, one
// rejection pass (Eqs. (1)/(3)), or the bonus draw.  Scalars are float64 (see
// children_mb0 and the parity notes of the repository's design document).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "tv_device.cuh"

namespace tvk {
namespace fused {

constexpr int kTileElems = 256;       // one warp x 8 elements

enum : int { kJobStats = 1, kJobPass = 2, kJobBonusLeaf = 3, kJobBonusRes = 4, kJobDone = 5 };
enum : uint8_t { kAlive = 0, kRejected = 1, kPruned = 2 };

struct Job {
  int kind;
  int n_rows;        // rows listed in job_rows (kJobStats), else 1
  int node;          // row of kJobPass / bonus jobs
  int nmask;         // removed tokens of that row (sorted in mask_tok / mask_val)
  float alpha1;      // kJobPass: coefficient of e(x); bonus residual: a / s
  float beta;        // kJobPass: coefficient of q(x); bonus residual: b
  float rowmax;      // row max used by e(x)
};

struct Ctl {
  Job job;
  uint32_t bad;        // TV_STATUS_* bits
  int accepted;        // accepted node (-1: invalid tree)
  float S;             // result of the last pass, in the units of its job:
  double s_unit;       // x s_unit is the sum of Eqs. (1)/(3) (job_ahead)
  float bmargin;       // margin of the bonus draw (out_margin[b][1])
  // serial control state (thread 0)
  int node;
  int pending;         // child whose rejection the running pass serves
  double masked_sum;
  int n_tests, n_passes;
};

// Per node i: rate p, (a, b) of its residual, normaliser (rowm, rows, invs =
// 1 / rows).  Per child c: m the stored mass once removed, mb0 and zq / invZ
// (child_order).
struct TreeSmem {
  double *p, *a, *b, *invZ, *m, *mb0, *zq, *invs;
  int32_t *par, *tok, *first, *next, *npass, *mask_tok, *job_rows;
  float *gl, *gq, *rowm, *rows, *dbgp, *mask_val, *tsum, *tmax;
  uint8_t* state;
};

__host__ __device__ inline int slice_len(int V, int C) {
  int per = (V + C - 1) / C;
  return (per + kChunk - 1) / kChunk * kChunk;
}

// Bonus tiles of a cluster CTA's slice (a slice may start inside an 8-element
// block, so up to 7 elements more).
__host__ __device__ inline int tree_tiles(int V, int C) {
  return (slice_len(V, C) + kChunk - 1 + kTileElems - 1) / kTileElems;
}

// Shared memory of one tree's state with `nt` bonus tiles.
__host__ __device__ inline size_t tree_smem_bytes_nt(int R, int nt) {
  return (size_t)R * (8 * 8 + 7 * 4 + 6 * 4 + 1) + (size_t)nt * 8 + 64;
}


__device__ __forceinline__ TreeSmem carve_tree_nt(char* base, int R, int nt) {
  TreeSmem s;
  double* dp = reinterpret_cast<double*>(base);
  s.p = dp; dp += R;
  s.a = dp; dp += R;
  s.b = dp; dp += R;
  s.invZ = dp; dp += R;
  s.m = dp; dp += R;
  s.mb0 = dp; dp += R;
  s.zq = dp; dp += R;
  s.invs = dp; dp += R;
  int32_t* ip = reinterpret_cast<int32_t*>(dp);
  s.par = ip; ip += R;
  s.tok = ip; ip += R;
  s.first = ip; ip += R;
  s.next = ip; ip += R;
  s.npass = ip; ip += R;
  s.mask_tok = ip; ip += R;
  s.job_rows = ip; ip += R;
  float* fp = reinterpret_cast<float*>(ip);
  s.gl = fp; fp += R;
  s.gq = fp; fp += R;
  s.rowm = fp; fp += R;
  s.rows = fp; fp += R;
  s.dbgp = fp; fp += R;
  s.mask_val = fp; fp += R;
  s.tsum = fp; fp += nt;
  s.tmax = fp; fp += nt;
  s.state = reinterpret_cast<uint8_t*>(fp);
  return s;
}

// ------------------------------------------------------------ control ----

__device__ __forceinline__ int first_alive_child(const TreeSmem& s, int i) {
  int j = s.first[i];
  while (j >= 0 && s.state[j] != kAlive) j = s.next[j];
  return j;
}

// A node's children are removed in index order (the traversal always tries the
// first remaining one), so Z_i when child c's turn comes is 1 less the draft
// masses of the children before it, known from the start: s.invZ[c] = 1 / Z (0
// if nothing is left) and s.zq[c] = Z / M_s^(0)(x_c).  First each node lists Z
// for its children, then (after a barrier) each child divides.
__device__ __forceinline__ void children_order(const TreeSmem& s, int i) {
  double Z = 1.0;
  for (int j = s.first[i]; j >= 0; j = s.next[j]) {
    s.invZ[j] = Z;
    Z -= (double)s.gq[j];
  }
}

__device__ __forceinline__ void child_order(const TreeSmem& s, int c) {
  const double Z = s.invZ[c];
  s.zq[c] = Z / (double)s.gq[c];
  s.invZ[c] = Z > 0.0 ? 1.0 / Z : 0.0;
}

// s.mb0[c] holds M_b^(0)(x_c | X^i) of child c of node i, in float64,
// exp2((l_i(x_c) - m_i) log2(e) / T) / s_i, computed as soon as row i's
// normaliser is known (a residual a M_b(x) - b M_s(x) of a sibling can cancel by
// orders of magnitude, so this single value must not carry a float32 rounding).
// s.p[c] holds M_b^(0)(x_c) / M_s^(0)(x_c) from then until the traversal reaches
// c, so that descending through nodes without a rejection yet costs one
// product per level (a dependent float64 operation takes 64 cycles here).
__device__ __forceinline__ void set_child_mass(const TreeSmem& s, int c, float rowmax,
                                               double inv_sum, double cd) {
  const double mb = exp2(((double)s.gl[c] - (double)rowmax) * cd) * inv_sum;
  s.mb0[c] = mb;
  s.p[c] = mb * s.zq[c];   // (only a first child, whose Z is 1, is reached this way)
}

// min(p_i M_b(x_c) / M_s(x_c), 1) from i's current state, with
// M_s(x_c) = q_c / Z_i; false if nothing of the draft support is left.
__device__ __forceinline__ bool child_rate(const TreeSmem& s, int i, int c, double* out) {
  if (s.npass[i] == 0) {   // the original rows: a = 1, b = 0, Z = 1
    *out = fmin(s.p[i] * s.p[c], 1.0);
    return true;
  }
  const double q = (double)s.gq[c];
  const double mb = fmax(s.a[i] * s.mb0[c] - s.b[i] * q, 0.0);
  if (!(s.invZ[c] > 0.0)) return false;
  *out = fmin(s.p[i] * mb * s.zq[c], 1.0);
  return true;
}

// Tokens of the children of node i removed before c (those in front of it),
// ascending, to list; returns how many.
__device__ inline int removed_tokens(const TreeSmem& s, int i, int c, int* list) {
  int n = 0;
  for (int j = s.first[i]; j != c; j = s.next[j]) {
    const int t = s.tok[j];
    int k = n;
    while (k > 0 && list[k - 1] > t) {
      list[k] = list[k - 1];
      --k;
    }
    list[k] = t;
    ++n;
  }
  return n;
}

// The stored masses of the children of node i removed before c.
__device__ inline double removed_mass(const TreeSmem& s, int i, int c) {
  double sum = 0.0;
  for (int j = s.first[i]; j != c; j = s.next[j]) sum += s.m[j];
  return sum;
}

__device__ inline void post_pass(const TreeSmem& s, Ctl& ctl, int i, int c) {
  ctl.pending = c;
  ctl.s_unit = 1.0;
  const double p = s.p[i];
  ctl.job.kind = kJobPass;
  ctl.job.n_rows = 1;
  ctl.job.node = i;
  ctl.job.alpha1 = (float)(p * s.a[i] * s.invs[i]);
  ctl.job.beta = (float)(p * s.b[i] + s.invZ[c]);
  ctl.job.rowmax = s.rowm[i];
  ctl.job.nmask = removed_tokens(s, i, c, s.mask_tok);
  ctl.masked_sum = removed_mass(s, i, c);
  ctl.n_passes++;
  s.npass[i]++;
}

__device__ inline void apply_rejection(const TreeSmem& s, Ctl& ctl, int i, int c) {
  const double p = s.p[i], a = s.a[i], b = s.b[i];
  const double S = (double)ctl.S * ctl.s_unit + p * ctl.masked_sum;
  const double alpha = p * a;
  const double beta = p * b + s.invZ[c];
  const double mb0 = s.mb0[c];
  const double q0 = (double)s.gq[c];
  if (S > 0.0) {
    const double invS = 1.0 / S;
    const double na = alpha * invS, nb = beta * invS, scale = p * invS;
    for (int j = s.first[i]; j != c; j = s.next[j]) s.m[j] *= scale;
    s.m[c] = fmax(na * mb0 - nb * q0, 0.0);
    s.a[i] = na;
    s.b[i] = nb;
    s.p[i] = S / (S + (1.0 - p));
  } else {
    ctl.bad |= 16u;
    s.m[c] = fmax(a * mb0 - b * q0, 0.0);
    s.p[i] = (p == 1.0) ? 1.0 : 0.0;
  }
}

// Lists the not-yet-normalised internal nodes of the chain that starts at
// `node` (following first remaining children); returns how many.
__device__ inline int chain_needing_stats(const TreeSmem& s, int node) {
  int n = 0;
  for (int i = node; i >= 0; i = first_alive_child(s, i)) {
    if (s.first[i] < 0) break;            // a leaf: no row statistics needed
    if (!(s.rows[i] > 0.f)) s.job_rows[n++] = i;
  }
  return n;
}

__device__ inline void post_bonus(const TreeSmem& s, Ctl& ctl, int a) {
  ctl.accepted = a;
  ctl.job.node = a;
  ctl.job.n_rows = 1;
  if (s.first[a] < 0) {
    ctl.job.kind = kJobBonusLeaf;
    ctl.job.nmask = 0;
    return;
  }
  ctl.job.kind = kJobBonusRes;
  ctl.job.alpha1 = (float)(s.a[a] * s.invs[a]);
  ctl.job.beta = (float)s.b[a];
  ctl.job.rowmax = s.rowm[a];
  int n = 0;
  for (int j = s.first[a]; j >= 0; j = s.next[j]) {
    const int t = s.tok[j];
    int k = n;
    while (k > 0 && s.mask_tok[k - 1] > t) {
      s.mask_tok[k] = s.mask_tok[k - 1];
      s.mask_val[k] = s.mask_val[k - 1];
      --k;
    }
    s.mask_tok[k] = t;
    s.mask_val[k] = (float)s.m[j];
    ++n;
  }
  ctl.job.nmask = n;
}

// ---------------------------------------------------- deciding ahead ----
//
// While the pass that rejects child c of node i runs, most of the next step is
// already fixed.  With
//   D = S + (1 - p_i),   alpha = p_i a_i,  beta = p_i b_i + 1/Z_i,  Z' = Z_i - q(c)
// Eqs. (1)-(3) give a child c2 the rate min(X / D, 1),
//   X = [alpha M_b0(c2) - beta q(c2)]_+ Z' / q(c2),
// and a pass that then rejects c2 uses alpha1 = alpha / (s_i D) and
// beta' = beta / D + 1/Z', posted as 2^-e alpha / s_i and 2^-e (beta + D / Z')
// with 2^e <= D < 2^(e+1): its sum then comes in units of D / 2^e (Ctl::s_unit) and
// no division stands before it.  Only D depends on the pass's S, so of the next
// remaining child c2 of i it is known before S arrives:
//   * kAheadTest: c2 is a leaf with X > 0: it is accepted iff u D < X;
//   * kAheadPrune: X = 0, c2 has rate 0 whatever S is: it is removed, and the
//     pass for it follows (about half of all passes of EAGLE-shaped trees);
//   * kAheadDescend: c2 has children and X > 0: the traversal goes down to c2,
//     whose chain's rows are normalised next;
//   * kAheadUp: no child remains: i itself is tested with its new rate S / D
//     and accepted iff u D < S; the pass that rejects i at its parent g depends
//     only on g's state.
// The next job is posted as soon as S arrives, the state update
// (control_step_ahead) done while it runs.
// Float64 is slow here (64 cycles a dependent operation, 426 a division), so what
// does not depend on S is in child tables (child_order) or worked out while the
// pass runs, and the three divisions S leads to are done by three lanes at once.
// With all four modes, against the leaf test and kAheadUp alone: the persistent
// kernel at V = 128256 takes 453 -> 421 us (B = 128), 256 -> 237 us (B = 32, given
// normalisers), the cluster kernel at V = 32000, B = 64 183 -> 148 us.
// The passes in units of D / 2^e, with 1 / D worked out after they are posted
// instead of before: persistent kernel, V = 128256, B = 128 408 -> 399 us; cluster
// kernel, V = 128256, B = 32, given normalisers 117 -> 112 us, V = 32000, B = 64
// 134 -> 132 us.
enum : int { kAheadTest = 1, kAheadPrune = 2, kAheadDescend = 3, kAheadUp = 4 };

struct Ahead {
  int ok;          // 1: the next step is decided from D alone (see mode)
  int mode;
  int i, c, c2, g, nmask, n_rows;
  double p, omp, pm;             // p_i, 1 - p_i, p_i x the removed tokens' mass
  double X, alpha, beta, invZn, mb0, q0, uu, msum_g;
  float ainvs;                        // the next pass at i: alpha / s_i
  float alpha1_g, beta_g, rowmax_g;   // kAheadUp: the pass at g that rejects i
};

// S-independent part of the next step, after posting the pass for ctl.pending;
// the next pass's removed tokens (ascending) go to mtok2, the rows to
// normalise next to s.job_rows.
__device__ inline void prepare_ahead(const TreeSmem& s, const Ctl& ctl, Ahead& ah,
                                     int* mtok2, const float* __restrict__ u) {
  ah.ok = 0;
  if (ctl.job.kind != kJobPass) return;
  const int c = ctl.pending, i = s.par[c];
  if (!(s.rows[i] > 0.f)) return;
  const double p = s.p[i], a = s.a[i], b = s.b[i];
  const double alpha = p * a, beta = p * b + s.invZ[c];
  ah.i = i;
  ah.c = c;
  ah.p = p;
  ah.omp = 1.0 - p;
  ah.pm = p * ctl.masked_sum;
  ah.alpha = alpha;
  ah.beta = beta;
  ah.mb0 = s.mb0[c];
  ah.q0 = (double)s.gq[c];
  const int c2 = s.next[c];   // (the children after c all remain)
  ah.c2 = c2;
  if (c2 < 0) {
    if (i == 0) return;   // the root: the bonus draw follows
    const int g = s.par[i];
    // the pass post_pass(s, ctl, g, i) would post (g's state does not change)
    const double pg = s.p[g];
    ah.alpha1_g = (float)(pg * s.a[g] * s.invs[g]);
    ah.beta_g = (float)(pg * s.b[g] + s.invZ[i]);
    ah.rowmax_g = s.rowm[g];
    ah.nmask = removed_tokens(s, g, i, mtok2);
    ah.msum_g = removed_mass(s, g, i);
    ah.uu = (double)u[i];
    ah.mode = kAheadUp;
    ah.g = g;
    ah.ok = 1;
    return;
  }
  const double invZn = s.invZ[c2];
  if (!(invZn > 0.0)) return;
  const double y = fmax(alpha * s.mb0[c2] - beta * (double)s.gq[c2], 0.0);
  if (y > 0.0 && s.first[c2] >= 0) {
    int n = 0;
    for (int k = c2; k >= 0 && s.first[k] >= 0; k = first_alive_child(s, k))
      if (!(s.rows[k] > 0.f)) s.job_rows[n++] = k;
    if (n == 0) return;
    ah.n_rows = n;
    ah.mode = kAheadDescend;
    ah.ok = 1;
    return;
  }
  ah.ainvs = (float)(alpha * s.invs[i]);
  ah.invZn = invZn;
  ah.X = y * s.zq[c2];
  ah.nmask = removed_tokens(s, i, c2, mtok2);
  ah.uu = (double)u[c2];
  ah.mode = ah.X > 0.0 ? kAheadTest : kAheadPrune;
  ah.g = -1;
  ah.ok = 1;
}

// e with 2^e <= D < 2^(e+1), within what a float32 scale can undo.
__device__ __forceinline__ int unit_exponent(double D) {
  return min(max((__double2hiint(D) >> 20) - 1023, -100), 100);
}

// The next job of the step described by `ah`, given the pass's S (D = S + 1 -
// p_i); false if that job needs the updated state first (the residual draw at i).
// `accept`: the test's outcome.
__device__ inline bool job_ahead(const TreeSmem& s, const Ahead& ah, double S, double D,
                                 Job& j, bool& accept) {
  accept = false;
  j.n_rows = 1;
  j.kind = kJobPass;
  j.nmask = ah.nmask;
  if (ah.mode == kAheadUp) {
    accept = ah.uu * D < S;
    j.node = ah.g;
    j.alpha1 = ah.alpha1_g;
    j.beta = ah.beta_g;
    j.rowmax = ah.rowmax_g;
    return !accept;
  }
  if (ah.mode == kAheadDescend) {
    j.kind = kJobStats;
    j.n_rows = ah.n_rows;
    j.node = ah.c2;
    return true;
  }
  if (ah.mode == kAheadTest) accept = ah.uu * D < ah.X;
  if (accept) {
    j.kind = kJobBonusLeaf;
    j.node = ah.c2;
    j.nmask = 0;
    return true;
  }
  j.node = ah.i;
  const float unit = __int_as_float((127 - unit_exponent(D)) << 23);
  j.alpha1 = ah.ainvs * unit;
  j.beta = (float)(ah.beta + ah.invZn * D) * unit;
  j.rowmax = s.rowm[ah.i];
  return true;
}

// Bookkeeping of a pass at i for child c whose job has been posted already
// (msum: the stored masses of i's other removed children).
__device__ inline void note_pass(const TreeSmem& s, Ctl& ctl, int i, int c, double msum,
                                 double s_unit) {
  ctl.pending = c;
  ctl.s_unit = s_unit;
  ctl.job.kind = kJobPass;
  ctl.job.n_rows = 1;
  ctl.job.node = i;
  ctl.masked_sum = msum;
  ctl.n_passes++;
  s.npass[i]++;
}

// control_step for the pass described by `ah`, given D, inv_d = 1 / D, inv_s = 1 /
// S and p_new = S / D, with the test going the way `accept` says (the decision
// taken ahead, so that the state follows the job already posted).
__device__ inline void control_step_ahead(const TreeSmem& s, Ctl& ctl, const Ahead& ah,
                                          bool accept, double D, double inv_d,
                                          double inv_s, double p_new) {
  const int i = ah.i, c = ah.c;
  const double na = ah.alpha * inv_s, nb = ah.beta * inv_s, scale = ah.p * inv_s;
  const double mc = fmax(na * ah.mb0 - nb * ah.q0, 0.0);
  for (int j = s.first[i]; j != c; j = s.next[j]) s.m[j] *= scale;
  s.m[c] = mc;
  s.a[i] = na;
  s.b[i] = nb;
  s.p[i] = p_new;
  const double msum = ctl.masked_sum * scale + mc;
  ctl.pending = -1;
  ctl.node = i;
  if (ah.mode == kAheadUp) {
    ctl.n_tests++;
    s.dbgp[i] = (float)p_new;
    if (accept) {
      post_bonus(s, ctl, i);
      return;
    }
    s.state[i] = kRejected;
    note_pass(s, ctl, ah.g, i, ah.msum_g, 1.0);
    return;
  }
  if (ah.mode == kAheadDescend) {   // (control_step goes down to c2 after the job)
    ctl.job.kind = kJobStats;
    ctl.job.n_rows = ah.n_rows;
    return;
  }
  const int c2 = ah.c2;
  const double s_unit = inv_d * __hiloint2double((unit_exponent(D) + 1023) << 20, 0);
  if (ah.mode == kAheadPrune) {
    s.state[c2] = kPruned;
    s.dbgp[c2] = 0.f;
    note_pass(s, ctl, i, c2, msum, s_unit);
    return;
  }
  const double pc = fmin(ah.X * inv_d, 1.0);
  s.p[c2] = pc;
  ctl.node = c2;
  ctl.n_tests++;
  s.dbgp[c2] = (float)pc;
  if (accept) {
    post_bonus(s, ctl, c2);
    return;
  }
  s.state[c2] = kRejected;
  note_pass(s, ctl, i, c2, msum, s_unit);
}

// Advances the serial traversal until it needs vocabulary work; posts it.
__device__ inline void control_step(const TreeSmem& s, Ctl& ctl, const float* __restrict__ u) {
  if (ctl.job.kind == kJobPass) {
    const int c = ctl.pending, i = s.par[c];
    apply_rejection(s, ctl, i, c);
    ctl.pending = -1;
    ctl.node = i;
    if (i != 0 && s.p[i] == 0.0) {   // rate 0: remove i with what is left below it
      s.state[i] = kPruned;
      s.dbgp[i] = 0.f;
      post_pass(s, ctl, s.par[i], i);
      return;
    }
  }
  for (;;) {
    const int node = ctl.node;
    const int c = first_alive_child(s, node);
    if (c < 0) {
      if (node == 0) { post_bonus(s, ctl, 0); return; }
      ctl.n_tests++;
      s.dbgp[node] = (float)s.p[node];
      if ((double)u[node] < s.p[node]) { post_bonus(s, ctl, node); return; }
      s.state[node] = kRejected;
      post_pass(s, ctl, s.par[node], node);
      return;
    }
    if (!(s.rows[node] > 0.f)) {
      ctl.job.kind = kJobStats;
      ctl.job.n_rows = chain_needing_stats(s, node);
      return;
    }
    double pc;
    if (!child_rate(s, node, c, &pc)) {
      ctl.bad |= 8u;
      ctl.accepted = -1;
      ctl.job.kind = kJobDone;
      return;
    }
    if (pc == 0.0) {
      s.state[c] = kPruned;
      s.dbgp[c] = 0.f;
      post_pass(s, ctl, node, c);
      return;
    }
    s.p[c] = pc;
    ctl.node = c;
  }
}

// ------------------------------------------- token-level verification ----
//
// The top-down verifier Traversal Verification is compared with (§2.2, "Tok.V"
// of §4): at the current node ctl.node its children are tried in order by
// Recursive Rejection Sampling without replacement (Algorithm 2).  That is
// Eqs. (1)-(3) with the node's rate held at 1: min(M_b'(x_c) / M_s'(x_c), 1) is
// child_rate at p = 1, and the residual update [M_b' - M_s']_+ / S with x_c
// removed from M_s' is apply_rejection at p = 1, which leaves p = 1.  An
// accepted child becomes the current node with its own rows (a = 1, b = 0,
// Z = 1 from the tree set-up); the bonus token comes from an accepted leaf's
// own row, or from the current node's residual once all its children are
// rejected.  Only the current node's row is normalised.  A child of rate 0
// is rejected without counting as a test (its uniform cannot accept it).
__device__ inline void control_step_token(const TreeSmem& s, Ctl& ctl,
                                          const float* __restrict__ u) {
  if (ctl.job.kind == kJobPass) {
    const int c = ctl.pending, i = s.par[c];
    apply_rejection(s, ctl, i, c);
    ctl.pending = -1;
    ctl.node = i;
  }
  for (;;) {
    const int node = ctl.node;
    if (s.first[node] < 0) {   // an accepted leaf (or a root without children)
      post_bonus(s, ctl, node);
      return;
    }
    if (!(s.rows[node] > 0.f)) {
      ctl.job.kind = kJobStats;
      ctl.job.n_rows = 1;
      s.job_rows[0] = node;
      return;
    }
    const int c = first_alive_child(s, node);
    if (c < 0) {               // every child rejected: the residual at node
      post_bonus(s, ctl, node);
      return;
    }
    double pc;
    if (!child_rate(s, node, c, &pc)) {
      ctl.bad |= 8u;
      ctl.accepted = -1;
      ctl.job.kind = kJobDone;
      return;
    }
    s.dbgp[c] = (float)pc;
    if (pc > 0.0) {
      ctl.n_tests++;
      if ((double)u[c] < pc) {   // accepted: c becomes the current node
        s.p[c] = 1.0;
        ctl.node = c;
        continue;
      }
    }
    s.state[c] = kRejected;
    post_pass(s, ctl, node, c);
    return;
  }
}

// One step of the tree's verification method until it needs vocabulary work.
__device__ inline void advance(const TreeSmem& s, Ctl& ctl, const float* __restrict__ u,
                               bool token_level) {
  if (token_level) control_step_token(s, ctl, u);
  else control_step(s, ctl, u);
}

}  // namespace fused
}  // namespace tvk
