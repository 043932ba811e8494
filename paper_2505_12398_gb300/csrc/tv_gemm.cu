// tv_gemm.cu -- the target model's LM head fused with the row normalisers
// (sm_103a).
//
// The target distributions M_b(.|X^i) = softmax(l_i / T) that Traversal
// Verification reads (§3.1) come from the logits l = H W^T of the target
// model's last layer (hidden states H [M][K], output embedding W [V][K],
// bf16).  This kernel computes them on the 5th-generation tensor cores and, in
// the same pass, each stored row's normaliser: m = max_v l[v] and
// s = sum_v 2^((l[v] - m) c), c = log2(e) / T, evaluated on the bf16 values
// it stores.  Given those, verification never streams a row for its
// normaliser.
//
// Two forms of one persistent kernel, one CTA per SM, walk tiles of l in
// groups of row tiles holding 32 MiB of H, row tile fastest inside a group, so
// that the CTAs running at the same time share W tiles through L2 while the
// group's H stays resident.  One group (976 x 4096 x 128256) reads W and H from HBM once,
// 1.11 GB; two (7808 rows) do not reach their 2.2 GB, 4.7 and 7.6 GB in two captures: the
// 2 GB of logits pass through the same L2.  The tensor cores bound that size all the
// same (1.01 of the burst rate, at up to 1.8 TB/s read).
//   * SM pairs (tcgen05 cta_group::2; more than 128 rows): the two CTAs of a
//     cluster own a 256 x bn tile, each holding 128 rows of H and bn / 2 of the
//     tile's W rows in its shared memory; the leader issues the MMAs of both.
//     Each SM then loads 32 KB for a stage's 128 x 256 x 64 multiply-adds
//     instead of the 48 KB that a tile of its own takes.  Bound by the tensor
//     cores and the clock that the power cap leaves them (27 waves for 26.3 and 4096
//     rows for 3904 at 3904 x 4096 x 32000): 645 -> 618 us there, 976 x 4096 x
//     128256 702 -> 585 us, 7808 x 4096 x 128256 4929 -> 4898 us, against single
//     SMs with 4 epilogue warps.
//   * single SMs (up to 128 rows): 128 x bn tiles, W's bytes from HBM bound
//     it.  Only the box of H rows that exist is loaded (the MMA's other rows
//     read whatever is next in shared memory; their results are not used).
// The tile width bn is chosen for the waves it makes (tile_width): at 61 rows and
// V = 128256, 4 waves of 224 columns on 152 SMs instead of 4 of 256 (3.3 full).
// With 30 to 55 KB more in flight per SM (the H box of the rows that exist) and
// a block per row in the merge, already waiting when this kernel ends (a
// programmatic dependent launch), 188.9 -> 163 us there (157 us of bytes at 6.8
// TB/s; 165 us without that launch), one row 225 -> 156 us.
// In both:
//   * warp 0 streams 64-element K slices of H and W into a ring of shared
//     memory with 2-D TMA copies (128-byte swizzle, the layout the tensor cores
//     read), across tile boundaries;
//   * warp 1 allocates all 512 columns of tensor memory, two fp32
//     accumulators of up to 256 columns, and (of the leader) issues tcgen05.mma
//     (K=16 per instruction) into them in turn, releasing each stage with
//     tcgen05.commit.  Both loops run in the whole warp and one elected lane
//     issues (elect_one): with loops of one lane the tensor cores waited for the
//     issue, 618 -> 590 us at 3904 x 4096 x 32000, 4929 -> 4608 us at 7808 x 4096 x
//     128256, 750 -> 695 us at 1952 x 2048 x 151936 (and 536 -> 469, 4000 -> 3477
//     us for the first two on operands of zeros, where no power cap bounds it);
//   * warps 2-9 (two per TMEM lane quarter, each taking every other 32
//     columns, one row per thread) read the finished accumulator with
//     tcgen05.ld, round to bf16, store the logits and keep the row's running
//     (max, sum) over their columns, while the tensor cores fill the other
//     accumulator.  With a short K the epilogue is what bounds the kernel:
//     packed bf16 maxima, two columns per instruction, 32-byte stores and the
//     next chunk's tensor-memory load in flight take 3904 x 512 x 32000 from 364
//     to 128 us.
// A second kernel merges the partial (max, sum) of each row.
//
// Every mbarrier wait is bounded; a wait that gives up raises
// TV_STATUS_TIMEOUT in the status word and the CTA still frees its tensor
// memory before it exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "tv_device.cuh"
#include "tv_launch.h"
#include "tv_ptx.cuh"

namespace tvk {
namespace gemm {

constexpr int kBM = 128;          // rows of a tile per CTA (TMEM lanes)
constexpr int kBN = 256;          // columns of a tile at most (TMEM columns)
constexpr int kBK = 64;           // K per stage: 128 bytes of bf16, one swizzle row
constexpr int kUmmaK = 16;        // K per tcgen05.mma of kind::f16
constexpr int kMaxStages = 8;
constexpr size_t kRingBytes = 200u << 10;
// Tile order: groups of row tiles holding about kGroupBytes of H, row tile
// fastest inside a group, so that the CTAs running at once share W tiles
// through L2 while the group's rows of H stay resident.
constexpr size_t kGroupBytes = 32u << 20;
constexpr int kEpiWarps = 8;      // two per TMEM lane quarter
constexpr int kThreads = 64 + 32 * kEpiWarps;   // TMA warp, MMA warp, epilogue warps
constexpr uint32_t kRowBytes = kBK * 2;         // one row of a stage's operand tile
constexpr int kAccBufs = 2;                     // accumulators in tensor memory
constexpr uint32_t kTmemCols = kAccBufs * kBN;  // fp32: one column per output column
constexpr size_t kSmemBytes = kRingBytes + 1024;   // + alignment slack

// Instruction descriptor of tcgen05.mma kind::f16: fp32 accumulator (bits
// 4-5 = 1), bf16 A and B (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 =
// 0), N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__device__ __forceinline__ uint32_t instr_desc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}

// Shared-memory matrix descriptor of a K-major operand tile written by TMA
// with the 128-byte swizzle: start address >> 4 (bits 0-13), leading byte
// offset (unused with this swizzle, set to 1; bits 16-29), stride byte offset
// 1024 B >> 4 between groups of 8 rows (bits 32-45), descriptor version 1
// (bit 46), swizzle mode 2 = 128 B (bits 61-63).  Tiles are 1024-byte aligned
// (base offset 0).  Stepping K by 16 bf16 inside the swizzled 128-byte row
// advances the start address by 32 bytes.
__device__ __forceinline__ uint64_t smem_desc(const void* p) {
  const uint64_t addr = smem_u32(p);
  return ((addr >> 4) & 0x3FFFull) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}

// 2-D tiled TMA load of box {x .. x+box0, y .. y+box1} (x in elements, a
// multiple of 64 here, so 16-byte aligned) into this CTA's shared memory,
// counted on the barrier at cluster address `bar` (kPair: the pair leader's).
template <bool kPair>
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y,
                                            uint32_t bar) {
  if constexpr (kPair)
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::"
        "bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// Row and column tile of the t-th tile in the kernel's order.
__device__ __forceinline__ void tile_coords(int t, int m_tiles, int n_tiles, int group,
                                            int& mt, int& nt) {
  const int g = group > 0 && group < m_tiles ? group : m_tiles;
  const int full = (m_tiles / g) * g * n_tiles;       // tiles in whole groups
  if (t < full) {
    const int grp = t / (g * n_tiles), r = t - grp * g * n_tiles;
    mt = grp * g + r % g;
    nt = r / g;
  } else {
    const int gt = m_tiles - (m_tiles / g) * g, r = t - full;
    mt = (m_tiles / g) * g + r % gt;
    nt = r / gt;
  }
}

// True in one lane of a converged warp.  The loops around the tensor-core and TMA
// instructions run in the whole warp with those instructions alone in the chosen
// lane: their operands (descriptors, addresses, coordinates) then stay in the
// warp's uniform registers, which the instructions read, instead of being moved
// there one by one from a divergent lane's.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p));
  return p != 0;
}

template <bool kPair>
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                          uint32_t accumulate) {
  if constexpr (kPair)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrives on `bar` (kPair: on the barrier at that offset in both CTAs) once
// every tcgen05.mma issued so far by this thread is done.
template <bool kPair>
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  if constexpr (kPair)
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
        " [%0], %1;" ::"r"(smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
  else
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}

template <bool kPair>
__device__ __forceinline__ void tmem_alloc(uint32_t* slot) {   // a whole warp (of each CTA)
  if constexpr (kPair) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  } else {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
}

template <bool kPair>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr) {   // the allocating warp(s)
  if constexpr (kPair)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                 "r"(kTmemCols)
                 : "memory");
  else
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                 "r"(kTmemCols)
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 32 consecutive fp32 accumulator columns of this warp's 32 TMEM lanes (lane
// i of the warp reads TMEM lane base + i): one row per thread.  The registers
// hold the columns after tmem_wait only, which takes them through an asm
// statement of its own so that no use of them precedes it.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
      "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
        "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]),
        "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]),
        "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]),
        "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :
      : "memory");
}

__device__ __forceinline__ void st_global_32b(void* p, const uint32_t* w) {   // 32-byte aligned
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity) ? 1 : 0) != 0;
}

// Launch shape: tile width, H rows a TMA box takes per CTA, ring stages.
struct Shape {
  int bn, a_box, stages;
  __host__ __device__ uint32_t a_bytes() const { return (uint32_t)a_box * kRowBytes; }
  __host__ __device__ uint32_t b_bytes(bool pair) const {
    return (uint32_t)(pair ? bn / 2 : bn) * kRowBytes;
  }
};

// Rounds 32 accumulator columns of a row to bf16, stores the first n (a
// multiple of 8) at dst (32-byte stores where `wide`: a 16-byte store writes
// half a sector) and adds the stored values to the row's running (max, sum).
__device__ __forceinline__ void store_and_sum(const uint32_t (&r)[32], __nv_bfloat16* dst, int n,
                                              bool wide, float2 ch, float2 cl, float& m_run,
                                              float& s_run) {
  uint32_t packed[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const __nv_bfloat162 h =
        __floats2bfloat162_rn(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
    packed[i] = *reinterpret_cast<const uint32_t*>(&h);
  }
  if (wide && n >= 32) {
    st_global_32b(dst, packed);
    st_global_32b(dst + 16, packed + 8);
  } else {
    uint4* d4 = reinterpret_cast<uint4*>(dst);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (8 * i < n)
        d4[i] = make_uint4(packed[4 * i], packed[4 * i + 1], packed[4 * i + 2],
                           packed[4 * i + 3]);
  }
  // the maximum (exact on bf16 pairs) and the sum, two columns at a time;
  // columns past the end count as -inf and weigh nothing
  if (n < 32) {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (2 * i >= n) packed[i] = 0xff80ff80u;   // two bf16 -inf
  }
  __nv_bfloat162 hm = *reinterpret_cast<const __nv_bfloat162*>(&packed[0]);
#pragma unroll
  for (int i = 1; i < 16; ++i)
    hm = __hmax2(hm, *reinterpret_cast<const __nv_bfloat162*>(&packed[i]));
  const float cm = fmaxf(__low2float(hm), __high2float(hm));
  if (cm > m_run) {
    if (m_run != TV_NEG_INF) s_run *= exp2_split(m_run - cm, 0.f, ch.x, cl.x);
    m_run = cm;
  }
  const float2 mm = make_float2(-m_run, -m_run);
  float2 acc[4];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float2 d = __fadd2_rn(make_float2(bf16_lo(packed[i]), bf16_hi(packed[i])), mm);
    d.x = fmaxf(d.x, -1.0e4f);      // -inf / NaN -> weight ~0
    d.y = fmaxf(d.y, -1.0e4f);
    float2 e = exp2_corrected_x2(d, ch, cl);
    if (2 * i >= n) e = make_float2(0.f, 0.f);   // (n is even)
    acc[i & 3] = i < 4 ? e : __fadd2_rn(acc[i & 3], e);
  }
  const float2 s2 = __fadd2_rn(__fadd2_rn(acc[0], acc[1]), __fadd2_rn(acc[2], acc[3]));
  s_run += s2.x + s2.y;
}

// The tiles t = first, first + step, ... of l = H W^T (in the order of
// tile_coords), stored as bf16, and each row's (max, sum of 2^((l - max) c))
// over a tile's columns in part[row][tile].  kPair: launched as clusters of two
// CTAs.
template <bool kPair>
__global__ void __launch_bounds__(kThreads, 1)
    lm_head_kernel(const __grid_constant__ CUtensorMap map_h,
                   const __grid_constant__ CUtensorMap map_w, int M, int V, int K, Shape shape,
                   float c_hi, float c_lo, __nv_bfloat16* __restrict__ logits,
                   float2* __restrict__ part, int m_tiles, int n_tiles, int group, bool wide,
                   uint32_t* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];   // (kPair: the leader's are used)
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t acc_full[kAccBufs];    // accumulator ready (tcgen05.commit)
  __shared__ __align__(8) uint64_t acc_empty[kAccBufs];   // accumulator read (epilogue warps;
                                                          // kPair: the leader's is used)
  __shared__ __align__(8) uint64_t drain_bar;
  // the odd chunks' (max, sum) of a row, from one warp of a lane quarter to the other
  __shared__ __align__(8) uint64_t half_full[4];
  __shared__ __align__(8) uint64_t half_empty[4];
  __shared__ float2 half_ms[kBM];
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  // the TMA tiles need 1024-byte alignment (128-byte swizzle atoms)
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t rank = kPair ? cluster_rank() : 0u;
  const int first = kPair ? (int)blockIdx.x >> 1 : (int)blockIdx.x;
  const int step = kPair ? (int)gridDim.x >> 1 : (int)gridDim.x;
  const int tile_rows = kPair ? 2 * kBM : kBM;
  const int bn = shape.bn, bn_own = kPair ? bn / 2 : bn;
  const uint32_t n_stages = (uint32_t)shape.stages;
  const uint32_t a_bytes = shape.a_bytes(), stage_bytes = a_bytes + shape.b_bytes(kPair);
  const int nkb = K / kBK;
  const int n_total = m_tiles * n_tiles;
  if (threadIdx.x == 0) {
    for (uint32_t s = 0; s < n_stages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int k = 0; k < kAccBufs; ++k) {
      mbar_init(&acc_full[k], 1);
      mbar_init(&acc_empty[k], kPair ? 2 * kEpiWarps : kEpiWarps);
    }
    mbar_init(&drain_bar, 1);
    for (int k = 0; k < 4; ++k) {
      mbar_init(&half_full[k], 1);
      mbar_init(&half_empty[k], 1);
    }
    failed = 0;
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc<kPair>(&tmem_slot);
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) cluster_sync_all();   // the peer's barriers and tensor memory are ready
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  asm volatile("griddepcontrol.launch_dependents;");   // (the merge waits for the whole grid)

  if (warp == 0) {
    // ---- TMA producer: one ring across all of this CTA's tiles ----
    uint32_t it = 0, s = 0, ph = 0;
    bool ok = true;
    for (int t = first; t < n_total && ok; t += step) {
      int mt, nt;
      tile_coords(t, m_tiles, n_tiles, group, mt, nt);
      const int m0 = mt * tile_rows + (int)rank * kBM, n0 = nt * bn + (int)rank * bn_own;
      for (int kb = 0; kb < nkb; ++kb, ++it) {
        if (it >= n_stages && !wait_warp(&empty_bar[s], ph ^ 1u)) {
          ok = false;
          break;
        }
        uint8_t* a = smem + s * stage_bytes;
        uint32_t bar = smem_u32(&full_bar[s]);
        if constexpr (kPair) bar = map_shared(&full_bar[s], 0);
        if (elect_one()) {
          // (kPair: the leader's barrier counts both CTAs' bytes)
          if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], kPair ? 2 * stage_bytes : stage_bytes);
          tma_load_2d<kPair>(a, &map_h, kb * kBK, m0, bar);
          tma_load_2d<kPair>(a + a_bytes, &map_w, kb * kBK, n0, bar);
        }
        __syncwarp();
        if (++s == n_stages) { s = 0; ph ^= 1u; }
      }
    }
    if (!ok) failed = 1;
    // the copies issued last have landed before the CTA may exit (kPair: the
    // leader waits for both CTAs' copies, the peer for the leader at the end)
    if (rank == 0)
      for (uint32_t j = it > n_stages ? it - n_stages : 0u; j < it; ++j)
        if (!wait_warp(&full_bar[j % n_stages], (j / n_stages) & 1)) failed = 1;
  } else if (warp == 1) {
    // ---- tensor-core issue, the two accumulators in turn ----
    if (rank == 0) {
      const uint32_t idesc = instr_desc(tile_rows, bn);
      const uint64_t desc0 = smem_desc(smem);
      uint32_t s = 0, ph = 0;
      bool ok = true;
      int j = 0;
      for (int t = first; t < n_total && ok; t += step, ++j) {
        const uint32_t acc = (uint32_t)j & 1u;
        if (j >= kAccBufs) {
          const uint32_t par = ((j >> 1) - 1) & 1;
          const bool got = kPair ? mbar_wait_cluster(&acc_empty[acc], par)
                                 : mbar_wait(&acc_empty[acc], par);
          if (!__all_sync(0xffffffffu, got)) {
            ok = false;
            break;
          }
        }
        tc_fence_after();
        const uint32_t d = tmem + acc * (uint32_t)kBN;
        for (int kb = 0; kb < nkb; ++kb) {
          if (!wait_warp(&full_bar[s], ph)) {
            ok = false;
            break;
          }
          tc_fence_after();
          // (the start address field counts 16 bytes)
          const uint64_t da = desc0 + (uint64_t)((s * stage_bytes) >> 4);
          const uint64_t db = da + (uint64_t)(a_bytes >> 4);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < kBK / kUmmaK; ++k) {
              const uint64_t off = (uint64_t)((k * kUmmaK * 2) >> 4);   // 32 bytes of K
              umma_bf16<kPair>(d, da + off, db + off, idesc, (kb > 0 || k > 0) ? 1u : 0u);
            }
            umma_commit<kPair>(&empty_bar[s]);   // the stage is free once these MMAs are done
            if (kb == nkb - 1) umma_commit<kPair>(&acc_full[acc]);   // the accumulator is complete
          }
          __syncwarp();
          if (++s == n_stages) { s = 0; ph ^= 1u; }
        }
      }
      if (!ok) failed = 1;
      // every MMA issued has finished before tensor memory is freed
      if (elect_one()) umma_commit<kPair>(&drain_bar);
      __syncwarp();
    }
    // (kPair, the peer: the leader's last signal; none is on its way to this CTA
    // after it)
    if (!wait_warp(&drain_bar, 0)) failed = 1;
  } else {
    // ---- epilogue: one row per thread, every other 32-column chunk ----
    const int q = warp & 3;                       // the TMEM lane quarter of this warp
    const int half = (warp - 2) >> 2;
    const float2 ch = make_float2(c_hi, c_hi), cl = make_float2(c_lo, c_lo);
    int j = 0;
    for (int t = first; t < n_total; t += step, ++j) {
      const uint32_t acc = (uint32_t)j & 1u;
      const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[acc], (j >> 1) & 1));
      if (!ok) {
        if (lane == 0) failed = 1;
        break;
      }
      tc_fence_after();
      int mt, n_tile;
      tile_coords(t, m_tiles, n_tiles, group, mt, n_tile);
      const int n0 = n_tile * bn;
      const int row = mt * tile_rows + (int)rank * kBM + q * 32 + lane;
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + acc * (uint32_t)kBN;
      float m_run = TV_NEG_INF, s_run = 0.f;
      // chunk k + 1 is on its way from tensor memory while chunk k is worked on
      uint32_t acc_regs[2][32];
      __syncwarp();
      tmem_ld32(tbase + (uint32_t)(half * 32), acc_regs[0]);
#pragma unroll
      for (int k = 0; k < kBN / 64; ++k) {
        const int c = half * 32 + 64 * k;
        if (c >= bn) break;                       // (the same in the whole warp)
        uint32_t (&r)[32] = acc_regs[k & 1];
        tmem_wait(r);
        if (c + 64 < bn) {
          __syncwarp();
          tmem_ld32(tbase + (uint32_t)(c + 64), acc_regs[(k + 1) & 1]);
        } else {
          // all read: this accumulator may be overwritten once every warp has
          // come here
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if constexpr (kPair) mbar_arrive_remote(map_shared(&acc_empty[acc], 0));
            else mbar_arrive(&acc_empty[acc]);
          }
        }
        const int col0 = n0 + c;
        const int n = min(bn - c, V - col0);      // columns of the chunk that exist
        if (row < M && n > 0)
          store_and_sum(r, logits + (size_t)row * V + col0, n, wide, ch, cl, m_run, s_run);
      }
      // the quarter's two warps: one partial per row and tile (one from each doubles
      // the scratch that a new handle allocates: its first pass over 183 rows of 2304,
      // V = 151936, took 284 us for 193; repeated passes 136 for 132)
      if (half == 1) {
        if (j > 0 && !wait_warp(&half_empty[q], (j - 1) & 1)) {
          if (lane == 0) failed = 1;
          break;
        }
        half_ms[q * 32 + lane] = make_float2(m_run, s_run);
        __syncwarp();
        if (lane == 0) mbar_arrive(&half_full[q]);
      } else {
        if (!wait_warp(&half_full[q], j & 1)) {
          if (lane == 0) failed = 1;
          break;
        }
        const float2 o = half_ms[q * 32 + lane];
        __syncwarp();
        if (lane == 0) mbar_arrive(&half_empty[q]);
        const float mx = fmaxf(m_run, o.x);
        float sum = 0.f;
        if (m_run != TV_NEG_INF) sum = s_run * exp2_split(m_run - mx, 0.f, c_hi, c_lo);
        if (o.x != TV_NEG_INF) sum += o.y * exp2_split(o.x - mx, 0.f, c_hi, c_lo);
        if (row < M) part[(size_t)row * n_tiles + n_tile] = make_float2(mx, sum);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  // (the leader's drain is over: no MMA or copy still touches either CTA)
  if constexpr (kPair) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc<kPair>(tmem);
  }
  if (threadIdx.x == 0 && failed) atomicOr(status, 32u);
}

// Merges the partial (max, sum) of each row into the row's normaliser: one
// block per row, so that a few rows with a thousand partials each do not wait
// on one warp's loads (partials in order within each thread, then across
// lanes and warps).  Launched as a programmatic dependent of lm_head_kernel: its
// blocks are already waiting when that kernel ends.
constexpr int kMergeThreads = 128;
__global__ void __launch_bounds__(kMergeThreads)
    lm_head_merge_kernel(const float2* __restrict__ part, int n_parts, float c_hi, float c_lo,
                         float2* __restrict__ out) {
  __shared__ float red[2][kMergeThreads / 32];
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the partials are there
  const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const float2* p = part + (size_t)row * n_parts;
  constexpr int kKeep = 8;          // partials kept in registers (1024 a row)
  float2 v[kKeep];
  float mx = TV_NEG_INF;
#pragma unroll
  for (int k = 0; k < kKeep; ++k) {
    const int t = tid + k * kMergeThreads;
    v[k] = t < n_parts ? p[t] : make_float2(TV_NEG_INF, 0.f);
    mx = fmaxf(mx, v[k].x);
  }
  for (int t = tid + kKeep * kMergeThreads; t < n_parts; t += kMergeThreads)
    mx = fmaxf(mx, p[t].x);
  mx = warp_max(mx);
  if (lane == 0) red[0][wid] = mx;
  __syncthreads();
  mx = red[0][0];
  for (int w = 1; w < kMergeThreads / 32; ++w) mx = fmaxf(mx, red[0][w]);
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < kKeep; ++k)
    if (v[k].x != TV_NEG_INF) s += v[k].y * exp2_split(v[k].x - mx, 0.f, c_hi, c_lo);
  for (int t = tid + kKeep * kMergeThreads; t < n_parts; t += kMergeThreads) {
    const float2 u = p[t];
    if (u.x != TV_NEG_INF) s += u.y * exp2_split(u.x - mx, 0.f, c_hi, c_lo);
  }
  s = warp_sum(s);
  if (lane == 0) red[1][wid] = s;
  __syncthreads();
  if (tid == 0) {
    float sum = 0.f;
    for (int w = 0; w < kMergeThreads / 32; ++w) sum += red[1][w];
    out[row] = make_float2(mx, sum);
  }
}

}  // namespace gemm
}  // namespace tvk

// --------------------------------------------------------------- launcher --

namespace {

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                 const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                 const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, fetched once through the runtime (no link
// dependency on the driver library).
EncodeTiled encoder() {
  static std::once_flag once;
  static EncodeTiled fn = nullptr;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiled>(p);
    else
      cudaGetLastError();
  });
  return fn;
}

// Row-major bf16 [rows][K] as a 2-D tensor with 64 x box_rows boxes and the
// 128-byte swizzle (rows past the end read as zeros).
bool make_map(CUtensorMap* map, const void* base, int rows, int K, int box_rows) {
  const EncodeTiled enc = encoder();
  if (!enc) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  const cuuint32_t box[2] = {(cuuint32_t)tvk::gemm::kBK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
             box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

constexpr int kGemmDevices = 64;
std::mutex g_gemm_mutex;
struct GemmDevice {
  int sms = 0, pairs = 0;   // CTAs and clusters of two that run at once
};
GemmDevice g_gemm[kGemmDevices];

// Tile width: of the widths the MMA takes (multiples of 16, of 32 for a pair),
// the one whose waves cover the fewest columns, counting each tile as `extra`
// columns wider than it is for the H rows it loads again.  A pair loads 128 H
// rows per SM for bn / 2 W rows, so extra = 256 there (M = 244, V = 128256: 7 waves
// of 256 columns 196 us, 8 of 224 205, 14 of 128 292, the same columns each); on
// single SMs W's bytes from HBM bound the kernel and 64 fits (M = 61, V = 128256:
// 4 waves of 224 165 us, 5 of 176 167, 6 of 144 168, 4 of 256 169, 8 of 128 175).
int tile_width(size_t m_tiles, int V, int units, bool pair, int extra) {
  const int unit = pair ? 32 : 16;
  int best = tvk::gemm::kBN;
  long best_cost = 0;
  for (int bn = tvk::gemm::kBN; bn >= 128; bn -= unit) {
    const long tiles = (long)m_tiles * ((V + bn - 1) / bn);
    const long cost = (tiles + units - 1) / units * (bn + extra);
    if (best_cost == 0 || cost < best_cost) {
      best_cost = cost;
      best = bn;
    }
  }
  return best;
}

template <bool kPair>
cudaError_t launch_lm_head(const CUtensorMap& map_h, const CUtensorMap& map_w, int M, int V, int K,
                           const tvk::gemm::Shape& shape, float c_hi, float c_lo, void* logits,
                           float2* part, int m_tiles, int n_tiles, int group, int units,
                           uint32_t* status, cudaStream_t stream) {
  using namespace tvk::gemm;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(std::min(m_tiles * n_tiles, units) * (kPair ? 2 : 1)), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = kPair ? 1 : 0;
  // 32-byte stores where every row's 32-column chunks start on 32 bytes
  const bool wide = V % 16 == 0 && (reinterpret_cast<uintptr_t>(logits) & 31u) == 0;
  return cudaLaunchKernelEx(&cfg, lm_head_kernel<kPair>, map_h, map_w, M, V, K, shape, c_hi, c_lo,
                            static_cast<__nv_bfloat16*>(logits), part, m_tiles, n_tiles, group,
                            wide, status);
}

// The device's CTA and cluster counts, with the kernels' shared memory limits
// set; false on a CUDA error.
bool gemm_device(int device, GemmDevice* out) {
  using namespace tvk::gemm;
  std::lock_guard<std::mutex> lock(g_gemm_mutex);
  GemmDevice& g = g_gemm[device];
  if (g.pairs < 1) {
    int sms = 0, pairs = 0;
    if (cudaFuncSetAttribute(lm_head_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSmemBytes) != cudaSuccess ||
        cudaFuncSetAttribute(lm_head_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSmemBytes) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
      return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)sms / 2 * 2, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&pairs, lm_head_kernel<true>, &cfg) != cudaSuccess ||
        pairs < 1)
      return false;
    g.sms = sms;
    g.pairs = std::min(pairs, sms / 2);
  }
  *out = g;
  return true;
}

}  // namespace

namespace {

// One row tile: single SMs, bound by W's bytes; more: SM pairs.
bool pairs_for(size_t M) { return M > tvk::gemm::kBM; }

int width_for(size_t M, int V, const GemmDevice& g) {
  const bool pair = pairs_for(M);
  const size_t tile_rows = pair ? 2 * tvk::gemm::kBM : tvk::gemm::kBM;
  return tile_width((M + tile_rows - 1) / tile_rows, V, pair ? g.pairs : g.sms, pair,
                    pair ? 256 : 64);
}

}  // namespace

size_t tv_lm_head_scratch(size_t rows, int V) {
  using namespace tvk::gemm;
  int device = 0;
  GemmDevice g;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= kGemmDevices ||
      !gemm_device(device, &g)) {
    cudaGetLastError();
    return 0;
  }
  // the most any call of up to `rows` rows takes (the width depends on its row
  // tiles only; a call's rows are an int)
  rows = std::min<size_t>(rows, INT_MAX);
  size_t most = 0;
  for (size_t M = std::min<size_t>(rows, kBM);;
       M = std::min<size_t>(rows, (M / (2 * kBM) + 1) * 2 * kBM)) {
    const int bn = width_for(M, V, g);
    most = std::max(most, M * ((V + bn - 1) / bn));
    if (M >= rows) return most;
  }
}

int tv_launch_lm_head(const void* hidden, const void* weight, int M, int K, int V, float c_hi,
                      float c_lo, void* logits, float2* part, float2* row_stats,
                      uint32_t* status, cudaStream_t stream) {
  using namespace tvk::gemm;
  if (M <= 0) return 0;
  int device = 0;
  GemmDevice g;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= kGemmDevices ||
      !gemm_device(device, &g)) {
    cudaGetLastError();
    return -5;
  }
  const bool pair = pairs_for(M);
  const int tile_rows = pair ? 2 * kBM : kBM;
  const int units = pair ? g.pairs : g.sms;
  const int m_tiles = (M + tile_rows - 1) / tile_rows;
  Shape shape;
  shape.a_box = std::min(kBM, (M + 7) / 8 * 8);
  shape.bn = width_for(M, V, g);
  shape.stages = (int)std::min<size_t>(
      kMaxStages, kRingBytes / (shape.a_bytes() + shape.b_bytes(pair)));
  CUtensorMap map_h, map_w;
  if (!make_map(&map_h, hidden, M, K, shape.a_box) ||
      !make_map(&map_w, weight, V, K, pair ? shape.bn / 2 : shape.bn))
    return -5;
  const int n_tiles = (V + shape.bn - 1) / shape.bn;
  const int group = (int)std::max<size_t>(1, kGroupBytes / ((size_t)tile_rows * K * 2));
  const cudaError_t e =
      pair ? launch_lm_head<true>(map_h, map_w, M, V, K, shape, c_hi, c_lo, logits, part, m_tiles,
                                  n_tiles, group, units, status, stream)
           : launch_lm_head<false>(map_h, map_w, M, V, K, shape, c_hi, c_lo, logits, part, m_tiles,
                                   n_tiles, group, units, status, stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return -5;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)M, 1, 1);
  cfg.blockDim = dim3(kMergeThreads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, lm_head_merge_kernel, (const float2*)part, n_tiles, c_hi,
                         c_lo, row_stats) != cudaSuccess) {
    cudaGetLastError();
    return -5;
  }
  return 0;
}
