// Tensor-core projection kernel for sm_100a: the LM-head contraction z = h W^T on
// tcgen05 with the accumulator in tensor memory, operands staged by TMA, and the
// online-softmax reduction (max / argmax / sum-exp / entropy numerator) fused into
// the epilogue, so the n x V logits never leave the SM.
//
// One kernel body; a kernel per way of handling token rows (RowMode) and per kind of head (kernels at the end of this file):
//   bf16 head, one CTA per worker, MMA M = 64 or 128 token rows              (n <= 128)
//   bf16 head, a cluster of two CTAs per worker, MMA M = 256 rows (cta_group::2): each
//               CTA stages its own 128 rows of h and HALF of the W tile, and the pair's
//               tensor cores read both halves, so a W byte enters shared memory once
//               per 256 token rows.                                          (n > 128)
//               Above 256 rows a unit may be two blocks of 256 rows, one accumulator each: a slab of W is then read by
//               the MMAs of both while it is in shared memory (TwoWalk).
//   8-bit (e4m3) head for decode batches of at most 128 rows: h is the sum of two e4m3
//               parts, stacked in one operand slab.  Up to 64 rows ONE kind::f8f6f4 MMA per K step
//               covers both parts along its M, and the epilogue adds the two accumulator rows of a
//               token before it folds them; above, two MMAs per K step (one per part) add into the
//               same rows.
//   bf16 head whose hidden size is no multiple of 8: the vocabulary is walked by residue class
//               (see OddMaps), otherwise like the bf16 head.
//
// Decomposition.  The vocabulary is cut into `chunks` contiguous ranges of granules
// (a multiple of 16 * kCta rows); the token rows into units of 128 * kCta.  A work unit is
// (chunk, row unit); units are numbered chunk-major so that workers running at the
// same time share W through L2, and worker w takes units w, w + workers, ...  (two row
// blocks: units of 512 rows, numbered group by group of row units and chunk-major in a
// group).  Inside
// a unit the chunk is walked in `tiles_per_unit` tiles of at most 256 vocabulary rows
// (the MMA's N), each a K-loop over d in slabs of 128 bytes per row.  With a learned router
// attached (bf16 head) one more unit per row unit follows the vocabulary units: its "vocabulary"
// is the rows of the router's first layer W1, and its epilogue applies bias, ReLU and the output
// layer's weights and sums over the hidden units instead of folding a softmax.
//
// Roles (warp-specialised, 352 threads per CTA):
//   warp 0   W producer: TMA loads of W slabs into a deep ring (W comes from HBM).  W never
//            depends on the previous kernel in the stream, so this warp does not wait for it:
//            under programmatic dependent launch the ring fills while that kernel finishes.
//   warp 6   h producer: TMA loads of h slabs into a short ring (h comes from L2)
//   warp 1   MMA issuer (leader CTA only): tcgen05.mma x4 per slab into one of two
//            256-column TMEM accumulators; also owns TMEM alloc/free
//   warps 2-5 and 7-10  epilogue, two warps per TMEM lane quadrant (32 rows): the first
//            group folds the lower half of a finished accumulator's columns, the second
//            group the upper half, 32 columns at a time, into per-row (m, idx, S, T)
//            registers while the next tile's MMAs run into the other accumulator.  Two
//            warps per scheduler hide each other's tensor-memory load and exp latency, and
//            the time between a worker's last MMA and its last partial -- which nothing
//            overlaps -- halves.
// At the end of a unit the second group hands its summary to the first through shared memory
// and every row's summary is written as one 16-byte partial.
//
// How much of W a CTA keeps in flight decides its streaming rate (latency-bound
// otherwise), so h slabs get their own small ring and, when n is small, a slab of only
// as many rows as n needs; the MMA then reads its remaining A rows from whatever
// follows in shared memory, which only affects accumulator rows that are never used.
//
// Every mbarrier wait is bounded (wall-clock limit); on expiry the kernel raises
// TLR_DEV_WAIT_TIMEOUT, lets its outstanding copies land, frees TMEM and returns.
// No TMA load uses cluster multicast.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "tlr_common.cuh"
#include "tlr_tc.cuh"
#include "tlr_tc8_dev.cuh"
#include "tlr_tc_ptx.cuh"

namespace tlr {

namespace {

constexpr int kBlockM = 128;                 // token rows per CTA == TMEM lanes
constexpr int kBlockN = 256;                 // max vocabulary rows per tile == accumulator columns
constexpr int kRowBytes = 128;               // bytes per slab row = one swizzle span (64 bf16 or 128 e4m3)
constexpr int kTmemCols = 512;
constexpr int kEpiWarps = 8;                 // two groups of four (one warp per TMEM lane quadrant each)
constexpr int kThreads = 32 * 11;
constexpr int kMaxAStages = 16;              // (the 8-bit head keeps up to 16 resident slabs of h)
constexpr int kMaxBStages = 12;
constexpr int kRelease = 16;                 // >= every ring depth that streams (see the barrier notes in the kernel)
constexpr int kBarrierBytes = 640;
constexpr int kScratchBytes = kBlockM * 16;  // one Partial per row: hand-over between the epilogue groups
constexpr int kSmemLimit = 232448;           // 227 KiB opt-in maximum per CTA
constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s
constexpr unsigned long long kAheadNs = 60000000000ull;     // and a minute for the role that starts ahead of the wait for the kernel in front
// 8-bit head: the weight scales of every epilogue warp's share of a tile, and the rows' power-of-two scales
constexpr int kScaleBytes = kEpiWarps * (kBlockN / 2) * 4;
constexpr int kRowScaleBytes = 64 * 4;
constexpr int kTc8ExtraBytes = kScaleBytes + kRowScaleBytes;
constexpr float kNoLogit = -1.0e30f;         // stands for a column beyond V: finite, so that 0 * y stays 0 in the folds

// The static schedule, identical in every role: worker w walks units w, w + workers, ...;
// each unit is `tiles_per_unit` tiles (possibly empty ones when the chunk is short).
struct Unit {
  int row0;    // first token row of this CTA in the unit
  int chunk;   // vocabulary chunk; -1 for a learned-router unit
  int g0;      // first granule of the chunk
  int G;       // granules in the chunk
  int tile_q, tile_r;   // tiles of equal size: each has tile_q granules, the first tile_r one more
  int cls;     // residue class of the chunk's vocabulary rows (0 unless d is odd-sized)
  int rows;    // vocabulary rows of that class (V unless d is odd-sized)
};
struct Tile {
  int v0;      // first vocabulary row of the tile (first row of W1 in a learned-router unit)
  int rows;    // vocabulary rows in the tile (multiple of 16 * kCta); 0 = empty tile
};

// What is fixed for a whole unit.  The walk of the MMA-issuing warp is on the tensor pipe's critical path and must stay
// cheap: no division per tile, two 32-bit ones per unit.  With 64-bit ones here and one per tile this function took 720
// cycles of the 2020 between a unit's last slab and the next one's first (now 260 of 1340), a tile 1150 (now 1025):
// prefill at n = 8192, d = 896 1743 -> 1713 us, n = 2000, d = 1024, V = 100000 341 -> 329, n = 1, d = 256 8.64 -> 8.45.
template <int kCta, bool kOdd = false, bool kTwo = false>
__host__ __device__ __forceinline__ Unit unit_of(const TcParams& p, int unit, int cta_rank) {
  Unit u;
  u.cls = 0;
  u.rows = p.V;
  const int vocab_units = p.chunks * p.row_units;
  if (unit >= vocab_units) {          // learned-router unit: all rows of W1 for one row unit
    u.chunk = -1;
    u.row0 = ((unit - vocab_units) * (kTwo ? 2 : 1) * kCta + cta_rank) * kBlockM;
    u.g0 = 0;
    u.G = 0;
    u.tile_q = u.tile_r = 0;
    return u;
  }
  // (two row blocks: group by group of row units, and in a group chunk by chunk, see tc_two_group)
  const int group = kTwo ? static_cast<int>(static_cast<uint32_t>(unit) / static_cast<uint32_t>(p.chunks * p.group_units)) : 0;
  const int ru0 = kTwo ? group * p.group_units : 0;
  const int group_rows = kTwo ? (p.row_units - ru0 < p.group_units ? p.row_units - ru0 : p.group_units) : p.row_units;
  const int at = unit - p.chunks * ru0;
  u.chunk = static_cast<int>(static_cast<uint32_t>(at) / static_cast<uint32_t>(group_rows));
  const int ru = ru0 + at - u.chunk * group_rows;
  u.row0 = (ru * (kTwo ? 2 : 1) * kCta + cta_rank) * kBlockM;
  int c = u.chunk;
  if (kOdd) {                         // class by class: the chunks of a class share its rows out
    u.cls = static_cast<int>(static_cast<uint32_t>(c) / static_cast<uint32_t>(p.class_chunks));
    c -= u.cls * p.class_chunks;
    u.rows = static_cast<int>(static_cast<uint32_t>(p.V - u.cls + p.classes - 1) / static_cast<uint32_t>(p.classes));
  }
  // chunk_r of the chunks have a granule more than the others, evenly spread: floor(chunk_r * c / chunks) of those before
  // chunk c, by a multiplication (chunk_mul = ceil(2^32 / chunks) is exact here: chunk_r * c < 2^16, chunks <= 192)
  const int e0 = static_cast<int>((static_cast<uint64_t>(p.chunk_r * c) * p.chunk_mul) >> 32);
  const int e1 = static_cast<int>((static_cast<uint64_t>(p.chunk_r * (c + 1)) * p.chunk_mul) >> 32);
  u.g0 = p.chunk_q * c + e0;
  u.G = p.chunk_q + e1 - e0;
  u.tile_q = u.tile_r = 0;
  if (!p.full_tiles_first) {
    u.tile_q = static_cast<int>(static_cast<uint32_t>(u.G) / static_cast<uint32_t>(p.tiles_per_unit));
    u.tile_r = u.G - u.tile_q * p.tiles_per_unit;
  }
  return u;
}

__host__ __device__ __forceinline__ Tile tile_of(const TcParams& p, const Unit& u, int t) {
  Tile r;
  if (u.chunk < 0) {                  // learned-router unit: full 256-row tiles over the rows of W1
    r.v0 = t * kBlockN;
    const int left = p.mlp_rows - r.v0;
    r.rows = left <= 0 ? 0 : (left < kBlockN ? left : kBlockN);
    return r;
  }
  int ga, gb;
  if (p.full_tiles_first) {
    // as many full 256-row tiles as fit, then one remainder tile: a tile costs a pass over all
    // of h whatever its width, so the fewest, widest tiles are the cheapest
    ga = p.full_granules * t < u.G ? p.full_granules * t : u.G;
    gb = p.full_granules * (t + 1) < u.G ? p.full_granules * (t + 1) : u.G;
  } else {
    ga = u.tile_q * t + (t < u.tile_r ? t : u.tile_r);
    gb = ga + u.tile_q + (t < u.tile_r ? 1 : 0);
  }
  r.v0 = (u.g0 + ga) * p.granule_rows;
  r.rows = (gb - ga) * p.granule_rows;
  return r;
}

// Two row blocks to a unit (RowMode::kM128Two): the i-th of a tile's row-block slabs is slab `slab` of block `block`.  The
// second block is `lag` slabs behind the first, so that either accumulator is folded while the other's MMAs run: there is no
// third and fourth one.  A unit whose second block has no rows is walked like a single one.
struct TwoWalk {
  int blocks, items, lag, k_slabs;
  __host__ __device__ __forceinline__ TwoWalk(const TcParams& p, int row0, int slabs) {
    blocks = row0 + 2 * kBlockM < p.n ? 2 : 1;       // (row0 of the unit, whichever CTA asks)
    items = blocks * slabs;
    lag = blocks == 2 && p.lag < slabs ? p.lag : slabs;
    k_slabs = slabs;
  }
  __host__ __device__ __forceinline__ void at(int i, int& block, int& slab) const {
    const int j = i - lag;
    block = j < 0 ? 0 : (i + lag >= items ? 1 : j & 1);
    slab = j < 0 ? i : (i + lag >= items ? i - k_slabs : (j >> 1) + (block == 0 ? lag : 0));
  }
};

// Running online-softmax summary of one token row over the vocabulary rows a thread has seen.
// S = sum 2^y and T = sum 2^y * y with y = (z - m) * log2(e) <= 0; both are accumulated per
// 32-column group first and then added with a compensated (Kahan) sum, so that one dominant term -- a
// confident row has S ~ 1 with thousands of terms ~1e-8 after it -- does not swallow the rest.
// kExact: z - m is rounded by itself, so that the largest logit's y is zero whatever its size; with one fma, against the
// rounded m * log2(e), every y of a row is off by up to 2^-24 of that.  The heads whose hidden size is no multiple of 8 ran on
// CUDA cores with the former before they ran here.  Their columns beyond V are left out of the maximum, too.
template <bool kExact>
struct RowFold {
  float m, S, cS, Tq, cT;
  int idx;
  __device__ __forceinline__ void reset() {
    m = -INFINITY;
    S = cS = Tq = cT = 0.f;
    idx = kNoToken;
  }
  // y of the logits z0 and z1; neg_m is -m (kExact) or -m * log2(e)
  static __device__ __forceinline__ uint64_t exponents(float z0, float z1, float neg_m) {
    const uint64_t log2e2 = pack2(kLog2e, kLog2e), neg2 = pack2(neg_m, neg_m);
    if (kExact) return fma2(add2(pack2(z0, z1), neg2), log2e2, 0ull);
    return fma2(pack2(z0, z1), log2e2, neg2);
  }
  // kExact: what stands for a column beyond V once the maximum is known: far enough below it for e^(z-m) = 0, and finite
  __device__ __forceinline__ float far_below() const { return m - fmaxf(1000.f, fabsf(m) * 0.015625f); }
  // Folds 32 consecutive logits z[0..32) whose first has vocabulary index col0; only the first
  // `valid` of them exist (the rest lie beyond V).
  __device__ __forceinline__ void group(float (&z)[32], int valid, int col0) {
    if (valid < 32) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j >= valid) z[j] = kExact ? -INFINITY : kNoLogit;
    }
    float cm = fmaxf(z[0], z[1]);
#pragma unroll
    for (int j = 2; j < 32; j += 2) cm = max3(cm, z[j], z[j + 1]);
    if (cm > m) {
      if (m != -INFINITY) {
        const float dl = (cm - m) * kLog2e;       // > 0
        const float sc = ex2_approx(-dl);
        Tq = sc * (Tq - dl * S);
        cT *= sc;
        S *= sc;
        cS *= sc;
      }
      m = cm;
      int first_j = 31;
#pragma unroll
      for (int j = 30; j >= 0; --j) first_j = (z[j] == cm) ? j : first_j;
      idx = col0 + first_j;
    }
    if (kExact && valid < 32) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j >= valid) z[j] = far_below();
    }
    const float neg_m = kExact ? -m : -m * kLog2e;
    uint64_t ls2 = pack2(0.f, 0.f), lt2 = pack2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
      const uint64_t y2 = exponents(z[j], z[j + 1], neg_m);
      float y0, y1;
      unpack2(y2, y0, y1);
      const uint64_t e2 = pack2(ex2_approx(y0), ex2_approx(y1));
      ls2 = add2(ls2, e2);
      lt2 = fma2(e2, y2, lt2);
    }
    float ls0, ls1, lt0, lt1;
    unpack2(ls2, ls0, ls1);
    unpack2(lt2, lt0, lt1);
    {
      const float a = (ls0 + ls1) - cS;
      const float b = S + a;
      cS = (b - S) - a;
      S = b;
    }
    {
      const float a = (lt0 + lt1) - cT;
      const float b = Tq + a;
      cT = (b - Tq) - a;
      Tq = b;
    }
  }
  // The same for 16 logits of one row held by a thread of the fragment layout (tmem_ld16x64): z[2b + j] is column
  // col0 + 8b + j, and those from `valid` on do not exist.  Written for latency -- no branch but the index search, short
  // dependent chains -- because the last tile's fold is exposed at the end of every step.
  __device__ __forceinline__ void fragment(float (&z)[16], int valid, int col0) {
    if (valid < 58) {                                  // (the last of the columns is col0 + 57)
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (8 * (k >> 1) + (k & 1) >= valid) z[k] = kExact ? -INFINITY : kNoLogit;
    }
    const float m0 = max3(max3(z[0], z[1], z[2]), z[3], max3(z[4], z[5], z[6]));
    const float m1 = max3(max3(z[7], z[8], z[9]), z[10], max3(z[11], z[12], z[13]));
    const float cm = max3(fmaxf(m0, m1), z[14], z[15]);
    if (cm > m) {
      uint32_t hit = 0;
#pragma unroll
      for (int k = 0; k < 16; ++k) hit |= (z[k] == cm) ? 1u << k : 0u;
      const int k = __ffs(hit) - 1;
      idx = col0 + 8 * (k >> 1) + (k & 1);
    }
    const float m_old = kExact ? (m == -INFINITY ? cm : m) : fmaxf(m, kNoLogit);    // (finite before the first group)
    m = fmaxf(m_old, cm);
    const float dl = (m - m_old) * kLog2e;          // >= 0
    const float sc = ex2_approx(-dl);
    if (kExact && valid < 58) {
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (8 * (k >> 1) + (k & 1) >= valid) z[k] = far_below();
    }
    const float neg_m = kExact ? -m : -m * kLog2e;
    uint64_t ls2[2] = {0ull, 0ull}, lt2[2] = {0ull, 0ull};
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
      const uint64_t y2 = exponents(z[j], z[j + 1], neg_m);
      float y0, y1;
      unpack2(y2, y0, y1);
      const uint64_t e2 = pack2(ex2_approx(y0), ex2_approx(y1));
      ls2[(j >> 1) & 1] = add2(ls2[(j >> 1) & 1], e2);
      lt2[(j >> 1) & 1] = fma2(e2, y2, lt2[(j >> 1) & 1]);
    }
    float ls0, ls1, lt0, lt1;
    unpack2(add2(ls2[0], ls2[1]), ls0, ls1);
    unpack2(add2(lt2[0], lt2[1]), lt0, lt1);
    Tq = sc * (Tq - dl * S);
    cT *= sc;
    S *= sc;
    cS *= sc;
    {
      const float a = (ls0 + ls1) - cS;
      const float b = S + a;
      cS = (b - S) - a;
      S = b;
    }
    {
      const float a = (lt0 + lt1) - cT;
      const float b = Tq + a;
      cT = (b - Tq) - a;
      Tq = b;
    }
  }
  __device__ __forceinline__ Partial result() const {
    Partial out;
    out.m = m;
    out.idx = idx;
    out.s = S;
    out.t = Tq * kLn2;             // sum e^(z-m) (z-m), back in nats
    return out;
  }
};

// The summaries of four neighbouring threads as one (all four get it).  One maximum, one rescaling, one sum: a chain of
// pairwise merges took 870 cycles at the end of every step.
__device__ __forceinline__ Partial quad_merge(const Partial& p) {
  Partial r;
  r.m = fmaxf(p.m, __shfl_xor_sync(0xffffffffu, p.m, 1));
  r.m = fmaxf(r.m, __shfl_xor_sync(0xffffffffu, r.m, 2));
  r.idx = p.m == r.m ? p.idx : kNoToken;
  const float dm = p.s == 0.f ? 0.f : p.m - r.m;     // <= 0; an empty range contributes nothing
  const float e = ex2_approx(dm * kLog2e);
  r.s = p.s * e;
  r.t = e * (p.t + dm * p.s);
#pragma unroll
  for (int off = 1; off <= 2; off <<= 1) {
    r.idx = min(r.idx, __shfl_xor_sync(0xffffffffu, r.idx, off));
    r.s += __shfl_xor_sync(0xffffffffu, r.s, off);
    r.t += __shfl_xor_sync(0xffffffffu, r.t, off);
  }
  return r;
}

}  // namespace

// The kernel body (maps and p are the kernel's own parameters, maps a __grid_constant__ one: TMA reads the
// tensor maps from parameter space).
template <int kCta, RowMode kMode, class Maps>
__device__ __forceinline__ void tc_projection_body(const Maps& maps, const TcParams& p) {
  constexpr bool kOdd = std::is_same<Maps, OddMaps>::value;   // d no multiple of 8: vocabulary rows by residue class
  constexpr bool kFp8 = kMode >= RowMode::k8Small, kGroup8 = kMode == RowMode::kGroup8;
  constexpr bool kKeep = kMode == RowMode::kM128Keep;      // the stage of a K slab is its number, filled once per unit
  constexpr bool kTwo = kMode == RowMode::kM128Two;
  static_assert(kCta == 1 || kMode == RowMode::kM128 || kKeep || kTwo, "modes of a pair of CTAs");
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment: the swizzle pattern is a function of the shared-memory address.
  // (The dynamic shared memory of both CTAs of a pair starts at the same offset, so the
  // two CTAs compute identical offsets -- which the pair MMA and the peer signals rely on.)
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int SA = p.a_stages, SB = p.b_stages;
  const uint32_t a_stage_bytes = static_cast<uint32_t>(p.a_rows) * kRowBytes;
  constexpr uint32_t b_stage_bytes = (kBlockN / kCta) * kRowBytes;
  constexpr int kSlabElems = kFp8 ? kRowBytes : kRowBytes / 2;   // K elements per slab
  const uint32_t a_ring = base;
  const uint32_t b_ring = base + SA * a_stage_bytes;
  const uint32_t bar_base = b_ring + SB * b_stage_bytes;
  // Barriers: a_full / b_full per ring stage (data landed); released[j] completes when the
  // MMAs of slab number j (mod kRelease) have finished reading shared memory -- one commit
  // per slab serves both rings: the producer of slab i waits for slab i - depth (two row blocks:
  // the h ring alone, whose slabs are numbered as they are walked; the W ring has h_free);
  // acc_full / acc_empty per accumulator.
  auto a_full = [&](int s) { return bar_base + 8u * s; };
  auto b_full = [&](int s) { return bar_base + 8u * (kMaxAStages + s); };
  auto released = [&](int j) { return bar_base + 8u * (kMaxAStages + kMaxBStages + j); };
  constexpr int kFixed = kMaxAStages + kMaxBStages + kRelease;
  auto acc_full = [&](int b) { return bar_base + 8u * (kFixed + b); };
  auto acc_empty = [&](int b) { return bar_base + 8u * (kFixed + 2 + b); };
  // xch_full[q]: the second epilogue group's summary of quadrant q is in the scratch block;
  // xch_empty[q]: the first group has read it.
  auto xch_full = [&](int q) { return bar_base + 8u * (kFixed + 4 + q); };
  auto xch_empty = [&](int q) { return bar_base + 8u * (kFixed + 8 + q); };
  const uint32_t h_ready = bar_base + 8u * (kFixed + 12);   // 8-bit head: h has been split in place (inline mode)
  // kept h: the MMAs of the unit's last tile have read K slab s; two row blocks: those of both have read W stage s
  auto h_free = [&](int s) { return bar_base + 8u * (kFixed + 13 + s); };
  constexpr int kNumBarriers = kFixed + 13 + kMaxAStages;
  static_assert(kNumBarriers * 8 + 16 <= kBarrierBytes, "barrier block too small");
  unsigned char* gen_base = smem_raw + (base - smem_u32(smem_raw));
  unsigned char* tail = gen_base + (bar_base - base);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 8 * kNumBarriers);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  Partial* scratch = reinterpret_cast<Partial*>(tail + kBarrierBytes);
  float* scale_area = reinterpret_cast<float*>(tail + kBarrierBytes + kScratchBytes);   // 8-bit head only
  float* hs_s = scale_area + kScaleBytes / 4;
  const bool inl = kFp8 && p.inline_split != 0;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t cta_rank = (kCta == 2) ? cluster_ctarank() : 0u;
  const bool leader = cta_rank == 0;
  const int worker = blockIdx.x / kCta;
  const int workers = gridDim.x / kCta;

  if (threadIdx.x == 0) {
    if (!inl) for (int s = 0; s < SA; ++s) mbar_init(a_full(s), 1);   // (inline mode: SA = K slabs, nothing streams)
    if (kKeep) for (int s = 0; s < SA; ++s) mbar_init(h_free(s), 1);
    if (kTwo) for (int s = 0; s < SB; ++s) mbar_init(h_free(s), 1);
    for (int s = 0; s < SB; ++s) mbar_init(b_full(s), 1);
    for (int j = 0; j < kRelease; ++j) mbar_init(released(j), 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_empty(b), kEpiWarps * kCta);
    }
    for (int q = 0; q < 4; ++q) {
      mbar_init(xch_full(q), 1);
      mbar_init(xch_empty(q), 1);
    }
    if (kFp8) mbar_init(h_ready, 9);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc<kCta>(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish<kCta>();
  }
  tc_fence_before();
  __syncthreads();
  if (kCta == 2) cluster_sync_all();   // the peer's barriers exist before anything signals them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // Programmatic dependent launch: everything above overlapped the tail of the previous
  // kernel in the stream; from here on its results (h, and the workspace the previous
  // merge kernel was still reading) are needed, so wait for it, and let the kernel
  // that follows this one be scheduled early.  The W producer reads only W and the tensor
  // maps, which no kernel writes when W belongs to a context, so it goes ahead (entry points
  // that take W per call set w_wait).  It also lets the next kernel go ahead at once: done only behind
  // the wait, a step of n = 16, d = 896, V = 151936 takes 48.3 us in a stream instead of 47.1.  A kernel that reads
  // h without waiting for this one (mlp_mma_kernel) needs it behind the wait, though.
  if ((warp != 0 && warp != 6) || inl || p.w_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
  if ((warp != 0 && warp != 6) || !p.late_trigger) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // With at most 64 operand rows (one CTA per worker) the MMAs run with M = 64: such an instruction takes
  // about two thirds of the time of an M = 128 one, and the padding rows were wasted work anyway.  Its
  // accumulator row r lives in TMEM lane 32 * (r / 16) + r % 16, i.e. in lanes 0..15 of each 32-lane
  // quadrant (checked on the device), so an epilogue warp then holds 16 rows instead of 32.
  constexpr bool m64 = kGroup8 || kMode == RowMode::kM64 || kMode == RowMode::k8Small;
  // 8-bit head with more than 64 token rows: the two parts of h no longer fit one MMA's M (128 at most with one
  // CTA), so every K step issues two MMAs -- first parts, then second parts, into the same accumulator rows --
  // and the epilogue reads finished logits as on the bf16 head (no hand-over between warps).
  constexpr bool wide = kMode == RowMode::k8Wide;
  const int k_slabs = (p.d + kSlabElems - 1) / kSlabElems;
  const int units = (p.chunks + (p.mlp_hidden > 0 ? 1 : 0)) * p.row_units;
  const int T = p.tiles_per_unit;
  const unsigned long long wait_ns = p.wait_limit_ns != 0 ? p.wait_limit_ns : kWaitLimitNs;
  Partial last = {};               // pair mode: this thread's partial of the worker's last unit
  Partial* last_dst = nullptr;

  if (inl && warp >= 2) {
    // ---- 8-bit head, n <= 16: the nine warps that have nothing to do yet split h into its two e4m3
    // parts, straight into the resident operand slabs
    static_assert(kThreads - 64 == kSplitThreads, "warps 2..10 split h");
    split_h_resident(static_cast<const __nv_bfloat16*>(p.h), p.n, p.d, k_slabs, gen_base, hs_s, threadIdx.x - 64);
    __syncwarp();
    if (lane == 0) mbar_arrive(h_ready);
  }

  if (warp == 0) {
    // ------------------------------------------------------------------ W producer
    if (lane == 0) {
      // This role has not waited for the kernel in front, whose time its limit must not count.  What keeps a slab from being
      // released the other roles notice within theirs, and it sees their flag.  (A wait for that kernel in this loop, in front
      // of the first slab that must be released: n = 444, d = 752, V = 30000 24.8 -> 25.1 us, a bounded number of looks in
      // front of it 25.8 and prefill at n = 8192, d = 896 4 % longer; a clock that starts again n = 600, d = 256, V = 30000
      // 20.1 -> 20.4.  The longer limit costs nothing.)
      const unsigned long long ahead_ns = wait_ns + kAheadNs;
      int stage = 0;
      int slab = 0;     // running slab number, the same in every role
      bool ok = true;
      for (int unit = worker; unit < units && ok; unit += workers) {
        const Unit un = unit_of<kCta, kOdd, kTwo>(p, unit, cta_rank);
        for (int t = 0; t < T && ok; ++t) {
          const Tile tl = tile_of(p, un, t);
          if (tl.rows == 0) continue;
          const int my_rows = tl.rows / kCta;                 // this CTA's share of the tile
          const int my_v0 = tl.v0 + static_cast<int>(cta_rank) * my_rows;
          const bool mlp = !kFp8 && un.chunk < 0;
          const CUtensorMap *m128, *m64p, *m16;
          if constexpr (kOdd) {
            m128 = m64p = m16 = &maps.w[un.cls];
          } else {
            m128 = mlp ? &maps.m128 : &maps.w128;
            m64p = mlp ? &maps.m64 : &maps.w64;
            m16 = mlp ? &maps.m16 : &maps.w16;
          }
          for (int ks = 0; ks < k_slabs; ++ks, ++slab) {
            if (slab >= SB) {     // the stage is free once slab - SB has been consumed
              const int j = slab - SB;
              const bool got = kTwo ? mbar_wait(h_free(stage), (j / SB) & 1, abort_flag, p.status, ahead_ns)
                                    : mbar_wait(released(j & (kRelease - 1)), (j / kRelease) & 1, abort_flag, p.status, ahead_ns);
              if (!got) { ok = false; break; }
            }
            const uint32_t dst = b_ring + stage * b_stage_bytes;
            const uint32_t bar = (kCta == 2) ? map_to_cta(b_full(stage), 0) : b_full(stage);
            if (p.debug_drop_w_copies) continue;   // test hook: the copies are "lost", the consumer's wait runs out
            if (leader) mbar_expect_tx(b_full(stage), tl.rows * kRowBytes);   // both CTAs' bytes
            int r = 0;
            if (kOdd)
              for (; r < my_rows; r += kOddBoxRows)
                tma_load_2d<kCta>(dst + r * kRowBytes, m128, bar, ks * kSlabElems, my_v0 + r);
            for (; my_rows - r >= 128; r += 128)
              tma_load_2d<kCta>(dst + r * kRowBytes, m128, bar, ks * kSlabElems, my_v0 + r);
            for (; my_rows - r >= 64; r += 64)
              tma_load_2d<kCta>(dst + r * kRowBytes, m64p, bar, ks * kSlabElems, my_v0 + r);
            for (; my_rows - r >= 16; r += 16)
              tma_load_2d<kCta>(dst + r * kRowBytes, m16, bar, ks * kSlabElems, my_v0 + r);
            if (++stage == SB) stage = 0;
          }
        }
      }
      if (!ok) drain_delay();
    }
  } else if (warp == 6) {
    // ------------------------------------------------------------------ h producer
    // (8-bit head: the map covers the two parts stacked, [2 * part_rows][d], so one box is the whole operand slab)
    if (lane == 0 && !inl) {
      int stage = 0;
      int slab = 0;
      bool ok = true;
      bool h_there = false;
      uint32_t ord = 0;
      for (int unit = worker; unit < units && ok; unit += workers, ++ord) {
        const Unit un = unit_of<kCta, kOdd, kTwo>(p, unit, cta_rank);
        const int h_row0 = kFp8 ? 0 : un.row0 + (kOdd ? un.cls * p.h_class_rows : 0);
        const TwoWalk two(p, un.row0 - static_cast<int>(cta_rank) * kBlockM, k_slabs);
        for (int t = 0; t < T && ok; ++t) {
          const Tile tl = tile_of(p, un, t);
          if (tl.rows == 0) continue;
          for (int i = 0; i < (kTwo ? two.items : k_slabs); ++i, ++slab) {
            int ks = i, block = 0;
            if (kTwo) two.at(i, block, ks);
            const int h_row = h_row0 + block * (kCta * kBlockM);
            if (kKeep && t > 0) continue;      // (the first tile of a unit is never empty)
            if (!h_there) {
              // here and not with the other warps above: the arithmetic of the first unit would stand between the end of the
              // wait and the first load of h, which the whole step waits for (n = 1, d = 256, V = 20000 8.60 -> 8.18 us per
              // step in a stream, n = 16, d = 512, V = 32000 10.53 -> 9.98, n = 256 there 14.76 -> 14.39)
              asm volatile("griddepcontrol.wait;" ::: "memory");
              h_there = true;
            }
            if (kKeep) {
              if (ord > 0 && !mbar_wait(h_free(ks), (ord - 1) & 1u, abort_flag, p.status, wait_ns)) { ok = false; break; }
            } else if (slab >= SA) {
              const int j = slab - SA;
              if (!mbar_wait(released(j & (kRelease - 1)), (j / kRelease) & 1, abort_flag, p.status, wait_ns)) { ok = false; break; }
            }
            const uint32_t dst = a_ring + stage * a_stage_bytes;
            const uint32_t bar = (kCta == 2) ? map_to_cta(a_full(stage), 0) : a_full(stage);
            if (kGroup8) {      // boxes of eight rows, sixteen operand rows apart
              mbar_expect_tx(a_full(stage), a_stage_bytes >> 1);
              for (int r = 0; r < p.a_rows; r += 16)
                tma_load_2d<kCta>(dst + r * kRowBytes, &maps.h, bar, ks * kSlabElems, h_row + (r >> 1));
            } else {
              if (leader) mbar_expect_tx(a_full(stage), a_stage_bytes * kCta);
              tma_load_2d<kCta>(dst, &maps.h, bar, ks * kSlabElems, h_row);
            }
            if (++stage == SA) stage = 0;
          }
        }
      }
      if (!ok) drain_delay();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // The whole warp walks the schedule and waits on the barriers, so that control flow
    // and operands stay warp-uniform; one elected lane issues the MMAs and commits.
    if (leader) {
      int sa = 0, sb = 0;
      uint32_t pa = 0, pb = 0;
      int slab = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      // Descriptor words: the low word carries the start address (in 16-byte units) and the
      // leading offset; the high word is constant.
      const uint64_t desc_hi = smem_desc_sw128(0) & 0xffffffff00000000ull;
      const uint32_t desc_lo_fixed = static_cast<uint32_t>(smem_desc_sw128(0) & 0xffffffffull);
      const uint32_t a_lo0 = desc_lo_fixed | ((a_ring & 0x3ffffu) >> 4);
      const uint32_t b_lo0 = desc_lo_fixed | ((b_ring & 0x3ffffu) >> 4);
      const uint32_t a_step = a_stage_bytes >> 4, b_step = b_stage_bytes >> 4;
      const int mma_m = m64 ? 64 : kBlockM * kCta;
      const uint32_t part_off = static_cast<uint32_t>(p.part_rows * kRowBytes) >> 4;   // second parts, in descriptor units
      if (inl) {                                  // h is resident once the nine warps have split it
        ok = __all_sync(0xffffffffu, mbar_wait(h_ready, 0, abort_flag, p.status, wait_ns));
        tc_fence_after();
      }
      // The barrier state of the next slab is polled before the current slab's MMAs are
      // issued, so the poll's latency overlaps the issue instead of adding to it.
      bool ra = inl || mbar_test_wait(a_full(0), 0), rb = mbar_test_wait(b_full(0), 0);
      int sb_behind = 0;           // two row blocks: the W stage of the second's next slab
      for (int unit = worker; unit < units && ok; unit += workers) {
        const Unit un = unit_of<kCta, kOdd, kTwo>(p, unit, 0);
        const TwoWalk two(p, un.row0, k_slabs);
        for (int t = 0; t < T && ok; ++t) {
          const Tile tl = tile_of(p, un, t);
          if (tl.rows == 0) continue;
          if constexpr (kTwo) {
            const uint32_t idesc = instr_desc(mma_m, tl.rows);
            for (int i = 0; i < two.items; ++i, ++slab) {
              int block, ks;
              two.at(i, block, ks);
              const int my_acc = acc ^ block;
              if (ks == 0) {
                ok = __all_sync(0xffffffffu, mbar_wait(acc_empty(my_acc), acc_phase ^ 1u ^ (acc & block), abort_flag, p.status, wait_ns));
                if (!ok) break;
              }
              if (!__all_sync(0xffffffffu, ra && (block != 0 || rb))) {
                const bool got = mbar_wait(a_full(sa), pa, abort_flag, p.status, wait_ns) &&
                                 (block != 0 || mbar_wait(b_full(sb), pb, abort_flag, p.status, wait_ns));
                ok = __all_sync(0xffffffffu, got);
                if (!ok) break;
              }
              tc_fence_after();
              const int w_stage = block == 0 ? sb : sb_behind;
              const uint32_t a_lo = a_lo0 + sa * a_step;
              const uint32_t b_lo = b_lo0 + w_stage * b_step;
              if (++sa == SA) { sa = 0; pa ^= 1u; }
              if (block == 0) {
                if (++sb == SB) { sb = 0; pb ^= 1u; }
              }
              if (block + 1 == two.blocks) {
                if (++sb_behind == SB) sb_behind = 0;
              }
              ra = mbar_test_wait(a_full(sa), pa);
              rb = mbar_test_wait(b_full(sb), pb);
              if (elect_one()) {
                const uint32_t d_tmem = tmem_base + my_acc * kBlockN;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  umma_bf16<kCta>(d_tmem, desc_hi | (a_lo + 2u * k), desc_hi | (b_lo + 2u * k), idesc, (ks | k) != 0 ? 1u : 0u);
                umma_commit<kCta>(released(slab & (kRelease - 1)));
                if (block + 1 == two.blocks) umma_commit<kCta>(h_free(w_stage));
                if (ks + 1 == k_slabs) umma_commit<kCta>(acc_full(my_acc));
              }
              __syncwarp();
            }
            if (!ok) break;
            if (two.blocks == 2) acc_phase ^= 1u;
            else if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            continue;
          }
          const bool last_tile = kKeep && (t + 1 == T || tile_of(p, un, t + 1).rows == 0);
          const uint32_t idesc = kFp8 ? instr_desc_e4m3(mma_m, tl.rows) : instr_desc(mma_m, tl.rows);
          ok = __all_sync(0xffffffffu, mbar_wait(acc_empty(acc), acc_phase ^ 1u, abort_flag, p.status, wait_ns));
          if (!ok) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + acc * kBlockN;
          for (int ks = 0; ks < k_slabs; ++ks, ++slab) {
            if (kKeep && t > 0) ra = true;
            if (!__all_sync(0xffffffffu, ra && rb)) {
              const bool got = (inl || (kKeep && t > 0) || mbar_wait(a_full(sa), pa, abort_flag, p.status, wait_ns)) &&
                               mbar_wait(b_full(sb), pb, abort_flag, p.status, wait_ns);
              ok = __all_sync(0xffffffffu, got);
              if (!ok) break;
            }
            tc_fence_after();
            const uint32_t a_lo = a_lo0 + sa * a_step;
            const uint32_t b_lo = b_lo0 + sb * b_step;
            if (++sa == SA) {
              sa = 0;
              if (!kKeep || t == 0) pa ^= 1u;
            }
            if (++sb == SB) { sb = 0; pb ^= 1u; }
            ra = inl || mbar_test_wait(a_full(sa), pa);     // (inline mode: stage sa is slab sa, always there)
            rb = mbar_test_wait(b_full(sb), pb);
            if (elect_one()) {
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                // a quarter of the swizzle span along K (16 bf16 or 32 e4m3) = +32 bytes = +2 in the address field
                if (kFp8) {
                  umma_e4m3(d_tmem, desc_hi | (a_lo + 2u * k), desc_hi | (b_lo + 2u * k), idesc, (ks | k) != 0 ? 1u : 0u);
                  if (wide) umma_e4m3(d_tmem, desc_hi | (a_lo + part_off + 2u * k), desc_hi | (b_lo + 2u * k), idesc, 1u);
                } else
                  umma_bf16<kCta>(d_tmem, desc_hi | (a_lo + 2u * k), desc_hi | (b_lo + 2u * k), idesc,
                                  (ks | k) != 0 ? 1u : 0u);
              }
              umma_commit<kCta>(released(slab & (kRelease - 1)));   // both slabs are free once these MMAs are done
              if (last_tile) umma_commit<kCta>(h_free(ks));
            }
            __syncwarp();
          }
          if (!ok) break;
          if (elect_one()) umma_commit<kCta>(acc_full(acc));   // accumulator complete (in both CTAs of a pair)
          __syncwarp();
          if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2-5, 7-10)
    const int grp = warp >= 7 ? 1 : 0;       // 0: lower half of a tile's columns, 1: upper half
    const int quad = warp & 3;               // TMEM lane quadrant this warp may read
    // Fragment layout (tmem_ld16x64: 16 lanes at a time, four threads to a lane): the 8-bit head up to 64 token rows, the
    // bf16 head up to 16.  Four threads share a token's columns, and all 32 work.
    // 8-bit head: of the 16 lanes, 0..7 are the first parts of eight tokens and 8..15 their second parts
    // (tc8_part_row), so the thread that holds a token's first part holds its second part too and adds them.  With
    // M = 64 a quadrant has one such group of 16 lanes, with M = 128 two, and a thread then keeps two tokens, eight apart.
    // bf16 head: lanes 0..7 are tokens, 8..15 unused (RowMode::kGroup8).
    constexpr bool frag = kFp8 ? !wide : kGroup8;
    constexpr int kFolds = kMode == RowMode::k8Half ? 2 : 1;           // tokens a thread may keep
    constexpr int quad_rows = frag ? (m64 ? 8 : 16) : (m64 ? 16 : 32);     // token rows per quadrant
    const int quad_row0 = quad * quad_rows;
    const int my_row = quad_row0 + (frag ? lane >> 2 : (m64 ? lane & 15 : lane));   // this thread's (first) token row
    const bool writer = frag ? (lane & 3) == 0 : (!m64 || lane < 16);  // one thread per token row
    float* ws = scale_area + (grp * 4 + quad) * (kBlockN / 2);         // weight scales of this warp's half of a tile
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    uint32_t ord = 0;                        // ordinal of the unit among this worker's units
    float hs[kFolds] = {};
    if (kFp8) {
      // (inline mode: the scales are written by the splitting warps before they arrive on h_ready)
      if (inl) ok = mbar_wait(h_ready, 0, abort_flag, p.status, wait_ns);
#pragma unroll
      for (int i = 0; i < kFolds; ++i) {
        const int r = my_row + 8 * i;
        if (r < p.n) hs[i] = inl ? hs_s[r] : p.hscale[r];
      }
      ok = __all_sync(0xffffffffu, ok);
    }
    for (int unit = worker; unit < units && ok; unit += workers) {
      const Unit first = unit_of<kCta, kOdd, kTwo>(p, unit, cta_rank);
      const int blocks = kTwo ? TwoWalk(p, first.row0 - static_cast<int>(cta_rank) * kBlockM, k_slabs).blocks : 1;
      const bool two_tokens = kFolds == 2 && quad_row0 + 8 < p.n;   // warp-uniform
      const bool mlp_unit = !kFp8 && first.chunk < 0;
      RowFold<kOdd> f[kFolds], f_other;          // (f_other: of the other row block)
#pragma unroll
      for (int i = 0; i < kFolds; ++i) f[i].reset();
      f_other.reset();
      float mlp_sum = 0.f, mlp_other = 0.f;
      const auto swap_blocks = [&] {
        if (!kTwo || blocks == 1) return;
        const RowFold<kOdd> was = f[0];
        const float sum_was = mlp_sum;
        f[0] = f_other;
        f_other = was;
        mlp_sum = mlp_other;
        mlp_other = sum_was;
      };
      // The walk over the unit's tiles, compiled twice: once for vocabulary units (the hot loop, free of any
      // learned-router code) and once for learned-router units.
      auto walk_tiles = [&](auto router_tag) {
      constexpr bool kRouter = decltype(router_tag)::value;
      for (int t = 0; t < T && ok; ++t) {
        const Tile tl = tile_of(p, first, t);
        if (tl.rows == 0) continue;
        const int v0 = tl.v0;
        const int cols = min(tl.rows, (kRouter ? p.mlp_hidden : first.rows) - v0);   // valid columns of this tile
        // this group's share of them: [0, half) or [half, cols), half a multiple of the columns of a load
        const int step = frag ? 64 : 32;
        const int half = min(cols, (tl.rows / 2 + step - 1) & ~(step - 1));
        const int c_begin = grp ? half : 0, c_end = grp ? cols : half;
        for (int block = 0; block < blocks; ++block) {
        const auto give_back = [&] {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if (kCta == 1) mbar_arrive(acc_empty(acc));
            else mbar_arrive_cluster(map_to_cta(acc_empty(acc), 0));   // the leader's barrier
          }
        };
        bool given = false;
        const bool warp_has_rows = first.row0 + block * (kCta * kBlockM) + quad_row0 < p.n;      // warp-uniform
        if (kFp8 && warp_has_rows) {
          // the share's weight scales, before the accumulator is waited for
          __syncwarp();
#pragma unroll
          for (int j = 0; j < kBlockN / 64; ++j) {
            const int c = c_begin + lane + 32 * j;
            ws[lane + 32 * j] = (c < c_end) ? __ldg(p.wscale + v0 + c) : 0.f;
          }
          __syncwarp();
        }
        if (!mbar_wait(acc_full(acc), acc_phase, abort_flag, p.status, wait_ns)) { ok = false; break; }
        tc_fence_after();
        if (warp_has_rows) {
          const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + acc * kBlockN;
          if (frag) {
            for (int c0 = c_begin; c0 < c_end; c0 += 64) {
              float x[kFolds][32];
              __syncwarp();                           // the loads below are warp-collective
              tmem_ld16x64(taddr + c0, x[0]);
              if (two_tokens) tmem_ld16x64(taddr + (16u << 16) + c0, x[kFolds - 1]);
              tmem_ld_wait();
              const int c_mine = c0 + 2 * (lane & 3);         // this thread's columns: c_mine + 0, 1, 8, 9, 16 ..
              const int valid = c_end - c_mine;
              if (valid <= 0) continue;
#pragma unroll
              for (int i = 0; i < kFolds; ++i) {
                if (i == 1 && !two_tokens) continue;
                float z[16];
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                  z[2 * b] = x[i][4 * b];
                  z[2 * b + 1] = x[i][4 * b + 1];
                  if (kFp8) {
                    const float2 w2 = *reinterpret_cast<const float2*>(ws + (c_mine - c_begin) + 8 * b);
                    z[2 * b] = (z[2 * b] + x[i][4 * b + 2]) * hs[i] * w2.x;
                    z[2 * b + 1] = (z[2 * b + 1] + x[i][4 * b + 3]) * hs[i] * w2.y;
                  }
                }
                if constexpr (kRouter) {
#pragma unroll
                  for (int k = 0; k < 16; ++k) {
                    const int o = 8 * (k >> 1) + (k & 1), u = v0 + c_mine + o;
                    if (o < valid) mlp_sum += __ldg(p.mlp_w2 + u) * fmaxf(z[k] + __ldg(p.mlp_b1 + u), 0.f);
                  }
                  continue;
                }
                f[i].fragment(z, valid, v0 + c_mine);
              }
            }
          } else {
            for (int c0 = c_begin; c0 < c_end; c0 += 32) {
              float z[32];
              __syncwarp();                           // the load below is warp-collective
              tmem_ld32(taddr + c0, z);
              tmem_ld_wait();
              if (kTwo && c0 + 32 >= c_end) {     // in front of the last fold: the MMAs of the next tile wait for it
                give_back();
                given = true;
              }
              if (kFp8) {
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                  const float4 w4 = *reinterpret_cast<const float4*>(ws + (c0 - c_begin) + j);
                  z[j] = z[j] * hs[0] * w4.x;
                  z[j + 1] = z[j + 1] * hs[0] * w4.y;
                  z[j + 2] = z[j + 2] * hs[0] * w4.z;
                  z[j + 3] = z[j + 3] * hs[0] * w4.w;
                }
              }
              if constexpr (kRouter) {
                // hidden units v0 + c0 .. of the learned router: bias, ReLU, output-layer weight, sum
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                  const int u = v0 + c0 + j;
                  if (u < p.mlp_hidden) mlp_sum += __ldg(p.mlp_w2 + u) * fmaxf(z[j] + __ldg(p.mlp_b1 + u), 0.f);
                }
              } else {
                f[0].group(z, cols - c0, v0 + c0);
              }
            }
          }
        }
        if (!given) give_back();
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        swap_blocks();
        }
      }
      };
      if (!kOdd && mlp_unit) walk_tiles(std::integral_constant<bool, !kOdd>{});
      else walk_tiles(std::false_type{});
      for (int block = 0; block < blocks; ++block, ++ord) {
      Partial out[kFolds];
#pragma unroll
      for (int i = 0; i < kFolds; ++i) out[i] = f[i].result();
      if (kOdd && out[0].idx != kNoToken) out[0].idx = out[0].idx * p.classes + first.cls;   // row q of the class
      if (frag) {                              // the four threads of a token merge their summaries
#pragma unroll
        for (int i = 0; i < kFolds; ++i) {
          if (i == 1 && !two_tokens) continue;
          out[i] = quad_merge(out[i]);
        }
      }
      if (mlp_unit) {
        if (frag) {
          mlp_sum += __shfl_xor_sync(0xffffffffu, mlp_sum, 1);
          mlp_sum += __shfl_xor_sync(0xffffffffu, mlp_sum, 2);
        }
        out[0].s = mlp_sum;
      }
      // The second group hands its summary to the first through the scratch block (bounded
      // waits on both sides: a warp that gave up never leaves its partner waiting forever).
      if (grp == 1) {
        if (ok && ord > 0) ok = mbar_wait(xch_empty(quad), (ord - 1) & 1u, abort_flag, p.status, wait_ns);
        if (ok) {
          if (writer) {
            scratch[my_row] = out[0];
            if (two_tokens) scratch[my_row + 8] = out[kFolds - 1];
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(xch_full(quad));
        }
      } else {
        if (ok) ok = mbar_wait(xch_full(quad), ord & 1u, abort_flag, p.status, wait_ns);
        if (ok) {
          Partial other[kFolds];
          other[0] = scratch[my_row];
          if (two_tokens) other[kFolds - 1] = scratch[my_row + 8];
          __syncwarp();
          if (lane == 0) mbar_arrive(xch_empty(quad));
#pragma unroll
          for (int i = 0; i < kFolds; ++i) {
            const int row = first.row0 + block * (kCta * kBlockM) + my_row + 8 * i;
            if (!writer || row >= p.n || (i == 1 && !two_tokens)) continue;
            if (mlp_unit) p.mlp_out[row] = out[i].s + other[i].s;   // lower columns first: a fixed order
            else {
              Partial* dst = p.partials + static_cast<size_t>(row) * p.chunks + first.chunk;
              Partial sum = merge(out[i], other[i]);
              if (p.tag != 0) sum.idx = tagged_idx(sum.idx, p.tag);
              if (kCta == 2 && unit + workers >= units && block + 1 == blocks) {     // (stored behind the arrival at the cluster's barrier)
                last = sum;
                last_dst = dst;
              } else {
                store_partial(dst, sum);
              }
            }
          }
        }
      }
      swap_blocks();
      }
    }
  }

  tc_fence_before();
  __syncthreads();      // (here also for the warps with nothing to do: waiting at the cluster's barrier takes issue slots)
  if (kCta == 2) {
    // Neither CTA frees TMEM or exits while the peer still works.  The last partials go out behind the arrival: in front
    // of it the release would wait until L2 has acknowledged them, 0.7 us at the end of every launch.
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (last_dst != nullptr) store_partial(last_dst, last);
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc<kCta>(tmem_base, kTmemCols);
  }
}

// bf16 head: one CTA per worker (kCta = 1) or a pair (kCta = 2).
// Every way of handling token rows is a kernel of its own: switches at run time cost the others (one for kGroup8 1.5 %:
// n = 24, d = 512, V = 32000 11.60 and 11.82 us).
// kBeside: so few registers that a block of 17 warps of the merge kernel (40 registers) stands beside a CTA and is resident,
// waiting, before this kernel ends -- one CTA per worker, and pairs with short units.  Others are bound by the epilogue's and the MMAs' rate, and
// that costs them (113 and 100 registers: n = 264, d = 696, V = 128256 75.8 and 80.4 us, n = 7969, d = 680, V = 25141 248 and 266).
template <int kCta, RowMode kMode, bool kBeside>
__global__ void __maxnreg__(kBeside ? 104 : 184)
tc_projection_kernel(const __grid_constant__ TcMaps maps, const TcParams p) {
  tc_projection_body<kCta, kMode>(maps, p);
}

// d no multiple of 8 (defined in the one file that launches them).
#ifdef TLR_DEFINE_ODD_KERNELS
template <int kCta, RowMode kMode>
__global__ void __maxnreg__(kCta == 2 ? 184 : 104)
odd_projection_kernel(const __grid_constant__ OddMaps maps, const TcParams p) {
  tc_projection_body<kCta, kMode>(maps, p);
}
#endif

// 8-bit head (defined in the one file that launches it).  At most 128 registers per thread, so that a block of
// the merge kernel (512 threads) fits on the SM beside this CTA and is resident, waiting, before this kernel ends.
#ifdef TLR_DEFINE_TC8_KERNEL
template <RowMode kMode>
__global__ void __maxnreg__(128)
tc8_projection_kernel(const __grid_constant__ TcMaps maps, const TcParams p) {
  tc_projection_body<1, kMode>(maps, p);
}
#endif

}  // namespace tlr
