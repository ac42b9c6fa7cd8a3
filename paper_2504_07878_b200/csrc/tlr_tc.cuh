// Host/device interface of the tensor-core projection kernel (bf16 head and 8-bit head).
#pragma once

#include <cuda.h>

#include "tlr_common.cuh"

namespace tlr {

// How a projection kernel handles token rows.
enum class RowMode : int {
  kM128,      // bf16 head, more than 64 rows: MMA M = 128 (256 on a pair), one epilogue thread per row
  kM128Keep,  // the same on a pair, where all of a row unit's h fits beside the W ring: it is loaded once per unit
  kM128Two,   // the same on a pair, two row blocks of 256 to a unit: a slab of W is read by both while it is in shared memory
  kM64,       // bf16 head, 17..64 rows: M = 64, one thread per row
  kGroup8,    // bf16 head, up to 16 rows: M = 64, eight rows in every sixteen operand rows, four threads per row
  k8Small,    // 8-bit head, up to 32 rows: both parts through one MMA with M = 64, four threads per row
  k8Half,     // 8-bit head, 33..64 rows: M = 128, four threads per two rows
  k8Wide,     // 8-bit head, more than 64 rows: an MMA per part, M = 128, one thread per row
};

// Kernel shape for a given n (see tc_configure / tc8_configure).
struct TcConfig {
  int cta;          // 1: one CTA per worker (n <= 128); 2: a pair of CTAs per worker
  int a_rows;       // rows of an h slab held in shared memory (16..128); on the 8-bit head both parts of h stacked
  RowMode mode;
  int part_rows;    // 8-bit head: rows of one part (a_rows / 2); otherwise a_rows
  int lag;          // RowMode::kM128Two: how many slabs the second row block is behind the first
  int a_stages;     // depth of the h ring
  int b_stages;     // depth of the W ring
  int inline_split; // 8-bit head: 1 = n <= 16 and both parts of all of h fit in shared memory -- the kernel splits h
                    // itself at its start and keeps it resident (a_stages == number of K slabs); no split kernel runs
  int smem_bytes;   // dynamic shared memory per CTA
};

// Work decomposition for a given (n, V) on `workers` workers (see tc_plan).
struct TcPlan {
  int blocks;          // row blocks of 128 * cta rows in a unit (2: RowMode::kM128Two)
  int group_units;     // row units of a group (blocks == 2)
  int row_units;       // ceil(n / (128 * cta * blocks))
  int classes;         // residue classes of the vocabulary (1 unless d is odd-sized, see OddMaps)
  int chunks;          // vocabulary chunks == partials per row; a multiple of `classes`
  int granule_rows;    // a multiple of 16 * cta
  int granules;        // ceil(rows of a class / granule_rows)
  int tiles_per_unit;  // every unit is walked in this many tiles (<= 256 rows each)
  int full_tiles_first;  // 1: full 256-row tiles, then one remainder tile; 0: tiles of equal size
  long long passes;    // of the busiest worker: tiles times row blocks (pair mode)
  int mlp_rows;        // learned-router units: hidden width rounded up to the granule (0 = none); one such unit
                       // per row unit follows the vocabulary units
};

struct TcParams {
  int n, d, V;
  int row_units, chunks, tiles_per_unit, full_tiles_first, granule_rows;
  int group_units;                    // two row blocks to a unit: row units of a group (all groups but the last)
  int lag;                            // ... and how many slabs of a tile the second is behind the first
  int chunk_q, chunk_r;               // granules of a chunk: chunk_q, and one more in chunk_r of them (of a class)
  uint32_t chunk_mul;                 // ceil(2^32 / chunks of a class), 0 for one chunk
  int full_granules;                  // granules of a full tile
  int classes, class_chunks;          // odd-sized d only: residue classes, chunks per class (chunks == classes * class_chunks)
  int h_class_rows;                   // odd-sized d only: rows between the shifted copies of h
  int a_rows, part_rows, a_stages, b_stages;
  unsigned long long wait_limit_ns;   // 0 = the default limit of every barrier wait
  int debug_drop_w_copies;            // test hook: the W producer issues no copies
  int w_wait;                         // 1: W may have been written by the previous kernel in the stream, so the
                                      // W producer waits for it too (entry points that take W per call)
  int late_trigger;                   // 1: the next kernel may be scheduled only behind this one's own wait
  // learned router inside the launch (bf16 head): one extra unit per row unit over the rows of W1
  int mlp_hidden;                     // hidden width, 0 = no learned router in this launch
  int mlp_rows;                       // hidden width rounded up to the granule
  const float* mlp_b1;                // [mlp_hidden]
  const float* mlp_w2;                // [mlp_hidden]
  float* mlp_out;                     // [n]: sum_j w2_j relu(W1_j . h + b1_j)
  // 8-bit head
  int inline_split;
  const void* h;         // bf16 [n][d], read when inline_split
  const float* hscale;   // [n] power-of-two scale of every row of h (written by the split kernel)
  const float* wscale;   // [V] scale of every row of W
  Partial* partials;     // [n][chunks]
  uint32_t tag;          // not 0: they are tagged (tlr_common.cuh)
  uint32_t* status;
};

// The tensor maps one launch needs: h, W (boxes of 128, 64 and 16 rows) and, with a learned router, W1.
struct TcMaps {
  CUtensorMap h, w128, w64, w16, m128, m64, m16;
};

// Tensor maps when d is not a multiple of 8 ("odd-sized"): rows of W are then no multiple of 16 bytes apart, which TMA
// cannot address.  But C = 8 / gcd(d, 8) consecutive rows are, so the rows v = C q + r of one residue class r form a
// matrix with an addressable pitch.  Its first element lies s = (r d) mod 8 elements past a 16-byte boundary: the map
// of class r starts at that boundary, s elements early, and the class is multiplied by a copy of h shifted by s
// elements, whose first s are zero.  W stays where it is; only h is copied, C times (tlr_odd.cu).
constexpr int kMaxClasses = 8;
constexpr int kOddBoxRows = 32;      // rows of W per TMA box (the vocabulary granule is this many rows per CTA)
struct OddMaps {
  CUtensorMap h, w[kMaxClasses];
};
inline int odd_classes(int d) { return d % 8 == 0 ? 1 : (d % 4 == 0 ? 2 : (d % 2 == 0 ? 4 : 8)); }
inline int odd_shift(int d, int cls) { return static_cast<int>((static_cast<long long>(cls) * d) % 8); }
inline int odd_max_shift(int d) { return 8 - 8 / odd_classes(d); }   // the shifts are all multiples of gcd(d, 8)
// h [n][d] -> shifted copies [classes][class_rows][pitch]
cudaError_t launch_odd_shift(const void* h_bf16, int n, int d, int class_rows, int pitch, void* out,
                             cudaStream_t stream);
cudaError_t odd_prepare();
cudaError_t launch_odd_projection(const OddMaps& maps, const TcParams& p, const TcConfig& c, int workers,
                                  cudaStream_t stream);

inline int tc_h_box_rows(const TcConfig& c) { return c.mode == RowMode::kGroup8 ? 8 : c.a_rows; }   // rows of h per TMA box
// The fields of a launch's parameters that describe its work decomposition.
inline void tc_set_schedule(const TcPlan& plan, TcParams* p) {
  p->group_units = plan.group_units;
  p->row_units = plan.row_units;
  p->chunks = plan.chunks;
  p->tiles_per_unit = plan.tiles_per_unit;
  p->full_tiles_first = plan.full_tiles_first;
  p->granule_rows = plan.granule_rows;
  p->mlp_rows = plan.mlp_rows;
  p->classes = plan.classes;
  p->class_chunks = plan.chunks / plan.classes;
  p->chunk_q = plan.granules / p->class_chunks;
  p->chunk_r = plan.granules % p->class_chunks;
  p->chunk_mul = p->class_chunks > 1 ? static_cast<uint32_t>(((1ull << 32) + p->class_chunks - 1) / p->class_chunks) : 0u;
  p->full_granules = 256 / plan.granule_rows;
}
int tc_threads();
int tc_enumerate_tiles(const TcParams& p, int cta, int blocks, int workers, int* out, int capacity);
void tc_configure(int n, int d, int V, int sm_count, TcConfig* c);
// Units of two row blocks are walked group by group of row units, so many to a group that their h takes up to 50 MB.  There are
// more workers than row units then, several read the same h from either half of L2 (126 MB), which keep a copy each, and two copies
// must fit beside W.  W comes from HBM once more per group, which is little.  ms per step at d = 2048 with single blocks (each
// row unit's h is read by one worker there), with one group, with groups of up to 50 and of up to 34 MB: n = 16384, V = 128256
// 6.32, 6.35, 5.99 and 5.99, n = 14000, V = 100000 4.21, 4.21, 4.05 and 4.06; at 50 MB one group is as good as two (n = 12000,
// V = 60000 2.17, 2.11 and 2.10; d = 1536, n = 16384 there 2.24, 2.13 and 2.14).
inline int tc_two_group(int n, int d, int row_units) {
  constexpr long long kGroupBytes = 50ll << 20;
  const long long groups = (2ll * n * d + kGroupBytes - 1) / kGroupBytes;
  return static_cast<int>((row_units + groups - 1) / groups);
}
// Whether units of two row blocks pay, given both plans.  They halve what W brings from L2 into shared memory, and how much that is
// depends on where its rows begin: with d % 16 == 8 every other row begins off a 32-byte sector, so that a slab's 128 bytes take five
// sectors instead of four, and loads of W bound single blocks.  Rows on sectors bring the least, and with one row unit, where every
// worker reads the same h at the same time, nothing.  Single blocks and two, us per step at the power limit:
//   d % 16 == 8   n = 450, d = 1032, V = 108884 125.5 and 114.0, n = 860, d = 1288, V = 54527 140.2 and 127.4, n = 392, d = 2024,
//                 V = 37250 82.6 and 76.1 (128 slabs of row blocks per worker); below that n = 293, d = 568, V = 30010 21.1 and 23.3
//   one row unit  n = 402, d = 880, V = 87086 72.0 and 78.3, n = 434, d = 1120, V = 104871 107.8 and 114.1, n = 512, d = 2048,
//                 V = 128256 226 to 230 and 227 to 233
//   two row units 128 to 260 slabs 0.92 to 1.06 times as fast, 0.97 on average (n = 900, d = 1024, V = 60000 105.9 and 109.3), from 260 on
//                 1.01 (n = 1024, d = 2048, V = 128256 440 and 413); with a learned router's units in the launch 1.04 from 128 on
//                 (n = 833, d = 1184, V = 54769 119.6 and 112.8)
//   more          0.96 to 1.09, 1.00 on average up to 260 slabs, then 1.01 to 1.05 (n = 8192, d = 896, V = 151936 1697 and 1599)
// Few units may leave the busiest worker more passes than single blocks would, of which up to 4 % are given back (n = 777, d = 1536,
// V = 151936: 34 instead of 33, 351 to 372 and 357 to 364): a last unit of one block counts for two here, so that most batches of an
// odd number of blocks, up to some twenty, stay on single ones.
inline bool tc_two_blocks_pay(const TcPlan& two, const TcPlan& one, int d) {
  const int k_slabs = (d + 63) / 64;
  const bool off_sectors = d % 16 != 0;
  const int least = off_sectors || two.mlp_rows > 0 || two.row_units > 2 ? 128 : 260;
  return k_slabs >= 8 && (off_sectors || two.row_units >= 2) && two.passes * k_slabs >= least && two.passes * 100 <= one.passes * 104;
}
bool tc_configure_two(int d, TcConfig* c);
void tc_plan(int n, int V, int cta, int blocks, int workers, int max_chunks, int mlp_hidden, int classes, TcPlan* plan);
cudaError_t tc_prepare();   // opt in to the kernels' dynamic shared memory size (once per device)
cudaError_t launch_tc_projection(const TcMaps& maps, const TcParams& p, const TcConfig& c, int workers,
                                 cudaStream_t stream);

// ---- 8-bit head (tlr_tc8.cu): one CTA per worker, n <= tc8_max_rows()
int tc8_max_rows();
void tc8_configure(int n, int d, TcConfig* c);
cudaError_t tc8_prepare();
// h [n][d] bf16 -> parts [2][part_rows][d] e4m3 (rows n.. zero) and hscale[n]
cudaError_t launch_h_split(const void* h_bf16, int n, int d, int part_rows, uint8_t* parts, float* hscale,
                           cudaStream_t stream);
cudaError_t launch_tc8_projection(const TcMaps& maps, const TcParams& p, const TcConfig& c, int workers,
                                  cudaStream_t stream);

// Tuning switches, read from the environment once per process (defaults are the measured best).
struct Tuning {
  int granule;          // TLR_TC_GRANULE: vocabulary granule in rows (0 = default, 16 * cta)
  int even_tiles;       // TLR_TC_EVEN_TILES: equal-size tiles in pair mode
  int ring_a, ring_b;   // TLR_TC_RINGS="a,b": ring depths (0 = default)
  int tc8_inline;       // TLR_TC8_INLINE=0 keeps the separate split kernel
  int finish_threads;   // TLR_FINISH_THREADS: block size of finish_small_kernel (0 = default)
  int row_cost;         // TLR_TC_ROW_COST: pair mode plans by vocabulary rows per worker only, not by tile passes first
};
const Tuning& tuning();

}  // namespace tlr
