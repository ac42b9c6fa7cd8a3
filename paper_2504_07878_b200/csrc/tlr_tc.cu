// bf16 head: instantiations of the tensor-core projection kernel (one CTA per worker for
// n <= 128, a pair of CTAs above), their shared-memory configuration and launch, and the host
// view of the schedule the kernel walks.
#include <cuda.h>
#include <cuda_bf16.h>

#include "tlr_common.cuh"
#include "tlr_tc.cuh"
#include "tlr_tc_kernel.cuh"

namespace tlr {

int tc_threads() { return kThreads; }

// Host enumeration of the schedule the kernel walks (the same tile_of the device code uses):
// one record {worker, unit, row0, v0, rows} per non-empty tile of CTA rank 0, in walking order.
// Tiles of learned-router units are reported with v0 counted from V upwards.
int tc_enumerate_tiles(const TcParams& p, int cta, int blocks, int workers, int* out, int capacity) {
  int count = 0;
  const int units = (p.chunks + (p.mlp_hidden > 0 ? 1 : 0)) * p.row_units;
  for (int w = 0; w < workers; ++w) {
    for (int unit = w; unit < units; unit += workers) {
      const Unit un = blocks == 2 ? unit_of<2, false, true>(p, unit, 0) : cta == 2 ? unit_of<2>(p, unit, 0) : unit_of<1>(p, unit, 0);
      for (int t = 0; t < p.tiles_per_unit; ++t) {
        const Tile tl = tile_of(p, un, t);
        if (tl.rows == 0) continue;
        if (count < capacity) {
          int* r = out + 5 * count;
          r[0] = w;
          r[1] = unit;
          r[2] = un.row0;
          r[3] = un.chunk < 0 ? p.V + tl.v0 : tl.v0;
          r[4] = tl.rows;
        }
        ++count;
      }
    }
  }
  return count;
}

// Ring depths and shared-memory size for a given n.  The h ring is short (L2 latency),
// the W ring takes everything that is left (HBM latency).
void tc_configure(int n, int d, int V, int sm_count, TcConfig* c) {
  const int cta = n > kBlockM ? 2 : 1;
  int a_rows = kBlockM;
  RowMode mode = RowMode::kM128;
  if (cta == 1) {
    a_rows = ((n + 15) / 16) * 16;
    if (a_rows < 16) a_rows = 16;
    if (a_rows > kBlockM) a_rows = kBlockM;
    // Up to 16 token rows lie eight to every sixteen operand rows, so that two of the accumulator's lane quadrants have
    // rows and the epilogue reads them with four threads to a row.  In a stream, one thread per row and this: d = 512,
    // V = 32000 n = 1 11.26 and 10.55 us per step, n = 16 11.65 and 10.83; d = 2048, V = 128256 n = 16 88.7 and 86.
    // With four such groups the loads of h, eight rows each, cost more than that: n = 32 11.70 and 11.74, 89.6 and
    // 94.9; with two rows per thread n = 64 12.25 and 12.40.
    if (a_rows <= 64) mode = RowMode::kM64;
    if (n <= 16) {
      mode = RowMode::kGroup8;
      a_rows = n <= 8 ? 16 : 32;
    }
  }
  const int a_stage = a_rows * kRowBytes;
  const int b_stage = (kBlockN / cta) * kRowBytes;
  // h slabs come from L2 (about a microsecond away under load) and one is consumed per W
  // slab, so the h ring needs about half the depth of the W ring to keep up.  In pair mode five
  // stages: short units live on what the W ring holds when h arrives, and then h is what they wait for
  // (n = 256, d = 896, V = 18976: 4 / 5 / 6 / 8 stages 19.66 / 19.15 / 19.35 / 20.07 us per step;
  // n = 1024, d = 512, V = 32000: 39.2 / 38.5 / 38.6 / 39.4; no difference where W streams for long).
  int sa = cta == 2 ? 5 : (a_rows <= 32 ? 6 : 4);
  const int budget = kSmemLimit - 1024 - kBarrierBytes - kScratchBytes;
  int sb = (budget - sa * a_stage) / b_stage;
  if (sb > kMaxBStages) sb = kMaxBStages;
  const int k_slabs = (d + kRowBytes / 2 - 1) / (kRowBytes / 2);
  // Pair mode with all of a row unit's h beside at least four W stages (d = 193..576): h is loaded once per unit instead
  // of once per tile.  Worth it from twelve tiles per worker on: V = 64000, streamed and kept, d = 256 n = 1024 44.9 and
  // 43.8 us per step, n = 4096 156 and 151; d = 384 n = 4096 195 and 188; d = 512 n = 1024 69.7 and 67.5, n = 4096 246 and
  // 237; but n = 256 (3.4 tiles), d = 512 23.7 and 24.4, and at eight (V = 151936) no difference.
  const long long tiles = static_cast<long long>((n + 255) / 256) * ((V + kBlockN - 1) / kBlockN);
  if (cta == 2 && k_slabs >= 4 && k_slabs * a_stage + 4 * b_stage <= budget && tiles >= 12ll * (sm_count / 2)) {
    mode = RowMode::kM128Keep;
    sa = k_slabs;
    sb = (budget - sa * a_stage) / b_stage;
    if (sb > kMaxBStages) sb = kMaxBStages;
  }
  // Tuning override: TLR_TC_RINGS="<h stages>,<W stages>" (ignored if it does not fit).
  const Tuning& tn = tuning();
  if (mode != RowMode::kM128Keep && tn.ring_a >= 1 && tn.ring_a <= kRelease && tn.ring_b >= 1 && tn.ring_b <= kMaxBStages &&
      tn.ring_a * a_stage + tn.ring_b * b_stage <= budget) {
    sa = tn.ring_a;
    sb = tn.ring_b;
  }
  c->cta = cta;
  c->a_rows = a_rows;
  c->mode = mode;
  c->part_rows = a_rows;
  c->lag = 0;
  c->a_stages = sa;
  c->b_stages = sb;
  c->inline_split = 0;
  c->smem_bytes = 1024 + sa * a_stage + sb * b_stage + kBarrierBytes + kScratchBytes;
}

// The same with two row blocks to a unit.  The second block stays `lag` slabs of W behind the first: its MMAs of a tile's last
// slabs run while the first accumulator is folded (about 2100 cycles, 512 a slab) and the other way round, and the W stages of
// those slabs stay occupied meanwhile.  Lags of 3 / 4 / 5 with five stages of h and eight of W, of 5 with four and nine, and
// single blocks, us per step: n = 8192, d = 896, V = 151936 1738 / 1691 / 1648 / 1648 and 1738, n = 4096, d = 1536 there
// 1429 / 1405 / 1386 / 1391 and 1459, n = 512, d = 2048, V = 128256 228 / 226 / 225 / 225 and 235; 6 of eight stages leave too
// few for loads (407 instead of 364 at n = 777, d = 1536, V = 151936; 380 with single blocks).  False, and nothing changed, where
// the W ring (TLR_TC_RINGS) does not hold the slabs that lie between the two: lag + 1, before the second block frees the first.
bool tc_configure_two(int d, TcConfig* c) {
  if (c->b_stages < 2) return false;
  const int k_slabs = (d + kRowBytes / 2 - 1) / (kRowBytes / 2);
  c->mode = RowMode::kM128Two;
  c->lag = c->b_stages - 3;
  if (c->lag > 5) c->lag = 5;
  if (c->lag > k_slabs) c->lag = k_slabs;
  if (c->lag < 1) c->lag = 1;
  return true;
}

cudaError_t tc_prepare() {
  for (const auto kernel : {tc_projection_kernel<1, RowMode::kM128, true>, tc_projection_kernel<1, RowMode::kM64, true>,
                            tc_projection_kernel<1, RowMode::kGroup8, true>, tc_projection_kernel<2, RowMode::kM128, true>,
                            tc_projection_kernel<2, RowMode::kM128, false>, tc_projection_kernel<2, RowMode::kM128Keep, false>,
                            tc_projection_kernel<2, RowMode::kM128Two, false>}) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_tc_projection(const TcMaps& maps, const TcParams& p, const TcConfig& c, int workers,
                                 cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(workers * c.cta), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(c.smem_bytes);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = c.cta == 1 ? 1 : 2;
  // Pairs: short steps gain from a merge kernel that is resident before they end, others from registers (see the kernel).  At
  // n = 256 with 104 registers and without the limit: V = 32000, d = 512 14.25 and 14.55 us, V = 40000, d = 1024 24.1 and 24.9;
  // V = 64000, d = 512 22.9 and 22.6, d = 896 35.7 and 35.3.
  const bool beside = p.n <= 256 && p.tiles_per_unit <= 3;
  const auto kernel = c.mode == RowMode::kM128Two ? tc_projection_kernel<2, RowMode::kM128Two, false>
                      : c.mode == RowMode::kM128Keep ? tc_projection_kernel<2, RowMode::kM128Keep, false>
                      : c.cta == 2 && beside       ? tc_projection_kernel<2, RowMode::kM128, true>
                      : c.cta == 2                 ? tc_projection_kernel<2, RowMode::kM128, false>
                      : c.mode == RowMode::kGroup8 ? tc_projection_kernel<1, RowMode::kGroup8, true>
                      : c.mode == RowMode::kM64    ? tc_projection_kernel<1, RowMode::kM64, true>
                                                   : tc_projection_kernel<1, RowMode::kM128, true>;
  return cudaLaunchKernelEx(&cfg, kernel, maps, p);
}

}  // namespace tlr
