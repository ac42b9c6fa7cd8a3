// Decode batches on an 8-bit (e4m3, one scale per vocabulary row) copy of W.
//
// At decode sizes the step is the time to stream W from HBM; W stored in 8 bits halves it.  The
// tensor core multiplies fp8 by fp8 only (tcgen05.mma kind::f8f6f4), and h is bf16, so h is not
// rounded to fp8 but SPLIT: every row of h is scaled by a power of two r so that its largest
// magnitude lies in [128, 256), and written as the sum of two e4m3 numbers, h / r = p1 + p2 with
// p1 = round(h / r) and p2 = round(h / r - p1).  A bf16 number has 8 significant bits and e4m3
// has 4: the first rounding leaves a remainder of at most 8 units of the bf16 number's last
// place, which the second part holds exactly.  Only elements below 2^-10 of the row's largest
// fall under e4m3's smallest step (2^-9); their error is at most 2^-17 of that largest.
//
// The two parts are stacked along the MMA's M dimension in alternating groups of eight rows (tc8_part_row), and ONE
// MMA per K step computes both products (products of e4m3 numbers are exact in fp32).  A token's logit is the sum of
// two accumulator rows eight lanes apart; the epilogue reads tensor memory in the 16 x 256-bit fragment layout, which
// gives both to the same thread, so it adds them in registers, multiplies by r (per token row) and by the weight row's
// scale, and folds.  (With all first parts above all second parts the two sums sat in different lane quadrants and
// went through shared memory from one warp to another, one thread per row with half of the threads idle: what
// followed a CTA's last MMA took 5.5 us, now 2.0; decode16 -- d = 896, V = 151936 -- 33.9 -> 30.6 us per step in a
// graph, n = 32 37.5 -> 34.3, n = 64 39.9 -> 38.9.)
// One MMA per K step at twice the bf16 rate leaves the tensor pipe half as busy as the bf16 path; the
// bytes from HBM are half.
//
// This file holds what only the 8-bit head has: the split kernel, the shape of the launch and the
// launch of tc8_projection_kernel (the projection kernel's body in tlr_tc_kernel.cuh in the row modes
// k8Small, k8Half and k8Wide; device helpers in tlr_tc8_dev.cuh).
#include <cuda.h>
#include <cuda_bf16.h>

#include "tlr_common.cuh"
#include "tlr_tc.cuh"
#define TLR_DEFINE_TC8_KERNEL
#include "tlr_tc_kernel.cuh"

namespace tlr {

// One block per row of the padded batch (rows >= n are written as zeros): the row's power-of-two
// scale r (largest |h| / r in [128, 256)), and h / r as the sum of two e4m3 arrays, [2][part_rows][d].
__global__ void __launch_bounds__(128)
h_split_kernel(const __nv_bfloat16* h, int n, int d, int part_rows, uint8_t* __restrict__ parts,
               float* __restrict__ hscale) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int row = blockIdx.x;
  const size_t part_stride = static_cast<size_t>(tc8_part_stride(part_rows)) * d;
  uint8_t* out = parts + static_cast<size_t>(tc8_part_row(row, part_rows)) * d;
  if (row >= n) {
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    for (int k = threadIdx.x * 16; k < d; k += 128 * 16) {
      *reinterpret_cast<uint4*>(out + k) = zero;
      *reinterpret_cast<uint4*>(out + part_stride + k) = zero;
    }
    return;
  }
  // Bound by latency: this kernel stands between every step and the one before.  With two-byte loads, each row read
  // twice, a step of n = 20, d = 512, V = 30000 took 15.5 us; now 12.1.
  // Chunks of 16 elements; a thread keeps the first kKeep of its own in registers between the maximum and the
  // conversion (all of them up to d = 4096), so that the row is read once and its loads are in flight together.
  constexpr int kKeep = 2;
  const uint4* src = reinterpret_cast<const uint4*>(h + static_cast<size_t>(row) * d);
  const int chunks = d >> 4;                                   // d is a multiple of 16
  uint4 v[kKeep][2];
  uint32_t pair = 0u;
#pragma unroll
  for (int i = 0; i < kKeep; ++i) {
    const int c = threadIdx.x + 128 * i;
    const bool in = c < chunks;
    v[i][0] = in ? __ldcg(src + 2 * c) : make_uint4(0u, 0u, 0u, 0u);
    v[i][1] = in ? __ldcg(src + 2 * c + 1) : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int i = 0; i < kKeep; ++i) pair = abs_max8(abs_max8(pair, v[i][0]), v[i][1]);
  for (int c = threadIdx.x + 128 * kKeep; c < chunks; c += 128)
    pair = abs_max8(abs_max8(pair, src[2 * c]), src[2 * c + 1]);
  float amax = larger_of(pair);
  __shared__ float red[4];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
  __syncthreads();
  amax = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
  const float r = split_scale(amax);
  const float inv = 1.0f / r;         // exact: r is a power of two
  if (threadIdx.x == 0) hscale[row] = r;
  auto put = [&](int c, const uint4& lo, const uint4& hi) {
    uint4 q1, q2;
    split16(lo, hi, inv, q1, q2);
    *reinterpret_cast<uint4*>(out + c * 16) = q1;
    *reinterpret_cast<uint4*>(out + part_stride + c * 16) = q2;
  };
#pragma unroll
  for (int i = 0; i < kKeep; ++i)
    if (static_cast<int>(threadIdx.x) + 128 * i < chunks) put(threadIdx.x + 128 * i, v[i][0], v[i][1]);
  for (int c = threadIdx.x + 128 * kKeep; c < chunks; c += 128) put(c, src[2 * c], src[2 * c + 1]);
}

int tc8_max_rows() { return 128; }

void tc8_configure(int n, int d, TcConfig* c) {
  // rows per part; the operand slab stacks the two parts.  Up to 64 rows both parts go through one MMA (its M holds
  // 2 x 16, 32 or 64 rows); above, every K step takes two MMAs and a part is n rounded up to 16 rows.
  int part_rows = n <= 16 ? 16 : (n <= 32 ? 32 : (n <= 64 ? 64 : ((n + 15) / 16) * 16));
  const int a_stage = 2 * part_rows * kRowBytes;
  const int b_stage = kBlockN * kRowBytes;
  const int k_slabs = (d + kRowBytes - 1) / kRowBytes;
  const int extra = kTc8ExtraBytes;
  const int budget = kSmemLimit - 1024 - kBarrierBytes - kScratchBytes - extra;
  // n <= 16 and all of h (two parts) small enough: the kernel splits h itself and keeps it resident, one
  // launch less.  TLR_TC8_INLINE=0 is a tuning switch that keeps the separate split kernel.
  bool inl = n <= 16 && k_slabs * 8 <= kSplitLanes * kSplitChunks && tuning().tc8_inline != 0;
  // ... and only while the resident copy leaves the W ring five stages: with four (d = 2048) what the
  // missing launch gains is lost again to the shallower ring
  if (inl && (budget - k_slabs * a_stage) / b_stage < 5) inl = false;
  int sa = inl ? k_slabs : (part_rows <= 32 ? 6 : (part_rows <= 64 ? 4 : 3));
  if (!inl && tuning().ring_a > 0) sa = tuning().ring_a;
  int sb = (budget - sa * a_stage) / b_stage;
  if (sb > kMaxBStages) sb = kMaxBStages;
  c->cta = 1;
  c->a_rows = 2 * part_rows;
  c->mode = part_rows <= 32 ? RowMode::k8Small : (part_rows <= 64 ? RowMode::k8Half : RowMode::k8Wide);
  c->part_rows = part_rows;
  c->lag = 0;
  c->a_stages = sa;
  c->b_stages = sb;
  c->inline_split = inl ? 1 : 0;
  c->smem_bytes = 1024 + sa * a_stage + sb * b_stage + kBarrierBytes + kScratchBytes + extra;
}

cudaError_t tc8_prepare() {
  for (const auto kernel : {tc8_projection_kernel<RowMode::k8Small>, tc8_projection_kernel<RowMode::k8Half>,
                            tc8_projection_kernel<RowMode::k8Wide>}) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_h_split(const void* h_bf16, int n, int d, int part_rows, uint8_t* parts, float* hscale,
                           cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(part_rows), 1, 1);
  cfg.blockDim = dim3(128, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, h_split_kernel, static_cast<const __nv_bfloat16*>(h_bf16), n, d, part_rows, parts,
                            hscale);
}

cudaError_t launch_tc8_projection(const TcMaps& maps, const TcParams& p, const TcConfig& c, int workers,
                                  cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(workers), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(c.smem_bytes);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const auto kernel = c.mode == RowMode::k8Small  ? tc8_projection_kernel<RowMode::k8Small>
                      : c.mode == RowMode::k8Half ? tc8_projection_kernel<RowMode::k8Half>
                                                  : tc8_projection_kernel<RowMode::k8Wide>;
  return cudaLaunchKernelEx(&cfg, kernel, maps, p);
}

}  // namespace tlr
