// Learned routing score on the hidden state: score = sigmoid(w2 . relu(W1 h + b1) + b2).
// The router the paper deploys is a small learned classifier (an MLP) fed with the last-layer
// hidden state (Sec. 3.1; Sec. 2.1); neither its width nor its activation nor weights are given, so
// the shape here (one hidden layer, ReLU, sigmoid output) is this library's assumption and
// the weights are the caller's.  Where the tensor-core projection kernel runs, the first layer is
// part of that launch (tlr_tc_kernel.cuh); this CUDA-core kernel serves the shapes it cannot take
// (d % 8 != 0, an unaligned W1): a block stages kMlpRows hidden-state rows in shared
// memory and covers kMlpUnits hidden units, eight threads per unit.  The 8-bit head has a tensor-core kernel of its own
// (mlp_mma_kernel) that runs beside the projection.
#include "tlr_common.cuh"

namespace tlr {

constexpr int kMlpThreads = 256;
constexpr int kMlpRows = 8;          // token rows per block
constexpr int kMlpUnits = 32;        // hidden units per block
constexpr int kMlpSplitK = kMlpThreads / kMlpUnits;   // 8 threads share one hidden unit's dot product

int mlp_hidden_blocks(int d_hidden) { return (d_hidden + kMlpUnits - 1) / kMlpUnits; }

// Block (x = row group, y = hidden-unit group): writes, for each of its rows, the partial sum
// over its hidden units of w2_j * relu(W1_j . h + b1_j).  The merge kernel adds the partials of
// a row in a fixed order, adds b2 and applies the sigmoid, so the score is deterministic.
__global__ void __launch_bounds__(kMlpThreads)
mlp_partial_kernel(const MlpLaunch a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned short* hs = reinterpret_cast<unsigned short*>(smem_raw);  // [kMlpRows][d] bf16 bits
  __shared__ float red[kMlpThreads / 32][kMlpRows];
  // The hidden states may come from the previous kernel in the stream.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  const int row0 = blockIdx.x * kMlpRows;
  const int d = a.d;
  const unsigned short* h = reinterpret_cast<const unsigned short*>(a.h);
  const unsigned short* W1 = reinterpret_cast<const unsigned short*>(a.W1);
  if (d % 8 == 0 && (reinterpret_cast<uintptr_t>(a.h) & 15) == 0) {
    // rows of a multiple of 8 elements: the staged block is contiguous in h, copy it 16 bytes at a time
    const int vec_per_row = d / 8;
    const uint4* src = reinterpret_cast<const uint4*>(h + static_cast<size_t>(row0) * d);
    uint4* dst = reinterpret_cast<uint4*>(hs);
    const int valid_rows = min(kMlpRows, a.n - row0);
#pragma unroll 4
    for (int i = threadIdx.x; i < kMlpRows * vec_per_row; i += kMlpThreads)
      dst[i] = (i < valid_rows * vec_per_row) ? __ldg(src + i) : make_uint4(0u, 0u, 0u, 0u);
  } else {
    for (int i = threadIdx.x; i < kMlpRows * d; i += kMlpThreads) {
      const int r = i / d, k = i - r * d;
      hs[i] = (row0 + r < a.n) ? h[static_cast<size_t>(row0 + r) * d + k] : static_cast<unsigned short>(0);
    }
  }
  __syncthreads();

  const int unit = blockIdx.y * kMlpUnits + threadIdx.x / kMlpSplitK;   // hidden unit of this thread
  const int part = threadIdx.x % kMlpSplitK;                            // which slice of k it sums
  float acc[kMlpRows];
#pragma unroll
  for (int r = 0; r < kMlpRows; ++r) acc[r] = 0.f;
  if (unit < a.d_hidden) {
    const unsigned short* wrow = W1 + static_cast<size_t>(unit) * d;
    const bool vec = (d % 8 == 0) && ((reinterpret_cast<uintptr_t>(a.W1) & 15) == 0);
    if (vec) {
#pragma unroll 4
      for (int k = part * 8; k < d; k += 8 * kMlpSplitK) {
        const uint4 w8 = __ldg(reinterpret_cast<const uint4*>(wrow + k));
        const unsigned int wv[4] = {w8.x, w8.y, w8.z, w8.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float w_lo = __uint_as_float(wv[q] << 16);
          const float w_hi = __uint_as_float(wv[q] & 0xffff0000u);
#pragma unroll
          for (int r = 0; r < kMlpRows; ++r) {
            const unsigned int hh = *reinterpret_cast<const unsigned int*>(hs + r * d + k + 2 * q);
            acc[r] = fmaf(__uint_as_float(hh << 16), w_lo, acc[r]);
            acc[r] = fmaf(__uint_as_float(hh & 0xffff0000u), w_hi, acc[r]);
          }
        }
      }
    } else {
      for (int k = part; k < d; k += kMlpSplitK) {
        const float w = __uint_as_float(static_cast<unsigned int>(wrow[k]) << 16);
#pragma unroll
        for (int r = 0; r < kMlpRows; ++r)
          acc[r] = fmaf(__uint_as_float(static_cast<unsigned int>(hs[r * d + k]) << 16), w, acc[r]);
      }
    }
  }
  // the kMlpSplitK threads of a unit are adjacent lanes: finish the dot products
#pragma unroll
  for (int r = 0; r < kMlpRows; ++r) {
#pragma unroll
    for (int off = kMlpSplitK / 2; off > 0; off >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off);
  }
  float contrib[kMlpRows];
  const bool owner = (part == 0) && (unit < a.d_hidden);
  const float b1 = owner ? a.b1[unit] : 0.f, w2 = owner ? a.w2[unit] : 0.f;
#pragma unroll
  for (int r = 0; r < kMlpRows; ++r) contrib[r] = owner ? w2 * fmaxf(acc[r] + b1, 0.f) : 0.f;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < kMlpRows; ++r) {
    float v = contrib[r];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane == 0) red[warp][r] = v;
  }
  __syncthreads();
  if (threadIdx.x < kMlpRows && row0 + threadIdx.x < a.n) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kMlpThreads / 32; ++w) v += red[w][threadIdx.x];
    a.partial[static_cast<size_t>(row0 + threadIdx.x) * gridDim.y + blockIdx.y] = v;
  }
}

// 8-bit head (d a multiple of 16, W1 and h 16-byte aligned): the same partial sums with mma.sync, beside the projection.
// The projection kernel of the 8-bit head multiplies e4m3 only, so W1 cannot be units of that launch; what W1 needs is
// small (100 rows, 256 units, d = 2048: 0.1 GFLOP, 1.5 MB) and hides behind the stream of W if it does not wait for it.
// So this kernel reads h without waiting for the projection in front of it: that kernel lets its dependents be scheduled
// only after its own wait, when h is complete.  One block waits for the projection at the END, so that this grid is not
// complete before it and the merge kernel behind, which waits for this grid, finds both.  Four warps per block, each
// a quarter of K, and 2 KB of shared memory: such blocks fit beside the projection's CTAs whatever their rings take.
// As the CUDA-core kernel between projection and merge: 34 of 111 us per step at that size (V = 128256); now 4 of 79.
constexpr int kMmaRows = 16;
constexpr int kMmaWarps = 4;
constexpr int kMmaBatch = 4;         // steps of 32 k values whose loads a warp has in flight together
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__global__ void __launch_bounds__(32 * kMmaWarps)
mlp_mma_kernel(const MlpLaunch a) {
  __shared__ float sums[16][32];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;          // row / column of the fragments, and which eight of 32 k values
  const int row0 = blockIdx.x * kMmaRows + g, row1 = row0 + 8, unit0 = blockIdx.y * kMlpUnits;
  const unsigned short* h = static_cast<const unsigned short*>(a.h);
  const unsigned short* W1 = static_cast<const unsigned short*>(a.W1);
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  float acc[4][4] = {};
  // Bound by the trips to memory, one per batch, that take about 3 us each beside the stream of W where they go to HBM: with few
  // rows this kernel then ends behind the projection.  So the block's rows of W1 are asked for at once.  us per step without and
  // with it, where the step finds nothing in L2: n = 2, d = 1712, V = 49399, 225 units 31.2 and 27.4, n = 4, d = 2048, V = 20000, 128 units
  // 26.1 and 21.8, n = 33, d = 1696, V = 20698, 421 units 26.9 and 22.6, n = 16, d = 896, V = 151936, 256 units 29.0 and 28.9.  Where the step
  // before has left all of W and W1 there, the requests stand in the way of the loads: n = 4, d = 2048, V = 32000, 512 units 16.1 and
  // 18.6, n = 48, d = 1536, V = 30000, 300 units 17.0 and 18.5, n = 10, d = 896, V = 60000, 256 units 14.7 both; a decoder's other layers
  // see to it that it has not.
  if (blockIdx.x == 0) {
    const char* rows = reinterpret_cast<const char*>(W1 + static_cast<size_t>(unit0) * a.d);
    const size_t bytes = static_cast<size_t>(min(kMlpUnits, a.d_hidden - unit0)) * a.d * 2;
    for (size_t at = threadIdx.x * 128u; at < bytes; at += 32 * kMmaWarps * 128u)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(rows + at));
  }
  // A thread's 16 bytes are eight consecutive k values; which k an MMA calls which does not matter as long as both
  // operands agree, so words 0, 1 go to one MMA (16 k values over the four threads) and words 2, 3 to the next.
  const int steps = (a.d + 31) / 32, s0 = steps * warp / kMmaWarps, s1 = steps * (warp + 1) / kMmaWarps;
  for (int sb = s0; sb < s1; sb += kMmaBatch) {
    uint4 x[kMmaBatch], y[kMmaBatch], w[kMmaBatch][4];     // every load of a batch is in flight before its first MMA
#pragma unroll
    for (int i = 0; i < kMmaBatch; ++i) {
      const int k = (sb + i) * 32 + t * 8;
      const bool in = sb + i < s1 && k < a.d;
      x[i] = in && row0 < a.n ? __ldcg(reinterpret_cast<const uint4*>(h + static_cast<size_t>(row0) * a.d + k)) : zero;
      y[i] = in && row1 < a.n ? __ldcg(reinterpret_cast<const uint4*>(h + static_cast<size_t>(row1) * a.d + k)) : zero;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int u = unit0 + 8 * j + g;
        w[i][j] = in && u < a.d_hidden ? __ldg(reinterpret_cast<const uint4*>(W1 + static_cast<size_t>(u) * a.d + k)) : zero;
      }
    }
#pragma unroll
    for (int i = 0; i < kMmaBatch; ++i) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        mma_bf16(acc[j], x[i].x, y[i].x, x[i].y, y[i].y, w[i][j].x, w[i][j].y);
        mma_bf16(acc[j], x[i].z, y[i].z, x[i].w, y[i].w, w[i][j].z, w[i][j].w);
      }
    }
  }
  // the warps' sums, added in a fixed order through one 2 KB buffer
  for (int turn = kMmaWarps - 1; turn > 0; --turn) {
    if (warp == turn) {
#pragma unroll
      for (int i = 0; i < 16; ++i) sums[i][lane] = acc[i >> 2][i & 3] + (turn == kMmaWarps - 1 ? 0.f : sums[i][lane]);
    }
    __syncthreads();
  }
  if (warp == 0) {
    float v0 = 0.f, v1 = 0.f;                     // rows row0 and row1, units 2t and 2t + 1 of every eight
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int u = unit0 + 8 * j + 2 * t + i;
        if (u >= a.d_hidden) continue;
        const float b1 = __ldg(a.b1 + u), w2 = __ldg(a.w2 + u);
        v0 += w2 * fmaxf(acc[j][i] + sums[4 * j + i][lane] + b1, 0.f);
        v1 += w2 * fmaxf(acc[j][2 + i] + sums[4 * j + 2 + i][lane] + b1, 0.f);
      }
    }
    v0 += __shfl_xor_sync(0xffffffffu, v0, 1);
    v1 += __shfl_xor_sync(0xffffffffu, v1, 1);
    v0 += __shfl_xor_sync(0xffffffffu, v0, 2);
    v1 += __shfl_xor_sync(0xffffffffu, v1, 2);
    if (t == 0) {
      if (row0 < a.n) a.partial[static_cast<size_t>(row0) * gridDim.y + blockIdx.y] = v0;
      if (row1 < a.n) a.partial[static_cast<size_t>(row1) * gridDim.y + blockIdx.y] = v1;
    }
  }
  if (blockIdx.x == 0 && blockIdx.y == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

cudaError_t launch_mlp_beside(const MlpLaunch& a, cudaStream_t stream) {
  if (a.n <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>((a.n + kMmaRows - 1) / kMmaRows),
                     static_cast<unsigned>(mlp_hidden_blocks(a.d_hidden)), 1);
  cfg.blockDim = dim3(32 * kMmaWarps, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, mlp_mma_kernel, a);
}

cudaError_t launch_mlp_score(const MlpLaunch& a, cudaStream_t stream) {
  if (a.n <= 0) return cudaSuccess;
  const int smem = kMlpRows * a.d * 2;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(mlp_partial_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>((a.n + kMlpRows - 1) / kMlpRows),
                     static_cast<unsigned>(mlp_hidden_blocks(a.d_hidden)), 1);
  cfg.blockDim = dim3(kMlpThreads, 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(smem);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, mlp_partial_kernel, a);
}

}  // namespace tlr
