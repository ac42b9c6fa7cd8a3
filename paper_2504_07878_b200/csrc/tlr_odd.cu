// Hidden sizes that are no multiple of 8 on the tensor cores: the shifted copies of h and the launch of the projection
// kernel that walks the vocabulary by residue class (OddMaps in tlr_tc.cuh has the idea).
//
// Before, every such shape ran on the CUDA-core kernel (tlr_simt.cu), which is bound by its FMAs and by one thread
// reading one row of W.  The projection here does the work of the bf16 head plus at most one more K slab and is bound by
// what bounds that one; the copies of h cost a launch and C * n * d * 2 bytes, small beside W.  Per step in a graph,
// before and after: n = 64, d = 300, V = 33000 194 -> 14 us; n = 1, d = 999, V = 60000 624 -> 29 (120 MB of W: 18);
// n = 256, d = 999, V = 60000 3987 -> 48; n = 200, d = 101, V = 33000 160 -> 17.
#include <cuda.h>
#include <cuda_bf16.h>

#include "tlr_common.cuh"
#include "tlr_tc.cuh"
#define TLR_DEFINE_ODD_KERNELS
#include "tlr_tc_kernel.cuh"

namespace tlr {

namespace {

constexpr int kShiftThreads = 256;

// Copy r of h has its rows `pitch` elements apart (a multiple of 8), each beginning with the class's shift in zeros.
// One thread writes 16 bytes; the reads of h are 2 bytes wide (its rows have no alignment) and hit L1.  (h is not
// __restrict__: a copy kernel in front may still be writing it when this kernel starts, so it is not read-only data.)
__global__ void __launch_bounds__(kShiftThreads)
odd_shift_kernel(const unsigned short* h, int n, int d, int classes, int class_rows, int pitch,
                 unsigned short* __restrict__ out) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int vecs = pitch / 8;
  const long long total = static_cast<long long>(classes) * n * vecs;
  for (long long i = static_cast<long long>(blockIdx.x) * kShiftThreads + threadIdx.x; i < total;
       i += static_cast<long long>(gridDim.x) * kShiftThreads) {
    const int vec = static_cast<int>(i % vecs);
    const int rc = static_cast<int>(i / vecs);
    const int row = rc % n, cls = rc / n;
    const int shift = static_cast<int>((static_cast<long long>(cls) * d) % 8);
    const unsigned short* src = h + static_cast<size_t>(row) * d;
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = vec * 8 + 2 * j - shift;
      const uint32_t lo = (k >= 0 && k < d) ? src[k] : 0u;
      const uint32_t hi = (k + 1 >= 0 && k + 1 < d) ? src[k + 1] : 0u;
      w[j] = lo | (hi << 16);
    }
    *reinterpret_cast<uint4*>(out + (static_cast<size_t>(cls) * class_rows + row) * pitch + vec * 8) =
        make_uint4(w[0], w[1], w[2], w[3]);
  }
}

}  // namespace

cudaError_t launch_odd_shift(const void* h_bf16, int n, int d, int class_rows, int pitch, void* out,
                             cudaStream_t stream) {
  const int classes = odd_classes(d);
  const long long total = static_cast<long long>(classes) * n * (pitch / 8);
  long long blocks = (total + kShiftThreads - 1) / kShiftThreads;
  if (blocks > 1184) blocks = 1184;          // 8 per SM
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(blocks), 1, 1);
  cfg.blockDim = dim3(kShiftThreads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, odd_shift_kernel, static_cast<const unsigned short*>(h_bf16), n, d, classes,
                            class_rows, pitch, static_cast<unsigned short*>(out));
}

cudaError_t odd_prepare() {
  for (const auto kernel :
       {odd_projection_kernel<1, RowMode::kM128>, odd_projection_kernel<1, RowMode::kM64>,
        odd_projection_kernel<1, RowMode::kGroup8>, odd_projection_kernel<2, RowMode::kM128>,
        odd_projection_kernel<2, RowMode::kM128Keep>}) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_odd_projection(const OddMaps& maps, const TcParams& p, const TcConfig& c, int workers,
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
  const auto kernel = c.mode == RowMode::kM128Keep ? odd_projection_kernel<2, RowMode::kM128Keep>
                      : c.cta == 2                 ? odd_projection_kernel<2, RowMode::kM128>
                      : c.mode == RowMode::kGroup8 ? odd_projection_kernel<1, RowMode::kGroup8>
                      : c.mode == RowMode::kM64    ? odd_projection_kernel<1, RowMode::kM64>
                                                   : odd_projection_kernel<1, RowMode::kM128>;
  return cudaLaunchKernelEx(&cfg, kernel, maps, p);
}

}  // namespace tlr
