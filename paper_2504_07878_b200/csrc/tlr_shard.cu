// Sharded forms of the routing step (several GPUs, one process each).
//
// Vocabulary sharding (decode batches): each GPU holds a contiguous range of W's rows.  A shard's
// projection kernel leaves chunk partials as usual; they are folded into ONE 16-byte summary per row whose
// token index is global (shard offset added).  The summaries of all shards then reach every GPU in one of two
// ways, and the ordinary merge kernel scores, decides and compacts them (it reads the block of summaries,
// laid out [shards][rows], in place).  The merge of summaries is the same associative rule as the merge of
// chunk partials, so the sharded result differs from the one-GPU result only by fp32 summation order.
//   shard_summary_kernel  writes the summaries locally; the caller exchanges them (an all-gather of
//                         n x 16 bytes per GPU).
//   shard_push_kernel     the fused exchange: every summary is stored straight into this rank's slot of every
//                         peer's exchange block (plain peer stores; no peer loads, no multicast), and when
//                         the last block is done -- a system-wide fence after the stores -- this rank's flag on
//                         every peer is set to the call's epoch.  The peers' merge kernels wait on their own
//                         flags (bounded).
//
// Row sharding (prefill batches): every GPU routes its own rows; rows_merge_kernel turns the gathered
// per-rank index lists into one ascending list of global row numbers.
#include "tlr_common.cuh"

namespace tlr {

namespace {

constexpr int kWarps = 8;

// One warp folds one row's chunk partials; every lane ends with the result.
// kTies (d no multiple of 8): the shard's winner is settled among the residue classes, and m becomes its row_logit, so that
// equal rows of W in different shards tie exactly in the merge behind -- also where one shard ran on CUDA cores and another
// on tensor cores.
template <bool kTies>
__device__ __forceinline__ Partial row_summary(Partial* partials, uint32_t tag, uint32_t* status, int row, int chunks, int v_offset,
                                               const Ties& ties, int lane) {
  Partial* p = partials + static_cast<size_t>(row) * chunks;
  float second;
  Partial acc = fold_row(p, chunks, 1, lane, kTies ? &second : nullptr, kTies ? 0u : tag, status);
  if (!kTies && tag != 0) reset_tagged(p, lane, 32, chunks);
  if (kTies) settle_row(ties, row, p, chunks, 1, second, acc.m, acc.idx, acc.s, acc.t, lane, 32);
  if (acc.idx != kNoToken) acc.idx += v_offset;
  return acc;
}

template <bool kTies>
__global__ void __launch_bounds__(kWarps * 32)
shard_summary_kernel(Partial* partials, uint32_t tag, uint32_t* status, int n, int chunks, int v_offset, const Ties ties,
                     Partial* summary) {
  const int row = blockIdx.x * kWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  // A programmatic dependent launch like the kernels around it: its blocks (512 small ones at most fit beside the
  // projection's CTAs) wait for the projection or its tagged partials where they stand, and a merge kernel behind it may be
  // scheduled now.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tag == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (row >= n) return;
  const Partial acc = row_summary<kTies>(partials, tag, status, row, chunks, v_offset, ties, lane);
  if (lane == 0) summary[row] = acc;
  if (tag != 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <bool kTies>
__global__ void __launch_bounds__(kWarps * 32)
shard_push_kernel(const ShardPush a) {
  const int row = blockIdx.x * kWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  // Programmatic dependent launch: scheduled while the projection kernel finishes, and the merge kernel behind
  // this one may be scheduled now.  Untagged partials are read only after the projection has completed, tagged ones as they
  // arrive; either way the flags below are set behind it.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (a.tag == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (row < a.n) {
    const Partial acc = row_summary<kTies>(a.partials, a.tag, a.status, row, a.chunks, a.v_offset, a.ties, lane);
    for (int g = lane; g < a.shards; g += 32) a.peer_slot[g][row] = acc;     // lane g stores to peer g
  }
  if (a.tag != 0) asm volatile("griddepcontrol.wait;" ::: "memory");
  // every summary of this block is on its way; the last block to get here publishes the flags
  __threadfence_system();
  __shared__ int is_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int t = atomicAdd(a.ticket, 1u);
    is_last = (t == gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence_system();      // the other blocks' stores (fenced before their tickets) precede the flags
  for (int g = threadIdx.x; g < a.shards; g += blockDim.x) {
    uint32_t* f = a.peer_flag[g];
    asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(f), "r"(a.epoch) : "memory");
  }
  if (threadIdx.x == 0) *a.ticket = 0u;
}

// One block per rank: the rank's routed rows, shifted to global row numbers, go behind the lists of the
// ranks before it (counts are few, so every block adds them up itself).
__global__ void __launch_bounds__(256)
rows_merge_kernel(const int32_t* __restrict__ gathered_idx, const int32_t* __restrict__ counts,
                  const int32_t* __restrict__ row_offsets, int ranks, int cap, int32_t* __restrict__ global_idx,
                  int32_t* __restrict__ global_count) {
  const int g = blockIdx.x;
  int before = 0, total = 0;
  for (int r = 0; r < ranks; ++r) {
    const int c = counts[r];
    before += r < g ? c : 0;
    total += c;
  }
  const int mine = counts[g], off = row_offsets[g];
  for (int j = threadIdx.x; j < mine; j += blockDim.x)
    global_idx[before + j] = gathered_idx[static_cast<size_t>(g) * cap + j] + off;
  if (g == 0 && threadIdx.x == 0) *global_count = total;
}

}  // namespace

cudaError_t launch_shard_summary(Partial* partials, uint32_t tag, uint32_t* status, int n, int chunks, int v_offset,
                                 const Ties& ties, Partial* summary, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>((n + kWarps - 1) / kWarps), 1, 1);
  cfg.blockDim = dim3(kWarps * 32, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const auto kernel = ties.W != nullptr ? shard_summary_kernel<true> : shard_summary_kernel<false>;
  return cudaLaunchKernelEx(&cfg, kernel, partials, tag, status, n, chunks, v_offset, ties, summary);
}

cudaError_t launch_shard_push(const ShardPush& a, cudaStream_t stream) {
  const int blocks = a.n > 0 ? (a.n + kWarps - 1) / kWarps : 1;   // n == 0 still publishes the flags
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(blocks), 1, 1);
  cfg.blockDim = dim3(kWarps * 32, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, a.ties.W != nullptr ? shard_push_kernel<true> : shard_push_kernel<false>, a);
}

cudaError_t launch_rows_merge(const int32_t* gathered_idx, const int32_t* counts, const int32_t* row_offsets,
                              int ranks, int cap, int32_t* global_idx, int32_t* global_count, cudaStream_t stream) {
  rows_merge_kernel<<<ranks, 256, 0, stream>>>(gathered_idx, counts, row_offsets, ranks, cap, global_idx, global_count);
  return cudaGetLastError();
}

}  // namespace tlr
