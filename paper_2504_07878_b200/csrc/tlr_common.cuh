// Shared device-side definitions of the routing kernels: the per-row partial result
// that the projection kernels emit and the rule that merges two of them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "tlr.h"

namespace tlr {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr int kNoToken = 0x7fffffff;

// Online-softmax summary of one row over a range of the vocabulary:
//   m   = max logit in the range          idx = lowest vocabulary index attaining it
//   s   = sum exp(z - m)                  t   = sum exp(z - m) * (z - m)
// With the whole vocabulary folded in: conf = 1/s, entropy = ln s - t/s.
// An empty range is (m = -inf, idx = kNoToken, s = 0, t = 0).
struct __align__(16) Partial {
  float m;
  int idx;
  float s;
  float t;
};

__device__ __forceinline__ Partial empty_partial() {
  Partial p;
  p.m = -INFINITY;
  p.idx = kNoToken;
  p.s = 0.f;
  p.t = 0.f;
  return p;
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Associative and commutative merge; ties on m go to the lower vocabulary index.  (No branches, and ex2 without care for
// results below 2^-126: this and the folds below stand between the last logit and the decision, and nothing overlaps them.)
__device__ __forceinline__ Partial merge(const Partial& a, const Partial& b) {
  Partial r;
  const bool a_wins = (a.m > b.m) || (a.m == b.m && a.idx <= b.idx);
  r.m = a_wins ? a.m : b.m;
  r.idx = a_wins ? a.idx : b.idx;
  // Rescale each side to the new maximum.  A side with s == 0 (an empty range) contributes
  // nothing: its m is -inf, which must not reach the arithmetic below.  A NaN sum is not
  // "empty": it goes through and poisons the result, which the final step then flags.
  const float da = a.s == 0.f ? 0.f : a.m - r.m;  // <= 0
  const float db = b.s == 0.f ? 0.f : b.m - r.m;
  const float ea = ex2_approx(da * kLog2e), eb = ex2_approx(db * kLog2e);
  r.s = fmaf(b.s, eb, a.s * ea);
  r.t = fmaf(eb, fmaf(db, b.s, b.t), ea * fmaf(da, a.s, a.t));
  return r;
}

__device__ __forceinline__ Partial shfl_xor(const Partial& p, int lane_mask) {
  Partial r;
  r.m = __shfl_xor_sync(0xffffffffu, p.m, lane_mask);
  r.idx = __shfl_xor_sync(0xffffffffu, p.idx, lane_mask);
  r.s = __shfl_xor_sync(0xffffffffu, p.s, lane_mask);
  r.t = __shfl_xor_sync(0xffffffffu, p.t, lane_mask);
  return r;
}

__device__ __forceinline__ Partial warp_merge(Partial p) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) p = merge(p, shfl_xor(p, off));
  return p;
}

constexpr int kPerLane = 6;            // ceil(192 / 32): the most partials a lane can own
constexpr int kRowsPerLane = 5;        // ... in the kernels bound by latency (148 / 32): registers

// A lane's share of a row's partials -- first, first + stride, ... below `count`: maxima and sums, and the largest maximum
// with its lowest index.
template <int kN>
struct LaneFold {
  float m[kN], s[kN], t[kN];
  float best;
  int idx;
  __device__ __forceinline__ void clear() {
    best = -INFINITY;
    idx = kNoToken;
#pragma unroll
    for (int k = 0; k < kN; ++k) {
      m[k] = -INFINITY;
      s[k] = t[k] = 0.f;
    }
  }
  __device__ __forceinline__ void put(int k, const Partial& v) {
    m[k] = v.m;
    s[k] = v.s;
    t[k] = v.t;
    idx = v.m > best ? v.idx : (v.m == best ? min(v.idx, idx) : idx);
    best = fmaxf(best, v.m);
  }
  __device__ __forceinline__ void load(const Partial* p, int first, int stride, int count, size_t chunk_stride) {
    clear();
#pragma unroll
    for (int k = 0; k < kN; ++k) {
      const int j = first + stride * k;
      Partial v = empty_partial();
      if (j < count) {
        const float4 raw = __ldcg(reinterpret_cast<const float4*>(p + j * chunk_stride));
        v.m = raw.x;
        v.idx = __float_as_int(raw.y);
        v.s = raw.z;
        v.t = raw.w;
      }
      put(k, v);
    }
  }
  // The sums rescaled to the row's maximum.  An empty range contributes nothing; a NaN sum goes through.
  __device__ __forceinline__ void sums(float row_m, float& sum_s, float& sum_t) const {
    sum_s = sum_t = 0.f;
#pragma unroll
    for (int k = 0; k < kN; ++k) {
      const float dm = s[k] == 0.f ? 0.f : m[k] - row_m;    // <= 0
      const float e = ex2_approx(dm * kLog2e);
      sum_s = fmaf(s[k], e, sum_s);
      sum_t = fmaf(e, fmaf(dm, s[k], t[k]), sum_t);
    }
  }
  // The largest of the maxima below the row's.
  __device__ __forceinline__ float second(float row_m) const {
    float below = -INFINITY;
#pragma unroll
    for (int k = 0; k < kN; ++k) below = m[k] < row_m ? fmaxf(below, m[k]) : below;
    return below;
  }
};

// The largest maximum of a group of L lanes (a power of two, aligned) and its lowest index; all of them get it.
__device__ __forceinline__ void group_best(float& m, int& idx, int L) {
  if (L == 32) {      // two warp reductions, the floats as integers of the same order
    const int bits = __float_as_int(m);
    const int top = __reduce_max_sync(0xffffffffu, bits ^ ((bits >> 31) & 0x7fffffff));
    const float best = __int_as_float(top ^ ((top >> 31) & 0x7fffffff));
    idx = __reduce_min_sync(0xffffffffu, m == best ? idx : kNoToken);      // (+0 and -0 are equal here, too)
    m = best;
    return;
  }
  for (int off = L >> 1; off > 0; off >>= 1) {
    const float om = __shfl_xor_sync(0xffffffffu, m, off);
    const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
    idx = om > m ? oi : (om == m ? min(oi, idx) : idx);
    m = fmaxf(m, om);
  }
}
__device__ __forceinline__ void group_sum(float& s, float& t, int L) {
  for (int off = L >> 1; off > 0; off >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, off);
    t += __shfl_xor_sync(0xffffffffu, t, off);
  }
}
__device__ __forceinline__ float group_max(float v, int L) {
  for (int off = L >> 1; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
  return v;
}

// Folds one row's partials.  Every lane returns the same result.  `second` (optional): the largest of the partials' maxima
// below the row's.
__device__ __forceinline__ Partial fold_row(const Partial* p, int chunks, int chunk_stride, int lane,
                                            float* second = nullptr) {
  Partial r;
  LaneFold<kPerLane> f;
  f.load(p, lane, 32, chunks, chunk_stride);
  r.m = f.best;
  r.idx = f.idx;
  group_best(r.m, r.idx, 32);
  f.sums(r.m, r.s, r.t);
  group_sum(r.s, r.t, 32);
  if (second != nullptr) *second = group_max(f.second(r.m), 32);
  return r;
}

// Hidden sizes that are no multiple of 8 on the tensor cores: what settles a row's winner and its logit (settle_row).
struct Ties {
  const unsigned short* W;   // bf16 [V][d]; null = not needed
  const unsigned short* h;   // bf16 [n][d]
  int d, V;
};

__device__ __forceinline__ float bf16_value(unsigned short bits) { return __uint_as_float(static_cast<uint32_t>(bits) << 16); }

// The logit of token v in the row h by the L lanes of a row (lane gl of them, mask `group`), summed in fp32 in one fixed
// order: equal rows of W give equal bits, whatever kernel, shard or GPU asks with the same L.  `size` receives the sum of the
// products' magnitudes.  Bound by the trips to memory and, a row's lanes being few, by instructions: every line of the row of W
// is asked for before the first is used, a lane has six loads of either operand in flight, and they are two elements wide
// where d is even (rows have no alignment beyond one element or two).
template <bool kPairs>
__device__ __forceinline__ float2 lane_logit(const unsigned short* w, const unsigned short* h, int d, int gl, int L) {
  constexpr int kBatch = 6;
  const int loads = kPairs ? d >> 1 : d;
  float z = 0.f, size = 0.f;
  for (int k0 = gl; k0 < loads; k0 += kBatch * L) {
    uint32_t x[kBatch], y[kBatch];
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int k = k0 + i * L;
      x[i] = y[i] = 0u;
      if (k < loads) {
        x[i] = kPairs ? reinterpret_cast<const uint32_t*>(h)[k] : h[k];
        y[i] = kPairs ? reinterpret_cast<const uint32_t*>(w)[k] : w[k];
      }
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const float a = __uint_as_float(x[i] << 16), b = __uint_as_float(y[i] << 16);
      z = fmaf(a, b, z);
      size = fmaf(fabsf(a), fabsf(b), size);
      if (kPairs) {
        const float c = __uint_as_float(x[i] & 0xffff0000u), e = __uint_as_float(y[i] & 0xffff0000u);
        z = fmaf(c, e, z);
        size = fmaf(fabsf(c), fabsf(e), size);
      }
    }
  }
  return make_float2(z, size);
}
__device__ __forceinline__ float row_logit(const unsigned short* W, const unsigned short* h, int d, int v, int gl, int L,
                                           unsigned int group, float* size) {
  const unsigned short* w = W + static_cast<size_t>(v) * d;
  for (int k = gl * 64; k < d; k += L * 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(w + k));
  float2 r = (d & 1) == 0 ? lane_logit<true>(w, h, d, gl, L) : lane_logit<false>(w, h, d, gl, L);
  for (int off = L >> 1; off > 0; off >>= 1) {
    r.x += __shfl_xor_sync(group, r.x, off);
    r.y += __shfl_xor_sync(group, r.y, off);
  }
  *size = r.y;
  return r.x;
}

// The winner among idx and the partials of a row whose maxima are at least `least`, by row_logit (z, idx's): its index and its
// logit.  Equal rows of W tie exactly and the lowest index wins.  Rarely called; a candidate costs a trip to L2.  (Not a function
// of its own: around a call the loads of row_logit went out a few at a time, n = 200, d = 999, V = 60000 51.0 -> 55.5 us.)
struct Winner {
  int idx;
  float z;
};
static __device__ __forceinline__ Winner settle_ties(const Ties ties, int row, const Partial* __restrict__ p, int chunks,
                                               int chunk_stride, float least, int idx, float z, int gl, int L) {
  const unsigned short* h = ties.h + static_cast<size_t>(row) * ties.d;
  const unsigned int lane = threadIdx.x & 31;
  const unsigned int group = (L == 32 ? 0xffffffffu : (1u << L) - 1u) << (lane - gl);
  float size;
  Winner win = {idx, z};
  for (int j0 = 0; j0 < chunks; j0 += L) {
    const int j = j0 + gl;
    int mine = kNoToken;
    if (j < chunks) {
      const Partial* q = p + static_cast<size_t>(j) * chunk_stride;
      if (__ldcg(&q->m) >= least) mine = __ldcg(&q->idx);
    }
    unsigned int todo = __ballot_sync(group, mine < ties.V && mine != idx) & group;
    while (todo != 0u) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int v = __shfl_sync(group, mine, src);
      const float zv = row_logit(ties.W, h, ties.d, v, gl, L, group, &size);
      if (zv > win.z || (zv == win.z && v < win.idx)) {
        win.z = zv;
        win.idx = v;
      }
    }
  }
  return win;
}

// The row's summary (m, idx, s, t) with its winner settled among the residue classes and the winner's logit replaced by its
// row_logit; `second` is the largest of its partials' maxima below m.  Called by the L lanes of a row.
//
// Ties: equal rows of W in different classes get logits that agree to rounding only.  Candidates are the partials within what
// rounding can do to sums of the winner's products: 2^-21 of their magnitudes for each accumulation of 16 and 8 more, twice.
// Maxima that agree to the bit need no settling (the merge has taken the lowest index), so that a row of equal logits -- a
// hidden state of zeros, as padding leaves it -- costs nothing; with every partial within 1e-3 a candidate, one such row in the
// batch made a step of n = 16, d = 300, V = 33000 322 us long.
// The logit: the tensor cores truncate where they add, by more the larger the sum, so that the largest logit comes out low
// against the others; s counts the winner's own term as e^0 = 1 and everything else moves by m's error.  Confidences against
// 64 bits (2-norm) as the projection leaves them, here, and on CUDA cores, where these heads ran before: d = 300 6.7e-7,
// 1.7e-7, 3.2e-7; d = 999 2.3e-6, 1.7e-7, 8.7e-7.
// A row that is not finite stays as it is; so does one whose index lies beyond V.
__device__ __forceinline__ void settle_row(const Ties& ties, int row, const Partial* __restrict__ p, int chunks,
                                           int chunk_stride, float second, float& m, int& idx, float& s, float& t, int gl,
                                           int L) {
  if (idx >= ties.V) return;
  const unsigned int lane = threadIdx.x & 31;
  const unsigned int group = (L == 32 ? 0xffffffffu : (1u << L) - 1u) << (lane - gl);
  float size;
  float z = row_logit(ties.W, ties.h + static_cast<size_t>(row) * ties.d, ties.d, idx, gl, L, group, &size);
  const float least = m - (ties.d / 16 + 9) * 0x1p-20f * size;
  if (second >= least) {
    const Winner win = settle_ties(ties, row, p, chunks, chunk_stride, least, idx, z, gl, L);
    idx = win.idx;
    z = win.z;
  }
  if (!(fabsf(z) < INFINITY && fabsf(m) < INFINITY)) return;
  const float dm = m - z;
  m = z;
  if (fabsf(dm) > 1.0f) return;     // logits so large that neighbouring numbers are further apart
  const float e = exp2f(dm * kLog2e);
  t = e * (t + dm * (s - 1.0f));
  s = 1.0f + e * (s - 1.0f);
}

// Host-side launchers (one per .cu file).  All enqueue on `stream` and return the
// launch error, if any.
struct SimtLaunch {
  const void* W;
  const void* h;
  int n, d, V;
  int chunks;       // vocabulary chunks (partials per row)
  Partial* partials;  // [n][chunks]
};
cudaError_t launch_simt_projection(const SimtLaunch& a, cudaStream_t stream);
void simt_plan(int n, int d, int V, int sm_count, int* chunks, int* grid, int* block, int* smem);

struct FinishLaunch {
  const Partial* partials;  // partial j of row i at partials[i * row_stride + j * chunk_stride]
  bool small_blocks;        // the projection's CTAs leave room for small blocks only (and always with ties to settle)
  int n, chunks;
  int row_stride, chunk_stride;   // [n][chunks]: (chunks, 1); a block gathered shard-major [shards][rows]: (1, rows)
  // optional: before reading the partials, wait until wait_flags[0 .. wait_count) all hold wait_value (flags that
  // other GPUs set after storing their summaries into this GPU's memory); bounded by wait_limit_ns, after which
  // TLR_DEV_WAIT_TIMEOUT is raised and the kernel goes on with what is there
  const uint32_t* wait_flags;
  int wait_count;
  uint32_t wait_value;
  unsigned long long wait_limit_ns;
  float tau;
  const float* mlp_partial;   // optional [n][mlp_blocks]: partial sums of the learned router's output layer
  int mlp_blocks;
  float mlp_b2;
  int decide_on_mlp;          // 1: the learned score is compared with tau instead of conf
  float* mlp_score_out;       // optional [n]: the learned score
  const float* tau_rows;    // optional per-row thresholds [n]
  int route_above;          // 0: route iff conf < tau; 1: route iff conf > tau
  int seq_len;              // > 0: also report the first routed position of every sequence
  int32_t* first_routed;    // [n / seq_len] when seq_len > 0
  int32_t* token;
  float* conf;
  float* entropy;
  uint8_t* route_mask;
  int32_t* routed_idx;
  int32_t* routed_count;
  unsigned int* ticket;     // zero before the launch; the kernel leaves it zero again
  uint32_t* status;
  Ties ties;
  uint32_t* status_copy;    // optional: receives the status word once every row is scored (host-mapped memory)
};
cudaError_t launch_finish(const FinishLaunch& a, cudaStream_t stream);

// Vocabulary-sharded decode (tlr_shard.cu): one summary per row from a shard's chunk partials,
// and the gathered summaries [shards][n] laid out as partials [n][shards].
cudaError_t launch_shard_summary(const Partial* partials, int n, int chunks, int v_offset, const Ties& ties,
                                 Partial* summary, cudaStream_t stream);
// Fused exchange: the summaries are stored straight into slot `rank` of every peer's exchange block and, once all
// rows are out, this rank's flag in every peer's flag array is set to `epoch` (peer stores only).
struct ShardPush {
  const Partial* partials;   // this shard's chunk partials [n][chunks]
  int n, chunks, v_offset;
  Ties ties;
  int shards;                // peers, this rank included
  Partial* const* peer_slot; // device array [shards]: where this rank's n summaries go on peer g
  uint32_t* const* peer_flag;  // device array [shards]: this rank's flag on peer g
  uint32_t epoch;
  unsigned int* ticket;      // zero before the launch; left zero
};
cudaError_t launch_shard_push(const ShardPush& a, cudaStream_t stream);
// Row-sharded batches: the ranks' routed-index lists (slot g = rank g's list, `cap` entries each, the first
// counts[g] valid) become one ascending list of global row numbers, idx + row_offset[g].
cudaError_t launch_rows_merge(const int32_t* gathered_idx, const int32_t* counts, const int32_t* row_offsets,
                              int ranks, int cap, int32_t* global_idx, int32_t* global_count, cudaStream_t stream);

// Copy of `bytes` (a multiple of 16) from host memory the device can read directly to device
// memory, done by a kernel so that the projection kernel behind it can be launched early.
cudaError_t launch_host_copy(const void* src_mapped, void* dst, size_t bytes, cudaStream_t stream);

struct MlpLaunch {
  const void* h;        // bf16 [n][d]
  const void* W1;       // bf16 [d_hidden][d]
  const float* b1;      // [d_hidden]
  const float* w2;      // [d_hidden]
  float b2;
  int n, d, d_hidden;
  float* partial;       // [n][mlp_hidden_blocks(d_hidden)] out
};
int mlp_hidden_blocks(int d_hidden);
cudaError_t launch_mlp_score(const MlpLaunch& a, cudaStream_t stream);
// directly behind a projection launch of tlr_tc_kernel.cuh and beside it; d % 8 == 0, W1 and h 16-byte aligned
cudaError_t launch_mlp_beside(const MlpLaunch& a, cudaStream_t stream);

}  // namespace tlr
