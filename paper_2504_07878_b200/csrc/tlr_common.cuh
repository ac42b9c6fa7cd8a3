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

// Tagged partials.  A kernel that merges partials and stands behind the projection kernel as its programmatic dependent is
// resident, waiting, long before that kernel ends.  Instead of waiting for the end of that grid and reading the partials
// then -- about a microsecond for the grid to drain and the wait to be released, and a trip to L2 behind it -- it may look
// at the partials themselves until they are there.  For that the projection kernel puts the call's tag (1..254) into the
// index's top byte, and the reader leaves every slot it has read as kPendingIdx: a slot with the call's tag holds this
// call's partial.  The tag keeps a reader from taking the partials of the call before, whose merge kernel may still be
// running when this one looks; the reset makes a tag that comes back (after 254 calls, or in a replayed graph) as good as new.
//   * 16 bytes are written and read by one 128-bit access, so that a partial is never seen in part.
//   * The reader's grid starts when every CTA of the projection grid has started, so that looking never keeps a writer from
//     running; and it looks for a bounded number of times only, then waits for the grid like an untagged reader.
//   * A partial that is there says that its CTA has passed its own wait: whatever came before the projection in the stream
//     is complete, and outputs may be written.
//   * The reader waits for the projection grid before it ends, so that who waits for the reader's grid waits for both.
// Tagged steps have partials of their own (no other path writes there).  Per step in a stream with the calls queued ahead (a
// host that asks for one after the other has its own part in the smallest steps), untagged and tagged: n = 1,
// d = 256, V = 20000 7.30 and 6.20 us, n = 16, d = 896, V = 151936 44.26 and 42.90 (8-bit head 28.4 and 27.1), n = 64, d = 300,
// V = 33000 12.31 and 11.57, one of eight shards at n = 256 18.07 and 17.34; n = 256, d = 512, V = 32000 14.5 either way.
constexpr int kTagShift = 24;
constexpr int kTagIdxMask = (1 << kTagShift) - 1;      // an index; all ones stand for kNoToken
constexpr int kPendingIdx = 0;                         // (tag 0; a new workspace is all zeros)
constexpr int kMaxTag = 254;
constexpr int kTaggedPartials = 8 * 16 * 32 * 5;        // of a step: what finish_rows_kernel's lanes can own (328 KB)
constexpr int kMaxLooks = 1 << 14;                     // about 10 ms

__device__ __forceinline__ void store_partial(Partial* dst, const Partial& p) {
  asm volatile("{\n\t.reg .b128 v;\n\t.reg .b64 lo, hi;\n\t"
               "mov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\tmov.b128 v, {lo, hi};\n\t"
               "st.relaxed.gpu.global.b128 [%0], v;\n\t}"
               ::"l"(dst), "f"(p.m), "r"(p.idx), "f"(p.s), "f"(p.t) : "memory");
}
__device__ __forceinline__ Partial load_partial(const Partial* src) {
  Partial p;
  asm volatile("{\n\t.reg .b128 v;\n\t.reg .b64 lo, hi;\n\t"
               "ld.relaxed.gpu.global.b128 v, [%4];\n\tmov.b128 {lo, hi}, v;\n\t"
               "mov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"
               : "=f"(p.m), "=r"(p.idx), "=f"(p.s), "=f"(p.t) : "l"(src) : "memory");
  return p;
}
__device__ __forceinline__ int tagged_idx(int idx, uint32_t tag) {
  return static_cast<int>((static_cast<uint32_t>(idx) & kTagIdxMask) | (tag << kTagShift));
}
__device__ __forceinline__ int untagged_idx(int idx) {
  const int i = idx & kTagIdxMask;
  return i == kTagIdxMask ? kNoToken : i;
}

// Leaves the slots of a lane pending.
__device__ __forceinline__ void reset_tagged(Partial* p, int first, int stride, int count) {
  for (int j = first; j < count; j += stride) p[j].idx = kPendingIdx;
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

// A row without all of its partials is nobody's answer, whatever the projection itself has raised.
__device__ __forceinline__ void note_missing(uint32_t* status) {
  atomicOr(status, TLR_DEV_WAIT_TIMEOUT);
  __threadfence();                         // before this row's flag reaches the block that copies the status word
}

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
  __device__ __forceinline__ void put(int k, const Partial& v, int v_idx) {
    m[k] = v.m;
    s[k] = v.s;
    t[k] = v.t;
    idx = v.m > best ? v_idx : (v.m == best ? min(v_idx, idx) : idx);
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
      put(k, v, v.idx);
    }
  }
  // Tagged partials, chunk stride 1; called by whole warps.  One that is not there when the projection's grid
  // has ended counts as empty, and the status word is told.  hint: look at nothing but the row's last one until it is there.
  // A look is one trip to L2: all of a lane's loads go out before the first is examined (one after the other they took
  // 1.8 us a look).
  __device__ __forceinline__ void take(const Partial* p, int first, int stride, int count, uint32_t tag, bool hint,
                                       uint32_t* status) {
    const auto here = [&](int i) { return (static_cast<uint32_t>(i) >> kTagShift) == tag; };
    Partial v[kN];
    int looks = 0;
    if (hint)
      while (looks < kMaxLooks && !__all_sync(0xffffffffu, count == 0 || here(load_partial(p + count - 1).idx))) ++looks;
    bool waited = false;
    for (;;) {
      bool all = true;
#pragma unroll
      for (int k = 0; k < kN; ++k)
        if (first + stride * k < count) v[k] = load_partial(p + first + stride * k);
#pragma unroll
      for (int k = 0; k < kN; ++k)
        if (first + stride * k < count) all = all && here(v[k].idx);
      if (__all_sync(0xffffffffu, all)) break;
      if (waited) {
        if (!all) note_missing(status);
        break;
      }
      if (++looks >= kMaxLooks) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        waited = true;
      }
    }
    best = -INFINITY;
    idx = kNoToken;
#pragma unroll
    for (int k = 0; k < kN; ++k) {
      const bool there = first + stride * k < count && here(v[k].idx);
      put(k, there ? v[k] : empty_partial(), there ? untagged_idx(v[k].idx) : kNoToken);
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

// Folds one row's partials (tagged ones if tag is not 0; chunk_stride is 1 and `status` the context's word then).  Every lane
// returns the same result.  `second` (optional, untagged only): the largest of the partials' maxima below the row's.
__device__ __forceinline__ Partial fold_row(const Partial* p, int chunks, int chunk_stride, int lane,
                                            float* second = nullptr, uint32_t tag = 0, uint32_t* status = nullptr) {
  Partial r;
  if (tag != 0) {
    LaneFold<kRowsPerLane> f;
    f.take(p, lane, 32, chunks, tag, true, status);
    r.m = f.best;
    r.idx = f.idx;
    group_best(r.m, r.idx, 32);
    f.sums(r.m, r.s, r.t);
    group_sum(r.s, r.t, 32);
    return r;
  }
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
// kFresh: h may have been written since this grid started and is read past L1 (which costs n = 200, d = 999, V = 60000 51.6 -> 56.6 us).
template <bool kPairs, bool kFresh>
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
        if (kFresh) x[i] = kPairs ? __ldcg(reinterpret_cast<const uint32_t*>(h) + k) : __ldcg(h + k);
        else x[i] = kPairs ? reinterpret_cast<const uint32_t*>(h)[k] : h[k];
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
template <bool kFresh>
__device__ __forceinline__ float row_logit(const unsigned short* W, const unsigned short* h, int d, int v, int gl, int L,
                                           unsigned int group, float* size) {
  const unsigned short* w = W + static_cast<size_t>(v) * d;
  for (int k = gl * 64; k < d; k += L * 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(w + k));
  float2 r = (d & 1) == 0 ? lane_logit<true, kFresh>(w, h, d, gl, L) : lane_logit<false, kFresh>(w, h, d, gl, L);
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
template <bool kTagged>
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
      if (__ldcg(&q->m) >= least) {
        mine = __ldcg(&q->idx);
        if (kTagged) mine = mine != kPendingIdx ? untagged_idx(mine) : kNoToken;
      }
    }
    unsigned int todo = __ballot_sync(group, mine < ties.V && mine != idx) & group;
    while (todo != 0u) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int v = __shfl_sync(group, mine, src);
      const float zv = row_logit<kTagged>(ties.W, h, ties.d, v, gl, L, group, &size);
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
template <bool kTagged = false>
__device__ __forceinline__ void settle_row(const Ties& ties, int row, const Partial* __restrict__ p, int chunks,
                                           int chunk_stride, float second, float& m, int& idx, float& s, float& t, int gl,
                                           int L) {
  if (idx >= ties.V) return;
  const unsigned int lane = threadIdx.x & 31;
  const unsigned int group = (L == 32 ? 0xffffffffu : (1u << L) - 1u) << (lane - gl);
  float size;
  float z = row_logit<kTagged>(ties.W, ties.h + static_cast<size_t>(row) * ties.d, ties.d, idx, gl, L, group, &size);
  const float least = m - (ties.d / 16 + 9) * 0x1p-20f * size;
  if (second >= least) {
    const Winner win = settle_ties<kTagged>(ties, row, p, chunks, chunk_stride, least, idx, z, gl, L);
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
  Partial* partials;        // partial j of row i at partials[i * row_stride + j * chunk_stride]
  uint32_t tag;             // not 0: tagged partials, chunk_stride 1 (only where merges_tagged())
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
  uint8_t* flag_bits;       // the rows' flags, ceil(n / 32) words (finish_kernel)
  uint32_t* status;
  Ties ties;
  uint32_t* status_copy;    // optional: receives the status word once every row is scored (host-mapped memory)
};
cudaError_t launch_finish(const FinishLaunch& a, cudaStream_t stream);
bool merges_tagged(int n, int chunks, bool small_blocks);    // whether launch_finish takes tagged partials for this size

// Vocabulary-sharded decode (tlr_shard.cu): one summary per row from a shard's chunk partials,
// and the gathered summaries [shards][n] laid out as partials [n][shards].
// (tag not 0: tagged partials, and `status` is told if some never come)
cudaError_t launch_shard_summary(Partial* partials, uint32_t tag, uint32_t* status, int n, int chunks, int v_offset,
                                 const Ties& ties, Partial* summary, cudaStream_t stream);
// Fused exchange: the summaries are stored straight into slot `rank` of every peer's exchange block and, once all
// rows are out, this rank's flag in every peer's flag array is set to `epoch` (peer stores only).
struct ShardPush {
  Partial* partials;         // this shard's chunk partials [n][chunks]
  uint32_t tag;              // not 0: tagged ones, and
  uint32_t* status;          // ... is told if some never come
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
