// Merge of the per-chunk partial results, the scores, the route decision and the
// ordered stream compaction of routed rows -- one launch.
//
// Per row (a group of lanes, a whole warp for large n): lanes stride the row's partials; a shuffle butterfly finds the
// global maximum and its lowest index, each lane rescales its own partials to that
// maximum once, and a second butterfly adds the sums.  Lane 0 writes token,
// conf = 1/s, entropy = ln s - t/s and the route flag conf < tau (Sec. 3.1 of the
// paper: routed when the score falls below the threshold).
//
// Compaction (ballot / popcount / prefix sum, ascending order):
//   n <= 1024  a thread-block cluster of up to 8 blocks folds the rows (a group of L lanes
//              per row, all rows at once) and sends the route flags to block 0, which compacts
//              them.  No ticket, no second launch, one L2 round trip for the partials.
//              finish_rows_kernel where a lane owns at most 5 partials: the compaction has a warp
//              of its own.  Otherwise finish_small_kernel, 512 threads where a lane still owns
//              at most 6 partials (else 1024, and where that is not enough, the kernel for larger n; so, too,
//              with four lanes and ties to settle).  Blocks of 17 or 9 warps, and of 512 threads, fit on an
//              SM beside a CTA of the tensor-core projection kernel, so
//              the blocks are resident and waiting before that kernel ends, and the next
//              call's CTAs do not have to wait for the merge to leave their SMs.
//   larger n   many blocks of 8 warps, which leave their rows' flags as bits; the block that
//              finishes last (fence + ticket counter, no spinning) compacts those of all rows.
#include "tlr_common.cuh"
#include "tlr_tc.cuh"

namespace tlr {

constexpr int kFinishWarps = 8;
constexpr int kFinishThreads = kFinishWarps * 32;
constexpr int kSmallThreads = 1024;
constexpr int kSmallRows = 1024;
constexpr int kMaxBlocks = 8;           // of a cluster

// Scores and decision of one row from its folded summary.  The flag, which the compaction waits for, needs no entropy.
struct Scored {
  float conf, learned;
  int flag;
  bool finite;
};
__device__ __forceinline__ Scored decide_row(float s, float t, const FinishLaunch& a, int row) {
  Scored r;
  r.conf = 1.0f / s;
  r.finite = s > 0.f && s < INFINITY && t == t;        // (and so are both scores no NaN)
  if (r.finite) {
    r.conf = fminf(r.conf, 1.0f);
  } else {
    r.conf = __int_as_float(0x7fc00000);   // NaN: fails "conf >= tau", so the row is routed
    atomicOr(a.status, TLR_DEV_NONFINITE);
    __threadfence();                       // before this row's flag reaches the block that copies the status word
  }
  // "not (conf >= tau)": equals conf < tau for numbers, and routes a NaN row; likewise
  // "not (conf <= tau)" for the opposite polarity.
  const float tau = a.tau_rows != nullptr ? __ldcg(a.tau_rows + row) : a.tau;
  float score = r.conf;
  r.learned = 0.f;
  if (a.mlp_partial != nullptr) {
    // learned score: the output layer's partial sums in a fixed order, then the sigmoid
    float v = a.mlp_b2;
#pragma unroll 8
    for (int b = 0; b < a.mlp_blocks; ++b) v += __ldcg(a.mlp_partial + static_cast<size_t>(row) * a.mlp_blocks + b);
    r.learned = 1.0f / (1.0f + expf(-v));
    if (a.decide_on_mlp) score = r.learned;
  }
  r.flag = a.route_above ? ((score <= tau) ? 0 : 1) : ((score >= tau) ? 0 : 1);
  return r;
}
__device__ __forceinline__ void store_row(const Scored& r, int token, float s, float t, const FinishLaunch& a, int row) {
  a.token[row] = token;
  a.conf[row] = r.conf;
  a.entropy[row] = r.finite ? fmaxf(logf(s) - t / s, 0.0f) : r.conf;
  a.route_mask[row] = static_cast<uint8_t>(r.flag);
  if (a.mlp_partial != nullptr && a.mlp_score_out != nullptr) a.mlp_score_out[row] = r.learned;
}

// First routed position of every sequence: an atomic minimum per sequence over the
// routed rows.  Called by the one block that compacts, before (init) and during the pass.
__device__ __forceinline__ void first_routed_init(const FinishLaunch& a) {
  if (a.seq_len > 0) {
    for (int b = threadIdx.x; b < a.n / a.seq_len; b += blockDim.x) a.first_routed[b] = a.seq_len;
    __syncthreads();
  }
}
__device__ __forceinline__ void first_routed_note(const FinishLaunch& a, int row) {
  if (a.seq_len > 0) atomicMin(a.first_routed + row / a.seq_len, row % a.seq_len);
}

// Programmatic dependent launch: let the next kernel in the stream be scheduled now (it
// waits for this grid to complete before touching memory), then wait for the projection
// kernel's partials.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() {
  pdl_trigger();
  pdl_wait();
}

// Vocabulary-sharded step with the fused exchange: the other GPUs store their summaries into this GPU's
// memory and then set a flag each.  Warp 0 of every block polls the flags (lane g watches flag g, g + 32, ...)
// with acquire loads at system scope until all hold the expected value or the time limit runs out; the
// block then goes on either way (after a time-out the status word says the outputs are not to be trusted).
__device__ __forceinline__ void wait_for_peers(const FinishLaunch& a) {
  if (a.wait_flags == nullptr) return;
  if (threadIdx.x < 32) {
    unsigned long long t0 = 0;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (;;) {
      bool mine = true;
      for (int g = threadIdx.x; g < a.wait_count; g += 32) {
        uint32_t v;
        asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(a.wait_flags + g) : "memory");
        mine = mine && (v == a.wait_value);
      }
      if (__all_sync(0xffffffffu, mine)) break;
      unsigned long long t1;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t1));
      if (__any_sync(0xffffffffu, t1 - t0 > a.wait_limit_ns)) {
        if (threadIdx.x == 0) atomicOr(a.status, TLR_DEV_WAIT_TIMEOUT);
        break;
      }
      __nanosleep(200);
    }
  }
  __syncthreads();
}

// The barrier of block 0 that counts the bytes of `words` words, and a warp's word on its way there.
__device__ __forceinline__ void expect_words(uint32_t bar, int words) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(words * 4) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void send_word(const uint32_t* slot, uint32_t bar, uint32_t word) {
  const uint32_t at = static_cast<uint32_t>(__cvta_generic_to_shared(slot));
  uint32_t remote, remote_bar;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(at), "r"(0));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote_bar) : "r"(bar), "r"(0));
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
               ::"r"(remote), "r"(word), "r"(remote_bar) : "memory");
}
// Row i's flag in the words of warps with L lanes to a row.
__device__ __forceinline__ int flag_of(const uint32_t* words, int i, int log2_L) {
  const int log2_rpw = 5 - log2_L;
  return (words[i >> log2_rpw] >> ((i & ((1 << log2_rpw) - 1)) << log2_L)) & 1;
}

__device__ __forceinline__ bool words_here(uint32_t bar) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar) : "memory");
  return ok != 0u;
}
// Block 0 of the cluster waits until every warp's word has arrived; false if it gave up.  Bounded like every wait, and what the
// limit covers is the cluster's own blocks: nothing the projection waits for -- a kernel in front of it may wait for seconds
// for other GPUs -- counts.  So where the others look for their partials themselves (kTagged) this one looks for a while and
// then waits for the projection's grid before its clock starts.
template <bool kTagged>
__device__ __forceinline__ bool wait_for_words(uint32_t bar, uint32_t* status) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (words_here(bar)) return true;
    if ((it & 63u) == 63u && (!kTagged || it >= kMaxLooks)) {
      if (kTagged && t0 == 0) pdl_wait();
      unsigned long long t;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
      if (t0 == 0) t0 = t;
      if (t - t0 > 2000000000ull) {
        atomicOr(status, TLR_DEV_WAIT_TIMEOUT);
        return false;
      }
    }
  }
}
// After a time-out no row is listed, and block 0 stays until no other block can send to it any more (threads that have exited
// count as arrived).  By whole warps.
__device__ __forceinline__ void outlive_senders() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
constexpr int kNoList = -2 * kSmallRows;      // a warp's count after a time-out: the sum is below zero with it

// Cluster of gridDim.x blocks, n <= 1024.  A group of L lanes (L a power of two) folds one
// row: maximum and index first, then the sums rescaled to
// that maximum.  L is chosen on the host so that every row has its group, n * L <=
// gridDim.x * 1024, and a lane at most kPerLane partials.
template <bool kTies>
__device__ __forceinline__ void finish_small(const FinishLaunch& a, const int log2_L) {
  __shared__ int warp_count[kSmallThreads / 32];
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int L = 1 << log2_L;
  const int group = (blockIdx.x * blockDim.x + threadIdx.x) >> log2_L;
  const int gl = threadIdx.x & (L - 1);
  // Every warp of the cluster sends the flags of its 32 / L rows -- bit r * L for its row r -- as one word to block 0,
  // which waits for all words on a barrier of its own.  (st.async delivers the word and its arrival in one trip: n = 64, d = 512, V = 32000 11.90 us per step; flag
  // bytes in distributed shared memory with a cluster barrier behind them 12.96; n = 256 14.61 and 15.55.)
  __shared__ uint32_t flag_words[kSmallRows / 4];     // at most 8 blocks x 32 warps
  __shared__ __align__(8) unsigned long long all_here;
  const bool single_block = gridDim.x == 1;
  const int warps = blockDim.x >> 5;
  const uint32_t bar = static_cast<uint32_t>(__cvta_generic_to_shared(&all_here));
  if (!single_block) {
    if (blockIdx.x == 0 && threadIdx.x == 0) expect_words(bar, gridDim.x * warps);
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  pdl_enter();
  wait_for_peers(a);
  const int row = group;
  const bool valid = row < a.n;
  Scored out = {};
  int out_token;
  float out_s, out_t;
  {
    const Partial* p = a.partials + static_cast<size_t>(valid ? row : 0) * a.row_stride;
    const int cs = a.chunk_stride;
    float m = -INFINITY;
    int idx = kNoToken;
    float s = 0.f, t = 0.f, second = -INFINITY;
    {
      // one pass, the partials stay in registers: every load goes out before the first is looked at, and behind the last
      // partial the last one is loaded again
      Partial q[kPerLane];
      if (valid) {
#pragma unroll
        for (int k = 0; k < kPerLane; ++k) {
          const float4 raw = __ldcg(reinterpret_cast<const float4*>(p + min(gl + L * k, a.chunks - 1) * cs));
          q[k].m = raw.x;
          q[k].idx = __float_as_int(raw.y);
          q[k].s = raw.z;
          q[k].t = raw.w;
        }
      }
#pragma unroll
      for (int k = 0; k < kPerLane; ++k) {
        if (!valid || gl + L * k >= a.chunks) q[k] = empty_partial();
        if (q[k].m > m || (q[k].m == m && q[k].idx < idx)) {
          m = q[k].m;
          idx = q[k].idx;
        }
      }
      for (int off = L >> 1; off > 0; off >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, off);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
        if (om > m || (om == m && oi < idx)) {
          m = om;
          idx = oi;
        }
      }
#pragma unroll
      for (int k = 0; k < kPerLane; ++k) {
        if (!(q[k].s == 0.f)) {         // an empty range contributes nothing; a NaN sum goes through
          const float dm = q[k].m - m;  // <= 0
          const float e = exp2f(dm * kLog2e);
          s += q[k].s * e;
          t += e * (q[k].t + dm * q[k].s);
        }
        if constexpr (kTies) second = q[k].m < m ? fmaxf(second, q[k].m) : second;
      }
    }
    for (int off = L >> 1; off > 0; off >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, off);
      t += __shfl_xor_sync(0xffffffffu, t, off);
      if constexpr (kTies) second = fmaxf(second, __shfl_xor_sync(0xffffffffu, second, off));
    }
    if constexpr (kTies) {
      if (valid) settle_row(a.ties, row, p, a.chunks, a.chunk_stride, second, m, idx, s, t, gl, L);
    }
    if (valid && gl == 0) out = decide_row(s, t, a, row);
    out_token = idx;
    out_s = s;
    out_t = t;
  }
  const uint32_t word = __ballot_sync(0xffffffffu, valid && gl == 0 && out.flag != 0);
  if (lane == 0) {
    if (single_block) flag_words[warp] = word;
    else send_word(&flag_words[blockIdx.x * warps + warp], bar, word);
  }
  if (valid && gl == 0) store_row(out, out_token, out_s, out_t, a, row);
  if (blockIdx.x != 0) return;
  bool here = true;
  if (single_block) __syncthreads();
  else here = __all_sync(0xffffffffu, wait_for_words<false>(bar, a.status));
  first_routed_init(a);
  const int log2_rpw = 5 - log2_L;          // rows per warp
  int base_out = 0;
  for (int base = 0; base < a.n; base += blockDim.x) {       // one pass when the block has a thread per row
    const int i = base + threadIdx.x;
    const int flag = i < a.n ? (flag_words[i >> log2_rpw] >> ((i & ((1 << log2_rpw) - 1)) << log2_L)) & 1u : 0;
    const unsigned int bal = __ballot_sync(0xffffffffu, flag != 0);
    if (lane == 0) warp_count[warp] = here ? __popc(bal) : kNoList;
    __syncthreads();
    // at most 32 warps: lane w holds warp w's count
    const int c = lane < warps ? warp_count[lane] : 0;
    const int before = __reduce_add_sync(0xffffffffu, lane < warp ? c : 0);
    if (flag && base_out + before >= 0) {
      a.routed_idx[base_out + before + __popc(bal & ((1u << lane) - 1u))] = i;
      first_routed_note(a, i);
    }
    base_out += __reduce_add_sync(0xffffffffu, c);
    if (base + static_cast<int>(blockDim.x) < a.n) __syncthreads();
  }
  if (threadIdx.x == 0) {
    *a.routed_count = max(base_out, 0);
    if (a.status_copy != nullptr) *a.status_copy = atomicOr(a.status, 0u);   // every row has been scored by now
  }
  if (base_out < 0) outlive_senders();
}

// The same for steps whose lanes own few partials (rows_shape), and then what stands between the last partial and the end of
// the step is latency alone: the compaction has a warp of its own -- the last one of block 0 -- that waits for the words and
// does it while the others still work out their entropies and store their rows.  Per step in a stream, calls queued ahead,
// with finish_small_kernel and with this one (partials not tagged): n = 1, d = 256, V = 20000 8.36 and 7.30 us, n = 16, d = 896, V = 151936 45.73 and 44.26
// (8-bit head 30.0 and 28.4), n = 64, d = 512, V = 32000 12.24 and 11.03, n = 128 there 13.26 and 12.13.
// kTagged: the partials are tagged ones (tlr_common.cuh), no peers and no learned router.
// kRowWarps: 16, or 8 where a block of 17 warps would not stand beside a CTA of the projection.  No register may be spilled: a kernel that writes local memory ends a
// microsecond later (four bytes of it, n = 1, d = 256, V = 20000: 6.2 and 7.6 us per step).
template <bool kTies, bool kTagged, int kRowWarps>
__global__ void __maxnreg__(kTies ? 64 : 40)
finish_rows_kernel(const FinishLaunch a, const int log2_L) {
  constexpr int row_warps = kRowWarps;
  __shared__ uint32_t flag_words[kMaxBlocks * kRowWarps];
  __shared__ __align__(8) unsigned long long all_here;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t bar = static_cast<uint32_t>(__cvta_generic_to_shared(&all_here));
  if (blockIdx.x == 0 && threadIdx.x == 0) expect_words(bar, gridDim.x * row_warps);
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  pdl_trigger();
  if constexpr (!kTagged) {
    pdl_wait();
    wait_for_peers(a);
  }
  if (warp < row_warps) {
    const int L = 1 << log2_L;
    const int row = (blockIdx.x * row_warps * 32 + threadIdx.x) >> log2_L;
    const int gl = threadIdx.x & (L - 1);
    const bool valid = row < a.n;
    const int count = valid ? a.chunks : 0;
    Partial* p = a.partials + static_cast<size_t>(valid ? row : 0) * a.row_stride;
    LaneFold<kRowsPerLane> f;
    if constexpr (kTagged) f.take(p, gl, L, count, a.tag, gridDim.x > 1, a.status);
    else f.load(p, gl, L, count, static_cast<size_t>(a.chunk_stride));
    float m = f.best, s, t;
    int idx = f.idx;
    group_best(m, idx, L);
    f.sums(m, s, t);
    group_sum(s, t, L);
    if constexpr (kTies) {
      const float second = group_max(f.second(m), L);
      if (valid) settle_row<kTagged>(a.ties, row, p, a.chunks, a.chunk_stride, second, m, idx, s, t, gl, L);
    }
    const bool mine = valid && gl == 0;
    Scored out = {};
    if (mine) out = decide_row(s, t, a, row);
    const uint32_t word = __ballot_sync(0xffffffffu, out.flag != 0);
    if (lane == 0) send_word(&flag_words[blockIdx.x * row_warps + warp], bar, word);
    if (mine) store_row(out, idx, s, t, a, row);
    if (kTagged && valid) reset_tagged(p, gl, L, a.chunks);
  } else if (blockIdx.x == 0) {
    const bool here = __all_sync(0xffffffffu, wait_for_words<kTagged>(bar, a.status));
    if (a.seq_len > 0) {
      for (int b = lane; b < a.n / a.seq_len; b += 32) a.first_routed[b] = a.seq_len;
      __syncwarp();
    }
    if (__builtin_expect(!here, 0)) {
      if (lane == 0) {
        *a.routed_count = 0;
        if (a.status_copy != nullptr) *a.status_copy = atomicOr(a.status, 0u);
      }
      outlive_senders();
      return;
    }
    // (A scan over the words, every lane writing the rows of its own, took a microsecond at n = 1 and more than this loop's
    // eight turns at n = 256.)
    int total = 0;
    for (int base = 0; base < a.n; base += 32) {
      const int i = base + lane;
      const int flag = i < a.n ? flag_of(flag_words, i, log2_L) : 0;
      const unsigned int bal = __ballot_sync(0xffffffffu, flag != 0);
      if (flag) {
        a.routed_idx[total + __popc(bal & ((1u << lane) - 1u))] = i;
        first_routed_note(a, i);
      }
      total += __popc(bal);
    }
    if (lane == 0) *a.routed_count = total;
    if (kTagged) pdl_wait();
    if (lane == 0 && a.status_copy != nullptr) *a.status_copy = atomicOr(a.status, 0u);   // every row has been scored by now
  }
}

// 32 registers, none spilled (which costs 2 to 4 % of most small steps), and a lane's loads all in flight: with 36 and a
// condition per load n = 765, d = 976, V = 3005 13.5 instead of 13.0 us, n = 542, d = 888, V = 7195 17.1 and 16.7, n = 700, d = 400,
// V = 20000 19.1 and 18.6 (but n = 619, d = 160, V = 19901 16.1 and 16.4).
__global__ void __maxnreg__(32)
finish_small_kernel(const FinishLaunch a, const int log2_L) {
  finish_small<false>(a, log2_L);
}

// With settle_row, which would cost the other one registers; 40 is the most that lets a block of 512 threads stand beside a
// CTA of the projection kernel for d % 8 != 0.
__global__ void __maxnreg__(40)
finish_small_ties_kernel(const FinishLaunch a, const int log2_L) {
  finish_small<true>(a, log2_L);
}

template <bool kTies>
__global__ void __launch_bounds__(kFinishThreads)
finish_kernel(const FinishLaunch a) {
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * kFinishWarps + warp;
  pdl_enter();
  wait_for_peers(a);

  __shared__ int warp_flag[kFinishWarps];
  int flag = 0;
  if (row < a.n) {
    const Partial* p = a.partials + static_cast<size_t>(row) * a.row_stride;
    float second;
    Partial acc = fold_row(p, a.chunks, a.chunk_stride, lane, kTies ? &second : nullptr);
    if constexpr (kTies)
      settle_row(a.ties, row, p, a.chunks, a.chunk_stride, second, acc.m, acc.idx, acc.s, acc.t, lane, 32);
    if (lane == 0) {
      const Scored r = decide_row(acc.s, acc.t, a, row);
      store_row(r, acc.idx, acc.s, acc.t, a, row);
      flag = r.flag;
    }
  }
  if (lane == 0) warp_flag[warp] = flag;

  // ---- which block is last?
  __shared__ int is_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int bits = 0;
#pragma unroll
    for (int w = 0; w < kFinishWarps; ++w) bits |= static_cast<unsigned int>(warp_flag[w] != 0) << w;
    a.flag_bits[blockIdx.x] = static_cast<uint8_t>(bits);      // row i: bit i % 8 of byte i / 8
    __threadfence();
    const unsigned int t = atomicAdd(a.ticket, 1u);
    is_last = (t == gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();

  // ---- ordered compaction by the last block, which everything behind it in the stream waits for.  The flags are bits: a thread
  // has 64 rows, a pass 16384, and the second half of a pass writes word by word, a lane to a row.  (From the flag bytes of the
  // output, 256 rows a pass with a trip to L2 and two barriers each, over PCIe where the outputs are in host memory: n = 2000,
  // d = 256, V = 20000 33.4 us per step, so 31.2, n = 16384 there 228.5 and 211.5; n = 4000, d = 512, V = 30000 from and to host
  // memory 241 and 218.  Words through shuffles instead of shared memory, so that these blocks stand beside the projection's
  // CTAs: n = 2000 31.5 and 32.8.)
  first_routed_init(a);
  __shared__ unsigned int word_of[2 * kFinishThreads];
  __shared__ int before_of[2 * kFinishThreads];
  __shared__ int warp_count[kFinishWarps];
  const int words = (a.n + 31) >> 5;
  int base_out = 0;
  for (int base = 0; base < words; base += 2 * kFinishThreads) {
    unsigned int m[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int w = base + 2 * threadIdx.x + k;
      m[k] = w < words ? __ldcg(reinterpret_cast<const unsigned int*>(a.flag_bits) + w) : 0u;
      if (w == words - 1 && (a.n & 31) != 0) m[k] &= (1u << (a.n & 31)) - 1u;
    }
    const int mine = __popc(m[0]) + __popc(m[1]);
    int upto = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, upto, off);
      if (lane >= off) upto += v;
    }
    if (lane == 31) warp_count[warp] = upto;
    __syncthreads();
    int before = upto - mine, total = 0;
#pragma unroll
    for (int w = 0; w < kFinishWarps; ++w) {
      const int c = warp_count[w];
      before += (w < warp) ? c : 0;
      total += c;
    }
    word_of[2 * threadIdx.x] = m[0];
    word_of[2 * threadIdx.x + 1] = m[1];
    before_of[2 * threadIdx.x] = base_out + before;
    before_of[2 * threadIdx.x + 1] = base_out + before + __popc(m[0]);
    __syncthreads();
    const int here = min(words - base, 2 * kFinishThreads);
#pragma unroll 4
    for (int w = warp; w < here; w += kFinishWarps) {
      const unsigned int word = word_of[w];
      if ((word >> lane) & 1u) {
        const int i = 32 * (base + w) + lane;
        a.routed_idx[before_of[w] + __popc(word & ((1u << lane) - 1u))] = i;
        first_routed_note(a, i);
      }
    }
    base_out += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    *a.routed_count = base_out;
    if (a.status_copy != nullptr) *a.status_copy = atomicOr(a.status, 0u);
    *a.ticket = 0u;  // ready for the next call on this context
  }
}

namespace {

// The launch of the small merge kernel for n <= kSmallRows rows.
struct SmallShape {
  int blocks, threads, lanes;      // lanes: 0 where a lane would own more than kPerLane partials
};
SmallShape small_shape(int n, int chunks) {
  SmallShape s;
  s.blocks = 1;
  while (s.blocks < 8 && s.blocks * 16 < n) s.blocks <<= 1;       // 16 rows per block until 8 blocks
  // 512-thread blocks fit on an SM beside a CTA of the tensor-core projection kernel, so they
  // are resident (waiting) before it ends and do not keep the next call's CTAs off their SMs;
  // they are used whenever a lane group still owns few enough partials for the one-pass fold.
  const auto lanes_for = [&](int threads) {
    int l = 32;
    while (l > 1 && n * l > s.blocks * threads) l >>= 1;
    return l;
  };
  s.threads = kSmallThreads;
  if ((chunks + lanes_for(512) - 1) / lanes_for(512) <= kPerLane) s.threads = 512;
  const int e = tuning().finish_threads;   // tuning switch (TLR_FINISH_THREADS)
  if (e == 256 || e == 512 || e == 1024) s.threads = e;
  s.lanes = lanes_for(s.threads);
  // Eight blocks that walk a row's partials twice take 12 us, many blocks with a warp to a row 6: n = 640, d = 256, V = 18944
  // (49 partials, eight lanes) 21.8 and 17.3 us per step.  With at most kPerLane to a lane the eight blocks are the faster ones:
  // V = 60000 there (37 partials) 30.9 and 32.5.
  if ((chunks + s.lanes - 1) / s.lanes > kPerLane) s.lanes = 0;
  return s;
}

}  // namespace

// finish_rows_kernel for n rows of `chunks` partials: row warps per block, blocks and lanes per row; false where a lane would own
// more than kRowsPerLane partials.  small: blocks of 8 row warps.
bool rows_shape(int n, int chunks, bool small, int* row_warps, int* blocks, int* lanes) {
  if (n <= 0 || n > kSmallRows) return false;
  // Eight row warps as long as eight blocks of them give every row a warp: 8 and 16 at n = 16, d = 512, V = 32000 9.5 and 9.9 us,
  // n = 64 11.1 and 11.3; where only such blocks stand beside the projection's CTAs (64 rows of the 8-bit head, d = 896,
  // V = 60000) 18.0 and 19.0.
  *row_warps = small || n <= 8 * kMaxBlocks ? 8 : 16;
  *blocks = 1;
  while (*blocks < kMaxBlocks && *blocks * *row_warps < n) *blocks <<= 1;
  *lanes = 32;
  while (*lanes > 1 && n * *lanes > *blocks * *row_warps * 32) *lanes >>= 1;
  return n * *lanes <= *blocks * *row_warps * 32 && (chunks + *lanes - 1) / *lanes <= kRowsPerLane;
}

bool merges_tagged(int n, int chunks, bool small) {
  int row_warps, blocks, lanes;
  return rows_shape(n, chunks, small, &row_warps, &blocks, &lanes);
}

cudaError_t launch_finish(const FinishLaunch& a, cudaStream_t stream) {
  if (a.chunks > 32 * kPerLane) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int blocks = 0, threads = 0, lanes = 0, row_warps;
  const bool ties = a.ties.W != nullptr;
  auto kernel = ties ? finish_small_ties_kernel : finish_small_kernel;
  if (rows_shape(a.n, a.chunks, a.small_blocks, &row_warps, &blocks, &lanes)) {
    threads = (row_warps + 1) * 32;
    if (ties) kernel = a.tag != 0 ? finish_rows_kernel<true, true, 8> : finish_rows_kernel<true, false, 8>;
    else if (row_warps == 8) kernel = a.tag != 0 ? finish_rows_kernel<false, true, 8> : finish_rows_kernel<false, false, 8>;
    else kernel = a.tag != 0 ? finish_rows_kernel<false, true, 16> : finish_rows_kernel<false, false, 16>;
  } else if (a.tag != 0) {          // (tagged partials are rows_shape's only, see merges_tagged)
    return cudaErrorInvalidValue;
  } else if (a.n <= kSmallRows) {
    const SmallShape s = small_shape(a.n, a.chunks);
    blocks = s.blocks;
    threads = s.threads;
    // Settling a row's winner reads a row of W and of h by the row's lanes, beside the projection's shared memory with hardly any
    // L1: with four lanes that takes longer than all the rest, and by how much changes with the order of the loads.  So a warp
    // to a row in many blocks: n = 529, d = 522, V = 4165 36.0 and 21.1 us per step, n = 602, d = 794, V = 54687 125 and 80,
    // n = 740, d = 204, V = 16622 24.5 and 22.8; short rows take longer there, n = 856, d = 108, V = 16628 22.3 and 23.4, and so do
    // some with eight lanes, n = 480, d = 141, V = 40408 25.8 and 26.6.
    lanes = ties && s.lanes < 8 && a.ties.d > 128 ? 0 : s.lanes;
  } else {
    lanes = 0;
  }
  if (lanes > 0) {
    int log2_L = 0;
    while ((1 << log2_L) < lanes) ++log2_L;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(blocks);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;      // (a single block, too, is launched as a cluster: mapa and st.async are illegal without one)
    cfg.gridDim = dim3(static_cast<unsigned>(blocks), 1, 1);
    cfg.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
    return cudaLaunchKernelEx(&cfg, kernel, a, log2_L);
  }
  if (a.flag_bits == nullptr) return cudaErrorInvalidValue;
  cfg.gridDim = dim3(static_cast<unsigned>((a.n + kFinishWarps - 1) / kFinishWarps), 1, 1);
  cfg.blockDim = dim3(kFinishThreads, 1, 1);
  return cudaLaunchKernelEx(&cfg, ties ? finish_kernel<true> : finish_kernel<false>, a);
}

}  // namespace tlr
