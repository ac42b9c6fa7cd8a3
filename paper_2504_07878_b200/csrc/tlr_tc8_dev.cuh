// Device-side pieces that only the 8-bit (e4m3) head needs: the kind::f8f6f4 MMA and its
// instruction descriptor, e4m3 conversions, and the split of bf16 hidden states into two e4m3
// parts written straight into swizzled operand slabs.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace tlr {
namespace {

// D[tmem] (+)= A[smem] * B[smem]^T, e4m3 inputs, fp32 accumulate, K = 32 per instruction.
__device__ __forceinline__ void umma_e4m3(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Instruction descriptor: fp32 accumulator, e4m3 A and B (format code 0), both K-major.
__device__ __forceinline__ uint32_t instr_desc_e4m3(int m_rows, int n_cols) {
  return (1u << 4) | (static_cast<uint32_t>(n_cols >> 3) << 17) | (static_cast<uint32_t>(m_rows >> 4) << 24);
}

// Two halves -> two e4m3 (round to nearest even, saturating), and back.
__device__ __forceinline__ uint16_t to_e4m3x2(uint32_t h2) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(r) : "r"(h2));
  return r;
}
__device__ __forceinline__ uint32_t from_e4m3x2(uint16_t v) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(v));
  return h2;
}

// Where a token's two parts sit in the operand slab.  Up to 64 token rows they alternate in groups of eight -- rows
// 16g .. 16g + 7 hold the first parts of tokens 8g .. 8g + 7, the next eight their second parts -- so that one thread
// of the epilogue's fragment layout holds both sums of a token; above, the first parts of all rows come first.
__host__ __device__ __forceinline__ int tc8_part_row(int row, int part_rows) {
  return part_rows > 64 ? row : (row >> 3) * 16 + (row & 7);
}
__host__ __device__ __forceinline__ int tc8_part_stride(int part_rows) { return part_rows > 64 ? part_rows : 8; }

// The power of two r that puts a row's largest magnitude amax into [128, 256) after division.
__device__ __forceinline__ float split_scale(float amax) {
  float r = 1.0f;
  if (amax > 0.f && amax < INFINITY) {
    int e;
    frexpf(amax, &e);                 // amax = f * 2^e, f in [0.5, 1)
    e = e - 8 < -126 ? -126 : (e - 8 > 126 ? 126 : e - 8);   // keeps r and 1/r finite and normal
    r = ldexpf(1.0f, e);
  }
  return r;
}

// x * inv as the sum of two e4m3 numbers: p1 = round(x), p2 = round(x - p1), two elements at a time and in halves: down to
// 2^-17 a bf16 number below 256 is a half, and below that both parts are zero (e4m3's smallest step is 2^-9).
// (In floats, with the magnitudes compared one by one: n = 16, d = 896, V = 151936 26.9 us per step (calls queued ahead), so
// 26.5; n = 32, d = 512, V = 30000 9.36 and 9.19.)
__device__ __forceinline__ void split_pair(float x0, float x1, uint16_t& p1, uint16_t& p2) {
  const __half2 x = __floats2half2_rn(x0, x1);
  p1 = to_e4m3x2(*reinterpret_cast<const uint32_t*>(&x));
  const uint32_t back = from_e4m3x2(p1);
  const __half2 rest = __hsub2(x, *reinterpret_cast<const __half2*>(&back));
  p2 = to_e4m3x2(*reinterpret_cast<const uint32_t*>(&rest));
}

// The larger magnitudes of the pair m and of eight bf16, pair by pair (NaNs are dropped), and the larger of a pair.
__device__ __forceinline__ uint32_t abs_max8(uint32_t m, const uint4& v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t a = w[j] & 0x7fff7fffu;
    asm("max.bf16x2 %0, %0, %1;" : "+r"(m) : "r"(a));
  }
  return m;
}
__device__ __forceinline__ float larger_of(uint32_t pair) {
  return fmaxf(__uint_as_float(pair << 16), __uint_as_float(pair & 0xffff0000u));
}

// Sixteen bf16 (lo, hi), times inv, as first parts q1 and second parts q2.
__device__ __forceinline__ void split16(const uint4& lo, const uint4& hi, float inv, uint4& q1, uint4& q2) {
  const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
  uint32_t a[4] = {0u, 0u, 0u, 0u}, b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < 8; ++j) {                                // two elements per 32-bit word
    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[j]));
    uint16_t p1, p2;
    split_pair(f.x * inv, f.y * inv, p1, p2);
    a[j >> 1] |= static_cast<uint32_t>(p1) << (16 * (j & 1));
    b[j >> 1] |= static_cast<uint32_t>(p2) << (16 * (j & 1));
  }
  q1 = make_uint4(a[0], a[1], a[2], a[3]);
  q2 = make_uint4(b[0], b[1], b[2], b[3]);
}

// Splits the (at most 16) rows of h into resident operand slabs, done by 288 threads numbered t (the caller's
// warps 2..10; they synchronise among themselves with named barrier 1).  Slab ks is 32 rows of 128 bytes
// with the 128-byte swizzle TMA would have produced, the two parts in alternating groups of eight rows
// (tc8_part_row); the 16-byte chunk c of row r sits at position c ^ (r & 7).  hs_s[r] receives row r's scale
// (hs_s[32 + r] is scratch).  One pass over h: 18 threads per row, each keeps its (at most kSplitChunks) chunks of
// 16 elements in registers between the maximum and the conversion, so the row is read from memory once and all
// loads are in flight together.
constexpr int kSplitThreads = 288;
constexpr int kSplitLanes = kSplitThreads / 16;       // threads per row
constexpr int kSplitChunks = 6;                       // chunks of 16 elements per thread: 108 per row, 13 whole slabs of 8, d <= 1664
__device__ __forceinline__ void split_h_resident(const __nv_bfloat16* __restrict__ hb, int n, int d, int k_slabs,
                                                 unsigned char* slabs, float* hs_s, int t) {
  const int r = t / kSplitLanes, l = t - r * kSplitLanes;
  const int valid_chunks = d >> 4;                          // d is a multiple of 16
  uint4 va[kSplitChunks], vb[kSplitChunks];
  uint32_t amax = 0u;
#pragma unroll
  for (int i = 0; i < kSplitChunks; ++i) {
    const int c = l + kSplitLanes * i;
    va[i] = make_uint4(0u, 0u, 0u, 0u);
    vb[i] = va[i];
    if (r < n && c < valid_chunks) {
      const uint4* src = reinterpret_cast<const uint4*>(hb + static_cast<size_t>(r) * d + c * 16);
      va[i] = __ldcg(src);        // (not the read-only path: h may still have been on its way when this kernel started)
      vb[i] = __ldcg(src + 1);
    }
  }
#pragma unroll
  for (int i = 0; i < kSplitChunks; ++i) amax = abs_max8(abs_max8(amax, va[i]), vb[i]);
  // the row's largest magnitude: non-negative floats order like their bit patterns
  unsigned int* amax_bits = reinterpret_cast<unsigned int*>(hs_s + 32);
  if (t < 16) amax_bits[t] = 0u;
  asm volatile("bar.sync 1, %0;" ::"n"(kSplitThreads) : "memory");   // only the splitting warps; nothing asynchronous is waited for
  atomicMax(amax_bits + r, __float_as_uint(larger_of(amax)));    // (NaNs are dropped: a number >= 0)
  asm volatile("bar.sync 1, %0;" ::"n"(kSplitThreads) : "memory");
  const float sc = split_scale(__uint_as_float(amax_bits[r]));
  if (l == 0) hs_s[r] = sc;
  const float inv = 1.0f / sc;                                   // exact: a power of two
#pragma unroll
  for (int i = 0; i < kSplitChunks; ++i) {
    const int cc = l + kSplitLanes * i;
    if (cc >= k_slabs * 8) continue;                             // (chunks between d and the slab's end are zeros)
    const int ks = cc >> 3, c = cc & 7;
    uint4 q1, q2;
    split16(va[i], vb[i], inv, q1, q2);
    unsigned char* dst = slabs + ks * 4096 + tc8_part_row(r, 16) * 128 + ((c ^ (r & 7)) << 4);
    *reinterpret_cast<uint4*>(dst) = q1;
    *reinterpret_cast<uint4*>(dst + 1024) = q2;
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic stores -> the MMA's (async proxy) reads
}

}  // namespace
}  // namespace tlr
