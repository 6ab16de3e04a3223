// Device helpers shared by the probe kernels.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "tc_ptx.cuh"

namespace lc {

// Per-query reduction word of an accepted pair: IEEE bits of the FP32
// squared distance (non-negative, so bit order = value order) above the
// cache index; atomicMin keeps the nearest hit and, on equal distances, the
// lowest index (Eq. 14).
__device__ __forceinline__ unsigned long long pack_hit(float dist2, int64_t index) {
  return ((unsigned long long)__float_as_uint(dist2) << 32) | (unsigned long long)(uint32_t)index;
}

// Canonical FP32 squared distance sum_j (q_j - k_j)^2 over d_pad (multiple
// of 32) zero-padded features: a 32-wide fused-multiply-add chain per chunk,
// chunk sums added in order. Every probe path evaluates exactly this
// sequence of rounded operations, so all paths agree bit for bit. q and k
// are 16-byte aligned.
__device__ __forceinline__ float dist2_canonical(const float* __restrict__ q, const float* __restrict__ k, int dpad) {
  float total = 0.f;
  for (int c = 0; c < dpad; c += 32) {
    float p = 0.f;
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
      const float4 a = *reinterpret_cast<const float4*>(q + c + j);
      const float4 b = *reinterpret_cast<const float4*>(k + c + j);
      float e = __fsub_rn(a.x, b.x);
      p = __fmaf_rn(e, e, p);
      e = __fsub_rn(a.y, b.y);
      p = __fmaf_rn(e, e, p);
      e = __fsub_rn(a.z, b.z);
      p = __fmaf_rn(e, e, p);
      e = __fsub_rn(a.w, b.w);
      p = __fmaf_rn(e, e, p);
    }
    total = __fadd_rn(total, p);
  }
  return total;
}

// The same sequence with the query's d features as the caller passed them
// (the zero padding adds exact zeros: left out). vec: the row is 16-byte
// aligned and d a multiple of 4.
__device__ __forceinline__ float dist2_canonical_row(const float* __restrict__ q, bool vec, const float* __restrict__ k,
                                                     int d) {
  float total = 0.f;
  for (int c = 0; c < d; c += 32) {
    float p = 0.f;
    const int n = d - c < 32 ? d - c : 32;
    if (vec) {
#pragma unroll 8
      for (int j = 0; j < n; j += 4) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(q + c + j));
        const float4 b = *reinterpret_cast<const float4*>(k + c + j);
        float e = __fsub_rn(a.x, b.x);
        p = __fmaf_rn(e, e, p);
        e = __fsub_rn(a.y, b.y);
        p = __fmaf_rn(e, e, p);
        e = __fsub_rn(a.z, b.z);
        p = __fmaf_rn(e, e, p);
        e = __fsub_rn(a.w, b.w);
        p = __fmaf_rn(e, e, p);
      }
    } else {
#pragma unroll 8
      for (int j = 0; j < n; ++j) {
        const float e = __fsub_rn(__ldg(q + c + j), k[c + j]);
        p = __fmaf_rn(e, e, p);
      }
    }
    total = __fadd_rn(total, p);
  }
  return total;
}

// Operand kinds of the tensor screen. Both stream 128-byte rows (one swizzle
// row) per chunk and advance 32 bytes per MMA. kF16 reads the table's FP16
// copy: the same 11-bit significand as TF32, rounded to nearest instead of
// truncated, at half the bytes and twice the MMA rate.
constexpr int kTf32 = 0, kF16 = 1;
template <int KIND>
struct ScreenOp {
  static constexpr int kChunk = KIND == kF16 ? 64 : 32;  // features per chunk
  static constexpr int kStep = KIND == kF16 ? 16 : 8;    // features per MMA
  static __host__ __device__ constexpr uint32_t idesc(int M, int N) {
    return KIND == kF16 ? ptx::idesc_f16(M, N) : ptx::idesc_tf32(M, N);
  }
  static __device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if constexpr (KIND == kF16)
      ptx::mma_f16(d, a, b, idesc, acc);
    else
      ptx::mma_tf32(d, a, b, idesc, acc);
  }
  static __device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if constexpr (KIND == kF16)
      ptx::mma_f16_pair(d, a, b, idesc, acc);
    else
      ptx::mma_tf32_pair(d, a, b, idesc, acc);
  }
  // One chunk: four MMAs, or `steps` of them where only those hold features.
  template <bool PAIR = false>
  static __device__ __forceinline__ void chunk(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc,
                                               int steps) {
    auto one = [&](int u, uint32_t acc_u) {
      if constexpr (PAIR)
        mma_pair(d, a + 2 * u, b + 2 * u, idesc, acc_u);
      else
        mma(d, a + 2 * u, b + 2 * u, idesc, acc_u);
    };
    one(0, acc);
    if (KIND == kTf32 || steps == 4) {
      one(1, 1u);
      one(2, 1u);
      one(3, 1u);
    } else {
      if (steps > 1) one(1, 1u);
      if (steps > 2) one(2, 1u);
    }
  }
};

// The screen's comparison value of a pair (or, with the largest product and
// the smallest term, of a chunk): a - tau for TF32 operands; FP16 queries are
// scaled by a power of two, undone here (one rounding either way, monotone in
// a and in -tau).
template <int KIND>
__device__ __forceinline__ float screen_value(float a, float scale, float tau) {
  if constexpr (KIND == kF16)
    return __fmaf_rn(a, scale, -tau);
  else
    return __fsub_rn(a, tau);
}

}  // namespace lc
