// The FP16 copy of the key table, which the tensor screen reads.
//
// A key's copy serves when its rounding error is that of normal FP16 numbers:
// ||k - k16|| <= 2^-11 (1 + 2^-7) ||k||, which holds unless features overflow FP16
// (65,504) or most of the row lies below its normal range (6e-5). Rows for
// which it does not hold (or whose norm is not a comfortable FP32 number) are
// counted as unfit; a table holding one is screened in TF32 from then on.
//
// With q scaled to [1, 2) by a power of two (its error at most (2^-11 + 2^-20) ||q||)
// the screen's product is within 2^-10 (1 + 2^-6) ||q|| ||k|| of q.k plus the
// FP32 accumulation: about half of what c_screen (2.0 * 2^-9 + ..., made for TF32)
// allows, so kappa and tau are shared by both operand types.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "internal.cuh"

namespace lc {

// Rounding error and size of the values one lane holds of a row.
struct Half16Check {
  float n2 = 0.f, e2 = 0.f;
  bool any = false;  // a non-zero value
  __device__ __forceinline__ void add(float x, float x16) {
    const float e = __fsub_rn(x, x16);  // exact while x16 is finite
    n2 = fmaf(x, x, n2);
    e2 = fmaf(e, e, e2);
    any |= x != 0.f;
  }
  // the test on these sums; NaN and infinite values fail it
  __device__ __forceinline__ bool fits() const {
    const float lim = 2.4214e-7f;  // 2^-22 (1 + 2^-7)^2, rounded down
    return e2 <= lim * n2 && n2 <= 1e30f && (n2 >= 1e-24f || !any);
  }
  // the test on the whole row, summed over the warp
  __device__ __forceinline__ bool row_fits() const {
    Half16Check s = *this;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.n2 += __shfl_xor_sync(0xffffffffu, s.n2, o);
      s.e2 += __shfl_xor_sync(0xffffffffu, s.e2, o);
    }
    s.any = __any_sync(0xffffffffu, any);
    return s.fits();
  }
};

// Whether four values pass that test by their largest alone (most do: the sums
// took 2 of the scatter's 15 us per 65,536 rows of 128 features). With m =
// max |x_i| <= 65,504 every error is at most 2^-11 |x_i| or, below the normal
// range, 2^-25: e2 <= 2^-22 n2 + 2^-48, and n2 >= m^2 >= 2^-20 makes the last
// term at most 2^-28 n2, within 2^-22 (1 + 2^-6) n2. Four zeros pass. NaN does not
// show in the maximum: a sum that is not finite fails.
__device__ __forceinline__ bool four_fit(const float4& v) {
  const float m = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
  const float s = (v.x + v.y) + (v.z + v.w);
  return s == s && m <= 65504.f && (m >= 9.765625e-4f || m == 0.f);
}

// One row of the copy by one warp, from a zero-padded FP32 source of n
// features (n <= d16; the rest is zero). Returns whether the copy serves.
__device__ __forceinline__ bool store_key16(const float* __restrict__ src, int n, __half* __restrict__ dst, int d16,
                                            int lane) {
  Half16Check chk;
  for (int j = lane; j < d16; j += 32) {
    const float x = j < n ? src[j] : 0.f;
    const __half h = __float2half_rn(x);
    dst[j] = h;
    chk.add(x, __half2float(h));
  }
  return chk.row_fits();
}

// The rows past the last entry of its 256-key tile, which the screen multiplies
// too, are kept zero by whatever appends entries: thread `tid` of `n` clears
// its share of [size, size rounded up to 256).
__device__ __forceinline__ void zero_tail(const Table& t, int dpad, int64_t size, int tid, int n) {
  const int64_t end = (size + 255) / 256 * 256;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  float4* k = reinterpret_cast<float4*>(t.keys + (size_t)size * dpad);
  for (int64_t e = tid; e < (end - size) * (dpad / 4); e += n) k[e] = z;
  if (t.keys16) {
    float4* h = reinterpret_cast<float4*>(t.keys16 + (size_t)size * t.d16);
    for (int64_t e = tid; e < (end - size) * (t.d16 / 8); e += n) h[e] = z;
  }
}

}  // namespace lc
