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

// Where a probe's results go, and the counter of finished CTAs for the kernels
// that finalize themselves.
struct ProbeOut {
  unsigned long long* best;
  int64_t B;
  const int32_t* label;  // per entry
  int64_t* index;
  int32_t* out_label;  // nullable
  float* dist;         // nullable
  const int* abort;    // nullable: non-zero turns the batch into misses
  unsigned* done;      // zero at the launch and left so; null: k_finalize follows
};

// Unpack query q's word, and leave it empty for the next batch.
__device__ __forceinline__ void finalize_query(const ProbeOut& o, int64_t q, bool aborted) {
  unsigned long long v = __ldcg(o.best + q);
  o.best[q] = ~0ull;
  if (aborted) v = ~0ull;
  if (v == ~0ull) {
    o.index[q] = -1;
    if (o.out_label) o.out_label[q] = -1;
    if (o.dist) o.dist[q] = INFINITY;
  } else {
    const int64_t i = (int64_t)(v & 0xffffffffull);
    o.index[q] = i;
    if (o.out_label) o.out_label[q] = o.label[i];
    if (o.dist) o.dist[q] = sqrtf(__uint_as_float((unsigned)(v >> 32)));
  }
}

// Called by every thread of every CTA after the CTA's last update of `best`:
// the CTA that comes last finalizes the batch (a launch less than a kernel of
// its own; batches of at most kFusedQueries, which one CTA unpacks in ~2 us:
// with 4,000 queries it takes 6 and the call gets slower, 22.6 -> 24.6 us at
// d = 64 on 5,000 entries; no size in between was measured).
// `last_cta`: a word of shared memory.
constexpr int64_t kFusedQueries = 2048;
__device__ __forceinline__ void finalize_last_cta(const ProbeOut& o, unsigned n_ctas, volatile int* last_cta) {
  if (!o.done) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    *last_cta = atomicAdd(o.done, 1u) == n_ctas - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!*last_cta) return;
  __threadfence();
  const bool aborted = o.abort && __ldcg(o.abort) != 0;
  for (int64_t q = threadIdx.x; q < o.B; q += blockDim.x) finalize_query(o, q, aborted);
  if (threadIdx.x == 0) *o.done = 0u;
}

// Canonical FP32 squared distance sum_j (q_j - k_j)^2 over d_pad (multiple
// of 32) zero-padded features: a 32-wide fused-multiply-add chain per chunk,
// chunk sums added in order. Every probe path evaluates exactly this
// sequence of rounded operations, so all paths agree bit for bit.
//
// One 32-wide chunk of that sequence, features [c, c + n) of a query and a key;
// features past the query's d, zero in both rows, add exact zeros and are left
// out. vec: the query row is 16-byte aligned and n a multiple of 4 (key rows
// always are). All loads are issued before the chain starts.
__device__ __forceinline__ float dist2_chunk(const float* __restrict__ q, bool vec, const float* __restrict__ k, int n) {
  float4 a[8], b[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int m = n - 4 * u;
    a[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vec) {
      if (m > 0) a[u] = __ldg(reinterpret_cast<const float4*>(q) + u);
    } else {
      if (m > 0) a[u].x = __ldg(q + 4 * u);
      if (m > 1) a[u].y = __ldg(q + 4 * u + 1);
      if (m > 2) a[u].z = __ldg(q + 4 * u + 2);
      if (m > 3) a[u].w = __ldg(q + 4 * u + 3);
    }
    b[u] = m > 0 ? *(reinterpret_cast<const float4*>(k) + u) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float p = 0.f;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    float e = __fsub_rn(a[u].x, b[u].x);
    p = __fmaf_rn(e, e, p);
    e = __fsub_rn(a[u].y, b[u].y);
    p = __fmaf_rn(e, e, p);
    e = __fsub_rn(a[u].z, b[u].z);
    p = __fmaf_rn(e, e, p);
    e = __fsub_rn(a[u].w, b[u].w);
    p = __fmaf_rn(e, e, p);
  }
  return p;
}

// Recheck of screen candidates by a converged warp: bit j of a lane's `mask`
// is the pair (its query row, key key0 + j). A pair takes as many lanes as its
// rows have chunks (rounded up to a power of two), each running one chunk's
// chain, and the chunk sums are added in order, so the bits are those of
// the sequence above; with one lane per pair the loads and chains of all chunks
// came one after the other (3 us at d = 128), and the epilogue warp could not
// take its next tile meanwhile. Accepted pairs go to `best`.
struct Recheck {
  const float* q;  // query rows, qstride floats apart
  int64_t qstride;
  bool qvec;
  const float* keys;  // d_pad floats apart
  int dpad, d;
  const float* rr;
  unsigned long long* best;
};
// (Not inlined: its registers are not the epilogue loop's.)
static __device__ __noinline__ void recheck_warp(const Recheck& a, uint32_t mask, int64_t row, int64_t key0, int lane,
                                          unsigned long long& ncand) {
  const int nch = (a.d + 31) >> 5;
  const int lg = nch <= 1 ? 0 : 32 - __clz(nch - 1), sub = lane & ((1 << lg) - 1), grp = lane >> lg;
  for (;;) {
    uint32_t has = __ballot_sync(0xffffffffu, mask != 0);
    if (!has) break;
    const int64_t my_key = key0 + __ffs((int)mask) - 1;
    ncand += mask != 0 ? 1 : 0;
    mask &= mask - 1;
    while (has) {
      uint32_t b = has;
      for (int i = 0; i < grp; ++i) b &= b - 1;  // this group's pair: the grp-th lane that has one
      const int src = b ? __ffs((int)b) - 1 : 0;
      const int64_t key = __shfl_sync(0xffffffffu, my_key, src), r = __shfl_sync(0xffffffffu, row, src);
      float p = 0.f;
      const float thr = b ? __ldg(a.rr + key) : 0.f;  // (in flight with the rows)
      if (b && sub < nch) {
        const int n = a.d - 32 * sub;
        p = dist2_chunk(a.q + r * a.qstride + 32 * sub, a.qvec, a.keys + key * a.dpad + 32 * sub, n < 32 ? n : 32);
      }
      float total = __shfl_sync(0xffffffffu, p, grp << lg);
      for (int c = 1; c < nch; ++c) total = __fadd_rn(total, __shfl_sync(0xffffffffu, p, (grp << lg) + c));
      if (b && sub == 0 && total < thr) atomicMin(a.best + r, pack_hit(total, key));
      for (int i = 0; i < (32 >> lg); ++i) has &= has - 1;
    }
  }
}

// The screen constant of a row of a query tile: kappa, or a NaN for the rows from
// B on that fill the last tile up. An entry's screen term is -inf where its
// radius overflows (an empirical policy's, a head whose rows coincide or nearly
// vanish), which beats any constant that can be compared; every comparison with
// a NaN fails, so such a row passes neither the chunk test nor a pair's. The
// recheck reads the caller's own rows, which end with the last query, and the
// words of the rows past it stay empty. (Decided here by the launch's own B:
// scratch holds another batch's constants where calls overlap.)
__device__ __forceinline__ float row_kappa(const float* __restrict__ kappa, int64_t row, int64_t B) {
  return row < B ? __ldg(kappa + row) : __int_as_float(0x7fffffff);
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

// A chunk's 32 screen terms, loaded while the products leave tensor memory.
// tau: 16-byte aligned, in global memory (LDG) or shared memory.
struct ChunkTau {
  ulonglong2 t[8];
};
template <bool LDG>
__device__ __forceinline__ void load_chunk_tau(ChunkTau& c, const float* __restrict__ tau) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if constexpr (LDG)
      asm volatile("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(c.t[j].x), "=l"(c.t[j].y) : "l"(tau + 4 * j));
    else
      c.t[j] = *reinterpret_cast<const ulonglong2*>(tau + 4 * j);
  }
}

// Turns a row's 32 products into tau_j - value_j (value_j as screen_value's; a
// pair passes if that is <= -kappa, rounding to nearest being symmetric) and
// returns their minimum: two pairs per instruction, and no sign change of the
// terms.
template <int KIND>
__device__ __forceinline__ float screen_chunk(uint32_t (&v)[32], const ChunkTau& tau, float scale) {
  const uint64_t ns = ptx::pack_f32x2(__float_as_uint(-scale), __float_as_uint(-scale));
  float m = INFINITY;
#pragma unroll
  for (int j = 0; j < 32; j += 4) {
    const ulonglong2 tt = tau.t[j / 4];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint64_t a = ptx::pack_f32x2(v[j + 2 * u], v[j + 2 * u + 1]), tu = u ? tt.y : tt.x;
      const uint64_t x = KIND == kF16 ? ptx::fma_f32x2(a, ns, tu) : ptx::sub_f32x2(tu, a);
      v[j + 2 * u] = (uint32_t)x;
      v[j + 2 * u + 1] = (uint32_t)(x >> 32);
      m = fminf(m, fminf(__uint_as_float(v[j + 2 * u]), __uint_as_float(v[j + 2 * u + 1])));
    }
  }
  return m;
}

}  // namespace lc
