// Online certified lookup (Sec. 3.4, Algorithm 2; Eqs. 13-15).
//
//   H(q) = { i : ||q - z_i|| < r_i }          hit set, strict (Eq. 13)
//   i*   = argmin_{i in H(q)} ||q - z_i||     nearest hit, lowest index on ties (Eq. 14)
//   hit -> payload of i*, miss -> fall back to MainNet (Eq. 15)
//
// Acceptance. A pair (q, i) is accepted iff the canonical FP32 squared
// distance S~ (probe_common.cuh: direct differences, 32-wide FMA chunks added
// in order) is below rr_i = RZ(r_safe,i^2 (1 - eps_rc)). Since
// |S~ - S| <= gamma_{d_pad/32+33} S < eps_rc S, every accepted pair has an
// exact distance below r_safe,i <= r_i: the GPU never accepts a pair the
// exact rule rejects.
//
// Selection. Each accepted pair is reduced into a per-query 64-bit word
// (bits(S~) << 32 | i) with atomicMin. S~ >= 0, so its IEEE bits order like
// its value, and equal distances resolve to the lowest index.
//
// Kernels: k_prologue / k_prologue16 (pads or rounds the queries, per-query
// screen constant, clears the reduction words; not for the exact kernel), the
// main kernel (exact: every pair on CUDA cores; tensor: tcgen05 screen +
// recheck, probe_tc.cu and probe_pair.cu), which unpacks small batches itself,
// and else k_finalize. k_clear empties the words where nothing before did.
#include <algorithm>

#include "internal.cuh"
#include "probe_common.cuh"

namespace lc {
namespace {
// The kernel LIPCACHE_PROBE_AUTO picks: the tensor path where supported,
// except for batches so small (B N d_pad below 2^24 multiply-adds) that the
// exact kernel's smaller fixed cost wins (measured on GB300: 256 queries x
// 1,024 keys at d = 16 take 8.1 us exact against 11.7 us on tensor cores;
// 256 x 50,000 at d = 64 take 80 against 14 us). Both return the same bits.
int auto_path(const lipcache* h, int64_t B) {
  if (!tensor_path_supported(h->dpad) && !h->f16_screen()) return LIPCACHE_PROBE_EXACT;
  const double macs = (double)B * (double)h->size * (double)h->dpad;
  return macs < 16777216.0 ? LIPCACHE_PROBE_EXACT : LIPCACHE_PROBE_TENSOR;
}

constexpr unsigned kFull = 0xffffffffu;

__global__ void __launch_bounds__(256) k_prologue(const float* __restrict__ Q, int64_t B, int d, int dpad,
                                                  int64_t Bpad, float* __restrict__ qpad, float* __restrict__ kappa,
                                                  unsigned long long* __restrict__ best, double one_minus_c,
                                                  unsigned* __restrict__ done, DevStats* __restrict__ st) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  ptx::launch_dependents();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->abort_flag = 0;
    *done = 0u;
  }
  const int64_t row = (int64_t)blockIdx.x * 8 + warp;
  if (row >= Bpad) return;
  float part = 0.f;
  float* dst = qpad + (size_t)row * dpad;
  const float* src = Q + (size_t)row * d;
  for (int j = lane; j < dpad; j += 32) {
    const float x = (row < B && j < d) ? src[j] : 0.f;
    dst[j] = x;
    part = fmaf(x, x, part);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(kFull, part, o);
  if (lane == 0) {
    kappa[row] = __double2float_rd(one_minus_c * (double)part * 0.5);  // (not read from B on)
    best[row] = ~0ull;
  }
}

// Prologue of the FP16 screen: each query scaled by a power of two to a
// largest magnitude in [1, 2) and rounded to FP16 (its error then at most
// (2^-11 + 2^-20) ||q||, whatever the query's magnitude; NaN and infinities stay what
// they are), the scale that undoes it, the screen constant, and the reduction
// word. A warp per row, two features per lane and 64-feature chunk. The 1e-29
// taken off kappa covers queries below 2^-100, whose scaled features can
// underflow.
__global__ void __launch_bounds__(256) k_prologue16(const float* __restrict__ Q, int64_t B, int d, int d16,
                                                    int64_t Bpad, __half* __restrict__ q16, float* __restrict__ kappa,
                                                    float* __restrict__ qscale, unsigned long long* __restrict__ best,
                                                    double one_minus_c, unsigned* __restrict__ done,
                                                    DevStats* __restrict__ st) {
  constexpr int kMaxChunk = 8;  // d <= 512
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  ptx::launch_dependents();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->abort_flag = 0;
    *done = 0u;
  }
  const int64_t row = (int64_t)blockIdx.x * 8 + warp;
  if (row >= Bpad) return;
  const float* src = Q + (size_t)row * d;
  float x[kMaxChunk][2];
  float part = 0.f, m = 0.f;
#pragma unroll
  for (int i = 0; i < kMaxChunk; ++i)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = 64 * i + 2 * lane + u;
      x[i][u] = (row < B && j < d) ? __ldg(src + j) : 0.f;
      part = fmaf(x[i][u], x[i][u], part);
      m = fmaxf(m, fabsf(x[i][u]));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    part += __shfl_xor_sync(kFull, part, o);
    m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
  }
  int e = (int)((__float_as_uint(m) >> 23) & 0xffu) - 127;
  e = m == 0.f ? 0 : max(-100, min(126, e));
  const float down = __int_as_float((127 - e) << 23);
#pragma unroll
  for (int i = 0; i < kMaxChunk; ++i)
    if (64 * i < d16)
      *reinterpret_cast<__half2*>(q16 + (size_t)row * d16 + 64 * i + 2 * lane) =
          __floats2half2_rn(x[i][0] * down, x[i][1] * down);
  if (lane == 0) {
    kappa[row] = __fsub_rd(__double2float_rd(one_minus_c * (double)part * 0.5), 1e-29f);  // (not read from B on)
    qscale[row] = __int_as_float((127 + e) << 23);
    best[row] = ~0ull;
  }
}

// Exact probe: the canonical FP32 squared distance of every pair. It reads the
// caller's queries, needs no prologue (the reduction words are empty between
// probes) and, for small batches and grids, finalizes itself: one launch, so a
// single query costs one launch (1 x 2,000 at d = 64, called from Python: 20.9 us
// with three launches, 17.7 with one).
// CTA tile: 64 queries x 64 keys, 256 threads, 4 x 4 pairs per thread; the next
// 32-feature chunk is loaded while this one is computed; warps without a live
// query skip the product.
constexpr int kEQ = 64, kEK = 64, kES = kEQ + 4;

__global__ void __launch_bounds__(256) k_probe_exact(const float* __restrict__ Q, int64_t B, int d, int qvec,
                                                     const float* __restrict__ keys, const float* __restrict__ rr,
                                                     int64_t N, int dpad, unsigned long long* __restrict__ best,
                                                     ProbeOut out, DevStats* __restrict__ st) {
  __shared__ __align__(16) float qs[32][kES];
  __shared__ __align__(16) float ks[32][kES];
  const int tid = threadIdx.x;
  const int tq = tid >> 4, tk = tid & 15;
  const int64_t q0 = (int64_t)blockIdx.y * kEQ, k0 = (int64_t)blockIdx.x * kEK;
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) st->abort_flag = 0;
  const int lr = tid & 63, lp = tid >> 6;  // loader: row, 8-float part
  const bool busy = q0 + (tid >> 5) * 8 < B;  // this warp's eight queries hold a live one
  float tot[4][4], p[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) tot[a][b] = 0.f;
  float x[8], y[8];
  const int64_t qr = q0 + lr, kr = k0 + lr;
  auto load = [&](int c0) {
    const int c = c0 + lp * 8;
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = y[u] = 0.f;
    if (qr < B) {
      const float* src = Q + (size_t)qr * d + c;
      if (qvec) {
#pragma unroll
        for (int u = 0; u < 8; u += 4)
          if (c + u < d) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(src + u));
            x[u] = v.x, x[u + 1] = v.y, x[u + 2] = v.z, x[u + 3] = v.w;
          }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c + u < d) x[u] = __ldg(src + u);
      }
    }
    if (kr < N) {
      const float4* src = reinterpret_cast<const float4*>(keys + (size_t)kr * dpad + c);
      const float4 v = __ldg(src), w = __ldg(src + 1);
      y[0] = v.x, y[1] = v.y, y[2] = v.z, y[3] = v.w;
      y[4] = w.x, y[5] = w.y, y[6] = w.z, y[7] = w.w;
    }
  };
  load(0);
  for (int c0 = 0; c0 < dpad; c0 += 32) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      qs[lp * 8 + u][lr] = x[u];
      ks[lp * 8 + u][lr] = y[u];
    }
    __syncthreads();
    if (c0 + 32 < dpad) load(c0 + 32);
    if (busy) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) p[a][b] = 0.f;
#pragma unroll 8
      for (int j = 0; j < 32; ++j) {
        const float4 qv = *reinterpret_cast<const float4*>(&qs[j][tq * 4]);
        const float4 kv = *reinterpret_cast<const float4*>(&ks[j][tk * 4]);
        const float qa[4] = {qv.x, qv.y, qv.z, qv.w};
        const float kb[4] = {kv.x, kv.y, kv.z, kv.w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const float e = __fsub_rn(qa[a], kb[b]);
            p[a][b] = __fmaf_rn(e, e, p[a][b]);
          }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) tot[a][b] = __fadd_rn(tot[a][b], p[a][b]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int64_t key = k0 + tk * 4 + b;
    if (key >= N || !busy) continue;
    const float thr = rr[key];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int64_t row = q0 + tq * 4 + a;
      if (row < B && tot[a][b] < thr) atomicMin(best + row, pack_hit(tot[a][b], key));
    }
  }
  __shared__ int last_cta;
  finalize_last_cta(out, gridDim.x * gridDim.y, &last_cta);
}

__global__ void k_finalize(ProbeOut out) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < out.B) finalize_query(out, q, out.abort && *out.abort != 0);
}

// Empties the reduction words and clears the counter.
__global__ void k_clear(unsigned long long* __restrict__ best, int64_t B, unsigned* __restrict__ done) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < B) best[q] = ~0ull;
  if (q == 0) *done = 0u;
}

void clear_words(unsigned long long* best, int64_t n, unsigned* done, cudaStream_t s) {
  k_clear<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(best, n, done);
  LC_LAUNCH_CHECK("k_clear");
}

void ensure_probe_scratch(lipcache* h, int64_t Bpad) {
  if (Bpad <= h->q_cap) return;
  int64_t cap = h->q_cap ? h->q_cap : 1024;
  while (cap < Bpad) cap *= 2;
  h->q_cap = 0;
  carve_alloc(h->q_arena, [&](Carve& c) {
    c.take(h->qpad, (size_t)cap * h->dpad);
    c.take(h->kappa, (size_t)cap);
    c.take(h->qscale, (size_t)cap);
    c.take(h->best, (size_t)cap);
  });
  h->best_clean = false;  // (the next probe empties them, on its stream)
  h->q_cap = cap;
}

}  // namespace

bool tensor_path_supported(int dpad) { return dpad <= 256; }

void reserve_probe(lipcache* h, int64_t max_batch) {
  ensure_probe_scratch(h, (max_batch + 127) / 128 * 128);
}

// The small kernels around the tensor probe prefer the same shared-memory
// carveout as the probe itself, so that the SM does not switch its L1 /
// shared-memory split between the three launches of a probe.
void set_probe_carveout(lipcache* h) {
  if (h->probe_carveout_set) return;
  LC_CUDA(cudaFuncSetAttribute(k_prologue, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared));
  LC_CUDA(cudaFuncSetAttribute(k_prologue16, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared));
  LC_CUDA(cudaFuncSetAttribute(k_finalize, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared));
  h->probe_carveout_set = true;
}

namespace {
// The launch sequence of a probe on the given buffers. `clean`: every
// reduction word is empty and the counter is 0.
void probe_on(lipcache* h, int64_t B, const ProbeBuffers& b, bool clean, int64_t* out_index, int32_t* out_label,
              float* out_dist, bool timing, cudaStream_t s) {
  const int64_t Bpad = (B + 127) / 128 * 128;
  set_probe_carveout(h);
  int path = h->probe_path;
  if (path == LIPCACHE_PROBE_AUTO) path = auto_path(h, B);
  h->last_probe_path = path;
  const bool exact = path == LIPCACHE_PROBE_EXACT;
  const bool f16 = !exact && h->f16_screen();
  const int64_t ex = (h->size + kEK - 1) / kEK, ey = (B + kEQ - 1) / kEQ;  // the exact kernel's grid
  ProbeOut out{b.best, B, h->table.label, out_index, out_label, out_dist, &h->stats->abort_flag, nullptr};
  // the main kernel finalizes small batches itself (the exact one also only
  // where its CTAs, which count themselves, are few)
  if (h->size > 0 && B <= kFusedQueries && (!exact || ex * ey <= 4096)) out.done = b.done;
  if (exact || h->size == 0) {
    if (!clean) clear_words(b.best, B, b.done, s);
    if (h->size == 0) LC_CUDA(cudaMemsetAsync(&h->stats->abort_flag, 0, sizeof(int), s));
  } else {
    const unsigned pgrid = (unsigned)((Bpad + 7) / 8);
    if (f16) {
      k_prologue16<<<pgrid, 256, 0, s>>>(b.Q, B, h->d, h->table.d16, Bpad, static_cast<__half*>(b.q), b.kappa, b.scale,
                                         b.best, 1.0 - h->c_scr, b.done, h->stats);
      LC_LAUNCH_CHECK("k_prologue16");
    } else {
      k_prologue<<<pgrid, 256, 0, s>>>(b.Q, B, h->d, h->dpad, Bpad, static_cast<float*>(b.q), b.kappa, b.best,
                                       1.0 - h->c_scr, b.done, h->stats);
      LC_LAUNCH_CHECK("k_prologue");
    }
  }
  if (h->size > 0) {
    int slot = -1;
    if (timing && h->timing) {
      if (h->t_issued - h->t_harvested >= lipcache::kTimingRing) harvest_timing(h, false);
      slot = (int)(h->t_issued % lipcache::kTimingRing);
      h->t_kind[slot] = 0;
    }
    if (!exact) {
      // the start event is recorded by the launcher, after its host-side
      // preparation, right before the kernel
      h->launch_event = slot >= 0 ? h->tev0[slot] : nullptr;
      h->last_probe_path = launch_probe_tc(h, B, path, f16, b, out, s);
      h->launch_event = nullptr;
    } else {
      if (slot >= 0) LC_CUDA(cudaEventRecord(h->tev0[slot], s));
      h->last_grid = (int)(ex * ey);
      h->last_cluster = 1;
      const int qvec = h->d % 4 == 0 && ((uintptr_t)b.Q & 15) == 0;
      // (a grid has at most 65,535 rows of CTAs: batches above 4,194,240 take two
      // launches; they are not finalized by the kernel)
      constexpr int64_t kMaxRows = 65535;
      for (int64_t y0 = 0; y0 < ey; y0 += kMaxRows) {
        const int64_t q0 = y0 * kEQ, n = std::min(B - q0, kMaxRows * kEQ);
        const dim3 grid((unsigned)ex, (unsigned)((n + kEQ - 1) / kEQ));
        k_probe_exact<<<grid, 256, 0, s>>>(b.Q + (size_t)q0 * h->d, n, h->d, qvec, h->table.keys, h->probe_rr(),
                                           h->size, h->dpad, b.best + q0, out, h->stats);
        LC_LAUNCH_CHECK("k_probe_exact");
      }
    }
    if (slot >= 0) {
      LC_CUDA(cudaEventRecord(h->tev1[slot], s));
      ++h->t_issued;
    }
  }
  if (!out.done) {
    k_finalize<<<(unsigned)((B + 255) / 256), 256, 0, s>>>(out);
    LC_LAUNCH_CHECK("k_finalize");
  }
}
}  // namespace

void probe(lipcache* h, const float* Q, int64_t B, int64_t* out_index, int32_t* out_label, float* out_dist,
           cudaStream_t s) {
  ensure_probe_scratch(h, (B + 127) / 128 * 128);
  // A captured probe runs whenever its graph is replayed, so it assumes nothing
  // of the words and the counter. (A stream that cannot be asked: as captured.)
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
    cudaGetLastError();
    cap = cudaStreamCaptureStatusActive;
  }
  ProbeBuffers b{Q, h->qpad, h->kappa, h->qscale, h->best, h->done + lipcache::kDoneSlots};
  if (cap != cudaStreamCaptureStatusNone) {
    probe_on(h, B, b, false, out_index, out_label, out_dist, true, s);
    return;
  }
  b.done = h->done + h->done_next++ % lipcache::kDoneSlots;
  if (!h->best_clean) clear_words(h->best, h->q_cap, b.done, s);
  // (the finalizing kernel empties the words it reads; a call that throws on
  // the way leaves them in doubt)
  h->best_clean = false;
  probe_on(h, B, b, true, out_index, out_label, out_dist, true, s);
  h->best_clean = true;
}

// The same launch sequence as probe(), on scratch memory the caller
// provides (qpad: Bpad x d_pad floats, kappa and qscale: Bpad floats, best:
// Bpad words, Bpad = B rounded up to 128; done: one word; the FP16 form of the
// queries, d16 <= 2 d_pad halves per row, takes qpad's place). Allocates nothing.
void probe_external_scratch(lipcache* h, const float* Q, int64_t B, int64_t* out_index, int32_t* out_label,
                            float* out_dist, float* qpad, float* kappa, float* qscale, unsigned long long* best,
                            unsigned* done, cudaStream_t s) {
  probe_on(h, B, ProbeBuffers{Q, qpad, kappa, qscale, best, done}, false, out_index, out_label, out_dist, false, s);
}

}  // namespace lc
