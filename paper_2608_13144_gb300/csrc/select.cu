// Selection strategies S of Algorithm 1 (Sec. 5.5): radius-prioritised
// de-duplication (the paper's default) and K-center per class (at the end
// of the file).
//
// The candidates that Algorithm 1 accepts are visited in order of decreasing
// certified radius (the FP32 radius, ties to the lower row). A candidate is
// kept unless the lookup of Eq. 13 would already hit it -- it lies strictly
// inside the ball of an entry in the cache, whether there before the call or
// kept earlier in it -- or its class (payload label in [0, C)) or the call
// has used its budget. Kept entries are appended in visiting order.
//
// GPU schedule. The order is a bitonic sort of 64-bit keys (radius bits
// descending, row ascending). Candidates are then processed in chunks of up to
// kSelChunk in that order, leaving out those whose class has used its budget
// before the chunk (they cannot be kept): the chunk is probed against the cache
// as it stands (a hit = covered by an earlier entry), its pairwise coverage by
// earlier members of the same chunk is computed as a bit matrix (canonical FP32
// distance against the member's acceptance threshold rr, the probe's test),
// one block resolves the chunk 32 members at a time, and the kept members are
// appended. Coverage uses the probe's conservative thresholds, so a skipped
// candidate is always exactly covered; pairs within ~2e-6 relative of a
// radius may be judged "not covered" where exact arithmetic says "covered".
#include "internal.cuh"
#include "key16.cuh"
#include "probe_common.cuh"

namespace lc {
namespace {

constexpr int kSelChunk = 4096;
constexpr int kSelWords = kSelChunk / 32;

// Sort key: radius descending, row ascending; rejected rows last.
__global__ void k_sel_keys(const uint8_t* __restrict__ accept, const float* __restrict__ radius, int64_t n,
                           int64_t npow, unsigned long long* __restrict__ keys, int64_t* __restrict__ n_acc) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npow) return;
  unsigned long long k = ~0ull;
  bool acc = false;
  if (i < n && accept[i]) {
    acc = true;
    k = ((unsigned long long)(0xFFFFFFFFu - __float_as_uint(radius[i])) << 32) | (unsigned long long)(uint32_t)i;
  }
  keys[i] = k;
  const unsigned m = __ballot_sync(0xffffffffu, acc);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(reinterpret_cast<unsigned long long*>(n_acc), (unsigned long long)__popc(m));
}

// Bitonic sort (ascending) of npow keys, a power of two. Spans of up to
// kSortSpan keys are sorted, and the short-distance passes of longer merges
// done, in shared memory: 65,536 keys take 15 launches instead of 136.
constexpr int kSortSpan = 4096, kSortThreads = 1024;

__device__ __forceinline__ void order_pair(unsigned long long& x, unsigned long long& y, bool up) {
  if ((x > y) == up) {
    const unsigned long long z = x;
    x = y;
    y = z;
  }
}

// kmin == 2: sort every span; kmin = kmax > span: the passes j < span of the
// merge k = kmax.
__global__ void __launch_bounds__(kSortThreads) k_bitonic_span(unsigned long long* __restrict__ a, int span,
                                                               int64_t kmin, int64_t kmax) {
  __shared__ unsigned long long s[kSortSpan];
  const int64_t base = (int64_t)blockIdx.x * span;
  for (int i = threadIdx.x; i < span; i += kSortThreads) s[i] = a[base + i];
  __syncthreads();
  for (int64_t k = kmin; k <= kmax; k <<= 1)
    for (int j = (int)((k < span ? k : span) >> 1); j > 0; j >>= 1) {
      for (int p = threadIdx.x; p < span / 2; p += kSortThreads) {
        const int i = 2 * p - (p & (j - 1));  // the p-th index with bit j clear
        order_pair(s[i], s[i + j], ((base + i) & k) == 0);
      }
      __syncthreads();
    }
  for (int i = threadIdx.x; i < span; i += kSortThreads) a[base + i] = s[i];
}

// One pass (distance j >= kSortSpan) of the merge k.
__global__ void __launch_bounds__(256) k_bitonic(unsigned long long* __restrict__ a, int64_t npow, int64_t j, int64_t k) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npow / 2) return;
  const int64_t i = 2 * p - (p & (j - 1));
  unsigned long long x = a[i], y = a[i + j];
  if ((x > y) == ((i & k) == 0)) {
    a[i] = y;
    a[i + j] = x;
  }
}

void sort_keys(unsigned long long* a, int64_t npow, cudaStream_t s) {
  const int span = npow < kSortSpan ? (int)npow : kSortSpan;
  if (span < 2) return;
  const unsigned blocks = (unsigned)(npow / span);
  k_bitonic_span<<<blocks, kSortThreads, 0, s>>>(a, span, 2, span);
  LC_LAUNCH_CHECK("k_bitonic_span");
  for (int64_t k = 2 * (int64_t)span; k <= npow; k <<= 1) {
    for (int64_t j = k >> 1; j >= span; j >>= 1) {
      k_bitonic<<<(unsigned)((npow / 2 + 255) / 256), 256, 0, s>>>(a, npow, j, k);
      LC_LAUNCH_CHECK("k_bitonic");
    }
    k_bitonic_span<<<blocks, kSortThreads, 0, s>>>(a, span, k, k);
    LC_LAUNCH_CHECK("k_bitonic_span");
  }
}

// Device counters of a selection.
struct SelState {
  long long n_acc;   // certified candidates
  long long kept;    // kept by this call
  long long cursor;  // first candidate, in visiting order, not yet in a chunk
  int n_list;        // kept members of the current chunk
  int kc;            // members of the next chunk
};
static_assert(sizeof(SelState) <= 64, "fits the host block's tail");

// The next chunk: the first kSelChunk candidates from the cursor on whose class
// still has budget, in order (one block; four candidates per thread a round).
__global__ void __launch_bounds__(1024) k_sel_pick(const unsigned long long* __restrict__ keys,
                                                   const int32_t* __restrict__ label,
                                                   const int32_t* __restrict__ class_cnt, int C, int budget_pc,
                                                   int32_t* __restrict__ rows, SelState* __restrict__ st) {
  __shared__ int wsum[32];
  __shared__ long long first_left;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long n = st->n_acc;
  long long c = st->cursor;
  int got = 0;
  if (tid == 0) first_left = n;
  while (c < n && got < kSelChunk) {
    const long long c4 = c + 4 * (long long)tid;
    int32_t row[4];
    bool open[4];
    int mine = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      row[u] = c4 + u < n ? (int32_t)(keys[c4 + u] & 0xFFFFFFFFull) : -1;
      open[u] = row[u] >= 0;
      if (open[u] && budget_pc > 0) {
        const int32_t lab = label[row[u]];
        open[u] = !(lab >= 0 && lab < C && class_cnt[lab] >= budget_pc);
      }
      mine += open[u] ? 1 : 0;
    }
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      int x = wsum[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      wsum[lane] = x;
    }
    __syncthreads();
    int at = got + (warp ? wsum[warp - 1] : 0) + incl - mine;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (!open[u]) continue;
      if (at < kSelChunk)
        rows[at] = row[u];
      else if (at == kSelChunk)
        first_left = c4 + u;
      ++at;
    }
    got += wsum[31];
    c += 4 * 1024;
    __syncthreads();
  }
  if (tid == 0) {
    st->kc = got < kSelChunk ? got : kSelChunk;
    st->cursor = got > kSelChunk ? first_left : (c < n ? c : n);
  }
}

// The chunk members' features (kc x d).
__global__ void k_sel_gather(const int32_t* __restrict__ rows, int kc, const float* __restrict__ H, int d,
                             float* __restrict__ G) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p = blockIdx.x * 8 + warp;
  if (p >= kc) return;
  const int64_t row = rows[p];
  for (int j = lane; j < d; j += 32) G[(size_t)p * d + j] = H[(size_t)row * d + j];
}

// Coverage inside the chunk: bit i of cov[j * kSelWords + i / 32] is set iff
// i < j and member j lies inside member i's ball (canonical FP32 squared
// distance below rr of member i). Block (ti, tj), ti <= tj, computes the 64 x 64
// tile of members i in tile ti, j in tile tj, 4 x 4 pairs per thread (the
// layout of the exact probe: an eighth of the shared-memory reads per pair of
// one pair per thread; bound by the FP32 pipe); the d features stream through
// shared memory in 32-float chunks, which is the canonical summation order.
constexpr int kCovT = 64, kCovS = kCovT + 4;

__global__ void __launch_bounds__(256) k_sel_cover(const float* __restrict__ G, int d, int kc,
                                                   const int32_t* __restrict__ rows, const float* __restrict__ rr,
                                                   uint32_t* __restrict__ cov) {
  const int ti = blockIdx.x, tj = blockIdx.y;
  if (ti > tj) return;
  __shared__ __align__(16) float zi[32][kCovS], zj[32][kCovS];
  const int tid = threadIdx.x;
  const int ci = tid & 15, cj = tid >> 4;  // members i: 4 ci .., j: 4 cj ..
  const int lr = tid >> 2, lf = (tid & 3) * 8;  // loader: row, first of 8 features
  float tot[4][4], p[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) tot[x][y] = 0.f;
  for (int c = 0; c < d; c += 32) {
    {
      const int gi = ti * kCovT + lr, gj = tj * kCovT + lr;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int f = c + lf + u;
        zi[lf + u][lr] = (gi < kc && f < d) ? G[(size_t)gi * d + f] : 0.f;
        zj[lf + u][lr] = (gj < kc && f < d) ? G[(size_t)gj * d + f] : 0.f;
      }
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) p[x][y] = 0.f;
#pragma unroll 8
    for (int f = 0; f < 32; ++f) {
      const float4 a4 = *reinterpret_cast<const float4*>(&zi[f][4 * ci]);
      const float4 b4 = *reinterpret_cast<const float4*>(&zj[f][4 * cj]);
      const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const float e = __fsub_rn(bv[y], av[x]);
          p[x][y] = __fmaf_rn(e, e, p[x][y]);
        }
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) tot[x][y] = __fadd_rn(tot[x][y], p[x][y]);
    __syncthreads();
  }
  float thr[4];
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const int i = ti * kCovT + 4 * ci + x;
    thr[x] = i < kc ? rr[rows[i]] : 0.f;
  }
  // the 16 threads of a half-warp hold the 64 bits of four rows j
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    const int j = tj * kCovT + 4 * cj + y;
    uint32_t w = 0;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int i = ti * kCovT + 4 * ci + x;
      w |= (uint32_t)(i < kc && j < kc && i < j && tot[x][y] < thr[x]) << (4 * (ci & 7) + x);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, o);
    if ((ci & 7) == 0 && j < kc) cov[(size_t)j * kSelWords + 2 * ti + (ci >> 3)] = w;
  }
}

struct ResolveArgs {
  const uint32_t* cov;
  const int32_t* rows;
  const int64_t* hit;      // per member: cache index it hits, -1 if none
  const int32_t* label;    // per row (certify scratch)
  int32_t* class_cnt;      // per class, kept in this call
  SelState* st;
  int32_t* list;           // kept members in order
  const DevStats* stats;   // abort_flag set: the chunk's probe gave up, `hit` says nothing
  int kc, C, budget_pc;
  long long budget_total;
};

// The greedy pass over a chunk: member j is kept iff it hits nothing in the
// cache, no kept member i < j of the chunk covers it and its budgets allow. One
// block takes 32 members at a time: warp m tests member m of the group against
// the members kept in earlier groups (its coverage row, read one group ahead,
// against the kept-set words in shared memory); warp 0 then settles the group
// in batches: the undecided members before the first one that another
// undecided member covers are independent, so each is kept unless its class or
// the call runs out of budget before it (ranks by ballot); what they cover
// drops out. A chunk whose probe gave up keeps nothing. Labels, hits and class counts are in shared memory. Bound by the
// chain of groups, ~1,200 cycles each on a pool where a third of the members
// are near-duplicates; one warp walking the members took 160 ns for each
// (4,096 members: 80 us, before 665 us).
__global__ void __launch_bounds__(1024) k_sel_resolve(ResolveArgs a) {
  constexpr int kPer = kSelWords / 32;
  __shared__ uint32_t sel[kSelWords];
  __shared__ uint32_t intra[2][32];
  __shared__ uint8_t open_s[2][32];
  __shared__ uint8_t free_s[kSelChunk];
  __shared__ int16_t lab_s[kSelChunk];  // class with a budget, or -1
  __shared__ int32_t cnt_s[LIPCACHE_MAX_CLASSES];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int groups = (a.kc + 31) / 32;
  const bool aborted = a.stats->abort_flag != 0;
  auto load_row = [&](int g, uint32_t (&w)[kPer]) {
    const int j = 32 * g + warp;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int wi = lane + 32 * t;
      w[t] = (j < a.kc && wi <= g) ? __ldcg(a.cov + (size_t)j * kSelWords + wi) : 0u;
    }
  };
  uint32_t cur[kPer], nxt[kPer];
  load_row(0, cur);
  for (int w = tid; w < kSelWords; w += 1024) sel[w] = 0u;
  for (int c = tid; c < a.C; c += 1024) cnt_s[c] = a.class_cnt[c];
  for (int j = tid; j < kSelChunk; j += 1024) {
    const bool in = j < a.kc;
    const int32_t lab = in ? a.label[a.rows[j]] : -1;
    free_s[j] = in && a.hit[j] < 0 && !aborted ? 1 : 0;
    lab_s[j] = (int16_t)(a.budget_pc > 0 && lab >= 0 && lab < a.C ? lab : -1);
  }
  int nk = 0;
  long long tot = a.st->kept;
  __syncthreads();
  for (int g = 0; g < groups; ++g) {
    if (g + 1 < groups) load_row(g + 1, nxt);
    bool any = false;
    uint32_t own = 0;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int wi = lane + 32 * t;
      if (wi < g) any = any || (cur[t] & sel[wi]) != 0u;
      if (wi == g) own = cur[t];
    }
    any = __any_sync(0xffffffffu, any);
    if (lane == (g & 31)) {
      intra[g & 1][warp] = own;
      open_s[g & 1][warp] = any ? 0 : free_s[32 * g + warp];
    }
    __syncthreads();
    if (warp == 0) {
      const int jl = 32 * g + lane;
      const uint32_t in = intra[g & 1][lane];
      const uint32_t lt = (1u << lane) - 1u;
      uint32_t und = __ballot_sync(0xffffffffu, open_s[g & 1][lane] != 0);  // undecided
      const int lab = lab_s[jl];
      const uint32_t peers = __match_any_sync(0xffffffffu, lab >= 0 ? lab : -1 - lane);
      const int have = lab >= 0 ? cnt_s[lab] : 0;
      uint32_t taken = 0;
      while (und) {
        const uint32_t conf = __ballot_sync(0xffffffffu, ((und >> lane) & 1u) && (in & und) != 0u);
        const uint32_t batch = conf ? und & ((conf & (0u - conf)) - 1u) : und;
        const bool fits = ((batch >> lane) & 1u) &&
                          (lab < 0 || have + __popc(peers & (taken | (batch & lt))) < a.budget_pc);
        const uint32_t f = __ballot_sync(0xffffffffu, fits);
        const uint32_t now = __ballot_sync(
            0xffffffffu, fits && (a.budget_total <= 0 || tot + __popc(taken) + __popc(f & lt) < a.budget_total));
        taken |= now;
        und &= ~batch & ~__ballot_sync(0xffffffffu, (in & now) != 0u);
      }
      if ((taken >> lane) & 1u) {
        a.list[nk + __popc(taken & lt)] = jl;
        if (lab >= 0 && (peers & taken & lt) == 0u) cnt_s[lab] = have + __popc(peers & taken);
      }
      nk += __popc(taken);
      tot += __popc(taken);
      if (lane == 0) sel[g] = taken;
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kPer; ++t) cur[t] = nxt[t];
  }
  for (int c = tid; c < a.C; c += 1024) a.class_cnt[c] = cnt_s[c];
  if (tid == 0) {
    a.st->n_list = nk;
    a.st->kept = tot;
  }
}

constexpr int kTailBlocks = 8;  // blocks of a scatter that clear the rows past the new end

struct SelScatterArgs {
  const int32_t* list;
  const SelState* st;
  const int32_t* rows;
  const float* G;
  int d, dpad;
  int64_t size0;
  const float* rr;
  const float* tau;
  const float* kn;
  const float* radius;
  const int32_t* label;
  const int32_t* yG;
  Table t;
  int64_t* out_index;
  int64_t* unfit;
};

// Append the kept members in order; one warp per member.
__global__ void k_sel_scatter(SelScatterArgs a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (blockIdx.x < kTailBlocks) {
    zero_tail(a.t, a.dpad, a.size0 + a.st->n_list, (int)(blockIdx.x * 256 + threadIdx.x), kTailBlocks * 256);
    return;
  }
  const int q = (blockIdx.x - kTailBlocks) * 8 + warp;
  if (q >= a.st->n_list) return;
  const int p = a.list[q];
  const int32_t row = a.rows[p];
  const int64_t dst = a.size0 + q;
  float* kd = a.t.keys + (size_t)dst * a.dpad;
  for (int j = lane; j < a.dpad; j += 32) kd[j] = j < a.d ? a.G[(size_t)p * a.d + j] : 0.f;
  if (a.t.keys16 && !store_key16(a.G + (size_t)p * a.d, a.d, a.t.keys16 + (size_t)dst * a.t.d16, a.t.d16, lane) &&
      lane == 0)
    atomicAdd(reinterpret_cast<unsigned long long*>(a.unfit), 1ull);
  if (lane == 0) {
    a.t.rr[dst] = a.rr[row];
    a.t.tau[dst] = a.tau[row];
    a.t.kn[dst] = a.kn[row];
    a.t.radius[dst] = a.radius[row];
    a.t.label[dst] = a.label[row];
    a.t.yG[dst] = a.yG[row];
    if (a.out_index) a.out_index[row] = dst;
  }
}

__global__ void k_fill_i64(int64_t* __restrict__ p, int64_t n, int64_t v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}
__global__ void k_copy_f32(const float* __restrict__ s, float* __restrict__ d, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = s[i];
}

// ---------------------------------------------------------------- K-center
// Per class (payload label in [0, C)) among the certified candidates:
// Gonzalez's farthest-point greedy, first centre the largest radius, ties to
// the lower row, at most budget_per_class centres. The candidates are sorted
// by (label, row); one block per class walks its segment once per centre
// (cost: centres x class size x d). Distances are the canonical FP32 squared
// distance, so near-ties (~1e-6 relative) may resolve differently from an
// FP64 evaluation.
// Sort key of the per-class K-center: label, then row; others last.
__global__ void k_kc_keys(const uint8_t* __restrict__ accept, const int32_t* __restrict__ label, int64_t n,
                          int64_t npow, int C, unsigned long long* __restrict__ keys, int64_t* __restrict__ n_acc) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npow) return;
  unsigned long long k = ~0ull;
  bool in = false;
  if (i < n && accept[i] && label[i] >= 0 && label[i] < C) {
    in = true;
    k = ((unsigned long long)(uint32_t)label[i] << 32) | (unsigned long long)(uint32_t)i;
  }
  keys[i] = k;
  const unsigned m = __ballot_sync(0xffffffffu, in);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(reinterpret_cast<unsigned long long*>(n_acc), (unsigned long long)__popc(m));
}

// Class segments [seg[2c], seg[2c+1]) of the sorted keys (zero-initialised).
__global__ void k_kc_segments(const unsigned long long* __restrict__ keys, int64_t n_acc, int32_t* __restrict__ seg) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_acc) return;
  const uint32_t c = (uint32_t)(keys[p] >> 32);
  if (p == 0 || (uint32_t)(keys[p - 1] >> 32) != c) seg[2 * c] = (int32_t)p;
  if (p == n_acc - 1 || (uint32_t)(keys[p + 1] >> 32) != c) seg[2 * c + 1] = (int32_t)(p + 1);
}

constexpr int kKcThreads = 256;

__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long v, unsigned long long* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  unsigned long long m = red[0];
  for (int w = 1; w < kKcThreads / 32; ++w) m = red[w] > m ? red[w] : m;
  return m;
}

// Gonzalez's farthest-point greedy for one class per block: first the
// candidate of largest radius, then repeatedly the one farthest (canonical
// FP32 squared distance) from the centres so far; ties to the lower row.
// mind[p] holds each segment member's squared distance to the nearest centre
// (negative once chosen); the chosen rows go to out[s0 ..] in order.
__global__ void __launch_bounds__(kKcThreads) k_kcenter(const unsigned long long* __restrict__ keys,
                                                        const int32_t* __restrict__ seg, const float* __restrict__ H,
                                                        int d, const float* __restrict__ radius, int budget,
                                                        float* __restrict__ mind, int32_t* __restrict__ out,
                                                        int32_t* __restrict__ cnt) {
  extern __shared__ float zc[];  // the newest centre's features (d)
  __shared__ unsigned long long red[kKcThreads / 32];
  const int c = blockIdx.x, tid = threadIdx.x;
  const int s0 = seg[2 * c], s1 = seg[2 * c + 1];
  const int nc = s1 - s0;
  if (nc <= 0) {
    if (tid == 0) cnt[c] = 0;
    return;
  }
  unsigned long long best = 0ull;
  for (int p = s0 + tid; p < s1; p += kKcThreads) {
    const uint32_t row = (uint32_t)(keys[p] & 0xFFFFFFFFull);
    const unsigned long long k = ((unsigned long long)__float_as_uint(radius[row]) << 32) | (0xFFFFFFFFu - row);
    best = k > best ? k : best;
    mind[p] = INFINITY;
  }
  best = block_max_u64(best, red);
  const int want = budget < nc ? budget : nc;
  for (int t = 0; t < want; ++t) {
    const uint32_t row = 0xFFFFFFFFu - (uint32_t)(best & 0xFFFFFFFFull);
    if (tid == 0) out[s0 + t] = (int32_t)row;
    for (int j = tid; j < d; j += kKcThreads) zc[j] = H[(size_t)row * d + j];
    __syncthreads();
    if (t + 1 == want) break;
    best = 0ull;
    for (int p = s0 + tid; p < s1; p += kKcThreads) {
      const uint32_t r = (uint32_t)(keys[p] & 0xFFFFFFFFull);
      float m = mind[p];
      if (r == row) m = -1.f;  // chosen
      if (m >= 0.f) {
        const float* z = H + (size_t)r * d;
        float total = 0.f;
        for (int c0 = 0; c0 < d; c0 += 32) {
          float q = 0.f;
          const int ce = c0 + 32 < d ? c0 + 32 : d;
          for (int j = c0; j < ce; ++j) {
            const float e = __fsub_rn(z[j], zc[j]);
            q = __fmaf_rn(e, e, q);
          }
          total = __fadd_rn(total, q);
        }
        m = fminf(m, total);
        const unsigned long long k = ((unsigned long long)__float_as_uint(m) << 32) | (0xFFFFFFFFu - r);
        best = k > best ? k : best;
      }
      mind[p] = m;
    }
    best = block_max_u64(best, red);
  }
  if (tid == 0) cnt[c] = want;
}

// Append the centres class by class (offsets = exclusive scan of cnt).
__global__ void k_kc_scatter(const int32_t* __restrict__ seg, const int32_t* __restrict__ cnt,
                             const int32_t* __restrict__ off, const int32_t* __restrict__ out, const float* __restrict__ H,
                             int d, int dpad, int64_t size0, const float* __restrict__ rr, const float* __restrict__ tau,
                             const float* __restrict__ kn, const float* __restrict__ radius,
                             const int32_t* __restrict__ label, const int32_t* __restrict__ yG, Table t,
                             int64_t* __restrict__ out_index, int64_t* __restrict__ unfit,
                             const int64_t* __restrict__ total, int C) {
  const int c = blockIdx.y;
  if (c == C) {  // one more row of blocks clears the rows past the new end
    zero_tail(t, dpad, size0 + *total, (int)(blockIdx.x * 256 + threadIdx.x), (int)gridDim.x * 256);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = blockIdx.x * 8 + warp; q < cnt[c]; q += gridDim.x * 8) {
    const int32_t row = out[seg[2 * c] + q];
    const int64_t dst = size0 + off[c] + q;
    float* kd = t.keys + (size_t)dst * dpad;
    for (int j = lane; j < dpad; j += 32) kd[j] = j < d ? H[(size_t)row * d + j] : 0.f;
    if (t.keys16 && !store_key16(H + (size_t)row * d, d, t.keys16 + (size_t)dst * t.d16, t.d16, lane) && lane == 0)
      atomicAdd(reinterpret_cast<unsigned long long*>(unfit), 1ull);
    if (lane == 0) {
      t.rr[dst] = rr[row];
      t.tau[dst] = tau[row];
      t.kn[dst] = kn[row];
      t.radius[dst] = radius[row];
      t.label[dst] = label[row];
      t.yG[dst] = yG[row];
      if (out_index) out_index[row] = dst;
    }
  }
}

// Exclusive scan of C counts (C <= 1024), total in *total.
__global__ void __launch_bounds__(1024) k_kc_scan(const int32_t* __restrict__ cnt, int C, int32_t* __restrict__ off,
                                                  int64_t* __restrict__ total) {
  __shared__ int32_t buf[1024];
  const int t = threadIdx.x;
  const int v = t < C ? cnt[t] : 0;
  buf[t] = v;
  __syncthreads();
  for (int s = 1; s < 1024; s <<= 1) {
    const int x = t >= s ? buf[t - s] : 0;
    __syncthreads();
    buf[t] += x;
    __syncthreads();
  }
  if (t < C) off[t] = buf[t] - v;
  if (t == 1023) *total = buf[1023];
}

template <typename T>
void grow_to(T*& p, int64_t& cap, int64_t n) {
  if (n <= cap) return;
  if (p) cudaFree(p);
  p = nullptr;
  cap = 0;
  LC_CUDA(cudaMalloc(&p, sizeof(T) * (size_t)n));
  cap = n;
}

// The scratch of a chunk and the counters.
void ensure_chunk_scratch(lipcache* h) {
  SelectScratch& x = h->sel;
  if (x.chunk) return;
  carve_alloc(x.chunk, [&](Carve& c) {
    c.take(x.G, (size_t)kSelChunk * h->d);
    c.take(x.rows, kSelChunk);
    c.take(x.hit, kSelChunk);
    c.take(x.cov, (size_t)kSelChunk * kSelWords);
    c.take(x.list, kSelChunk);
    c.take(x.class_cnt, (size_t)h->C);
    c.take(x.state, 64);
  });
}

}  // namespace

int64_t select_insert(lipcache* h, const float* H, int64_t n, const int32_t* payload, int require_consistency,
                      int64_t budget_total, int budget_per_class, int64_t* out_index, float* out_radius,
                      cudaStream_t s) {
  SelectScratch& x = h->sel;
  certify_rows(h, H, n, payload, require_consistency, s);
  require_certify_ok(h, s);
  const unsigned nb = (unsigned)((n + 255) / 256);
  if (out_index) {
    k_fill_i64<<<nb, 256, 0, s>>>(out_index, n, -1);
    LC_LAUNCH_CHECK("k_fill_i64");
  }
  if (out_radius) {
    k_copy_f32<<<nb, 256, 0, s>>>(h->ins_radius, out_radius, n);
    LC_LAUNCH_CHECK("k_copy_f32");
  }
  // visiting order
  int64_t npow = 1;
  while (npow < n) npow <<= 1;
  grow_to(x.keys, x.keys_cap, npow);
  ensure_chunk_scratch(h);
  SelState* st = reinterpret_cast<SelState*>(x.state);
  SelState* hs = reinterpret_cast<SelState*>(h->sel_host);
  LC_CUDA(cudaMemsetAsync(st, 0, sizeof(SelState), s));
  LC_CUDA(cudaMemsetAsync(x.class_cnt, 0, sizeof(int32_t) * h->C, s));
  const unsigned npb = (unsigned)((npow + 255) / 256);
  k_sel_keys<<<npb, 256, 0, s>>>(h->ins_accept, h->ins_radius, n, npow, x.keys,
                                 reinterpret_cast<int64_t*>(&st->n_acc));
  LC_LAUNCH_CHECK("k_sel_keys");
  sort_keys(x.keys, npow, s);
  auto pick = [&]() {
    k_sel_pick<<<1, 1024, 0, s>>>(x.keys, h->ins_label, x.class_cnt, h->C, budget_per_class, x.rows, st);
    LC_LAUNCH_CHECK("k_sel_pick");
    LC_CUDA(cudaMemcpyAsync(hs, st, sizeof(SelState), cudaMemcpyDeviceToHost, s));
  };
  pick();
  LC_CUDA(cudaStreamSynchronize(s));

  while (hs->kc > 0 && !(budget_total > 0 && hs->kept >= budget_total)) {
    const int kc = hs->kc;
    k_sel_gather<<<(unsigned)((kc + 7) / 8), 256, 0, s>>>(x.rows, kc, H, h->d, x.G);
    LC_LAUNCH_CHECK("k_sel_gather");
    probe(h, x.G, kc, x.hit, nullptr, nullptr, s);
    const unsigned tiles = (unsigned)((kc + kCovT - 1) / kCovT);
    k_sel_cover<<<dim3(tiles, tiles), 256, 0, s>>>(x.G, h->d, kc, x.rows, h->ins_rr, x.cov);
    LC_LAUNCH_CHECK("k_sel_cover");
    ResolveArgs ra;
    ra.cov = x.cov;
    ra.rows = x.rows;
    ra.hit = x.hit;
    ra.label = h->ins_label;
    ra.class_cnt = x.class_cnt;
    ra.st = st;
    ra.list = x.list;
    ra.stats = h->stats;
    ra.kc = kc;
    ra.C = h->C;
    ra.budget_pc = budget_per_class;
    ra.budget_total = budget_total;
    k_sel_resolve<<<1, 1024, 0, s>>>(ra);
    LC_LAUNCH_CHECK("k_sel_resolve");
    SelScatterArgs sa;
    sa.list = x.list;
    sa.st = st;
    sa.rows = x.rows;
    sa.G = x.G;
    sa.d = h->d;
    sa.dpad = h->dpad;
    sa.size0 = h->size;
    sa.rr = h->ins_rr;
    sa.tau = h->ins_tau;
    sa.kn = h->ins_kn;
    sa.radius = h->ins_radius;
    sa.label = h->ins_label;
    sa.yG = h->ins_yG;
    sa.t = h->table;
    sa.out_index = out_index;
    sa.unfit = &h->report->unfit;
    k_sel_scatter<<<(unsigned)(kTailBlocks + (kc + 7) / 8), 256, 0, s>>>(sa);
    LC_LAUNCH_CHECK("k_sel_scatter");
    pick();  // the next chunk's members, so that one wait serves both
    fetch_report(h, s);  // (the next chunk's probe: whether the FP16 copies still serve; an aborted one)
    LC_CUDA(cudaStreamSynchronize(s));
    h->size += hs->n_list;
    if (h->stats_host->abort_flag) {
      store_size_dev(h, s);  // the chunks before this one stay
      LC_CUDA(cudaStreamSynchronize(s));
      throw Error(LIPCACHE_E_DEVICE, "a bounded wait of the probe kernel expired: the selection stopped");
    }
  }
  store_size_dev(h, s);  // the table grew from the host
  return hs->kept;
}

int64_t select_kcenter(lipcache* h, const float* H, int64_t n, const int32_t* payload, int require_consistency,
                       int budget_per_class, int64_t* out_index, float* out_radius, cudaStream_t s) {
  SelectScratch& x = h->sel;
  const int C = h->C;
  certify_rows(h, H, n, payload, require_consistency, s);
  require_certify_ok(h, s);
  const unsigned nb = (unsigned)((n + 255) / 256);
  if (out_index) {
    k_fill_i64<<<nb, 256, 0, s>>>(out_index, n, -1);
    LC_LAUNCH_CHECK("k_fill_i64");
  }
  if (out_radius) {
    k_copy_f32<<<nb, 256, 0, s>>>(h->ins_radius, out_radius, n);
    LC_LAUNCH_CHECK("k_copy_f32");
  }
  int64_t npow = 1;
  while (npow < n) npow <<= 1;
  grow_to(x.keys, x.keys_cap, npow);
  ensure_chunk_scratch(h);
  // counters: [0] candidates, [1] centres
  int64_t* small = reinterpret_cast<int64_t*>(x.state);
  int64_t* small_host = reinterpret_cast<int64_t*>(h->sel_host);
  LC_CUDA(cudaMemsetAsync(small, 0, sizeof(int64_t) * 2, s));
  const unsigned npb = (unsigned)((npow + 255) / 256);
  k_kc_keys<<<npb, 256, 0, s>>>(h->ins_accept, h->ins_label, n, npow, C, x.keys, small);
  LC_LAUNCH_CHECK("k_kc_keys");
  sort_keys(x.keys, npow, s);
  LC_CUDA(cudaMemcpyAsync(small_host, small, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  LC_CUDA(cudaStreamSynchronize(s));
  const int64_t n_in = small_host[0];
  if (n_in == 0) return 0;
  // per-class segments, counts and offsets share one int32 scratch: seg[2C], cnt[C], off[C]
  grow_to(x.kc_seg, x.kc_seg_cap, 4 * (int64_t)C);
  int32_t* seg = x.kc_seg;
  int32_t* cnt = seg + 2 * C;
  int32_t* off = cnt + C;
  LC_CUDA(cudaMemsetAsync(seg, 0, sizeof(int32_t) * 2 * C, s));
  k_kc_segments<<<(unsigned)((n_in + 255) / 256), 256, 0, s>>>(x.keys, n_in, seg);
  LC_LAUNCH_CHECK("k_kc_segments");
  grow_to(x.kc_mind, x.kc_mind_cap, n_in);
  grow_to(x.kc_rows, x.kc_rows_cap, n_in);
  k_kcenter<<<C, kKcThreads, sizeof(float) * (size_t)h->d, s>>>(x.keys, seg, H, h->d, h->ins_radius, budget_per_class,
                                                                x.kc_mind, x.kc_rows, cnt);
  LC_LAUNCH_CHECK("k_kcenter");
  k_kc_scan<<<1, 1024, 0, s>>>(cnt, C, off, small + 1);
  LC_LAUNCH_CHECK("k_kc_scan");
  const int per = budget_per_class;
  k_kc_scatter<<<dim3((unsigned)((per + 7) / 8 < 64 ? (per + 7) / 8 : 64), (unsigned)(C + 1)), 256, 0, s>>>(
      seg, cnt, off, x.kc_rows, H, h->d, h->dpad, h->size, h->ins_rr, h->ins_tau, h->ins_kn, h->ins_radius,
      h->ins_label, h->ins_yG, h->table, out_index, &h->report->unfit, small + 1, C);
  LC_LAUNCH_CHECK("k_kc_scatter");
  LC_CUDA(cudaMemcpyAsync(small_host + 1, small + 1, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  LC_CUDA(cudaStreamSynchronize(s));
  const int64_t kept = small_host[1];
  h->size += kept;
  store_size_dev(h, s);  // the table grew from the host
  return kept;
}

void release_select(lipcache* h) {
  SelectScratch& x = h->sel;
  cudaFree(x.chunk);
  cudaFree(x.keys);
  cudaFree(x.kc_mind);
  cudaFree(x.kc_seg);
  cudaFree(x.kc_rows);
  x = SelectScratch{};
}

}  // namespace lc
