// Tensor-core probe: screen every (query, key) pair with a tcgen05 contraction
// in FP16 (or TF32, below), recheck the few candidates with the exact canonical
// FP32 distance (Sec. 3.4, Algorithm 2, Eqs. 13-15; cost model Eq. 16).
//
// Operands. The screen reads the table's FP16 copy and FP16 queries scaled per
// row by a power of two (key16.cuh): the same 11-bit significand as TF32, at
// half the bytes and twice the MMA rate. Its error against q.k in 64 bits is
// that of cuBLAS' TF32 product (both 2.59e-5 |q| |k| root mean square, 1.5e-4
// at most, d = 128; equal to three digits from d = 16 to 512). 4,096 queries x
// 4M keys, d = 128: 4.26 ms in TF32, 2.25 ms in FP16 (1.87 PFLOP/s, against
// 2.19 ms at the cuBLAS bf16 rate); bound by the tensor pipe and the ~100
// issue cycles between accumulators. A table with an entry outside FP16's
// range, or whose copy found no memory, is screened in TF32 from the FP32
// keys. Either way the recheck below decides every pair in FP32, so the
// results are the same bits.
//
// Screen. For a pair with exact squared distance S = |q|^2 + |k|^2 - 2 q.k,
// the tensor cores return a = q.k up to |a - q.k| <= c |q| |k| <= c (|q|^2 +
// |k|^2) / 2 (FP32 accumulation; c = c_screen). Every pair the
// recheck can accept has S < R_k = rr_k / (1 - gamma_rc), hence
//     a > (1 - c) |q|^2 / 2 + ((1 - c) |k|^2 - R_k) / 2 = kappa_q + tau_k,
// with kappa_q (per query, k_prologue) rounded down and tau_k (per key,
// stored at insertion) rounded down. The epilogue keeps a pair iff
// fl(a - tau_k) >= kappa_q, which therefore never drops an acceptable pair. The
// rows that fill the last query tile up get a NaN for kappa and pass nothing.
// It first tests each 32-key chunk with fl(max a - min tau) >= kappa_q, which no
// chunk holding a kept pair fails; the maximum comes with the TMEM load
// (tcgen05.ld.red), and only a passing chunk's products are looked at.
//
// Schedule. Persistent CTAs, one per SM, launched as clusters of two. The two
// CTAs of a cluster own two adjacent key tiles and stream the SAME sequence of
// query tiles: each CTA TMA-loads one half of every query stage with
// .multicast::cluster into both CTAs' shared memory, so the L2 delivers each
// query byte once per pair of SMs (the query stream from L2 is what limits a
// single CTA). Per CTA (352 threads):
//   warp 0     TMA producer: the CTA's key tile (BN keys x d_pad, resident,
//              one barrier pair per 128-byte chunk so the next tile streams in
//              while the last query tile still runs) and its half of each
//              query stage (128 queries x 128 bytes per stage, multi-stage ring);
//   warp 1     allocates TMEM, issues tcgen05.mma kind::f16 / kind::tf32 (M=128
//              queries, N=BN keys, 32 bytes of K) into one of two TMEM
//              accumulators; releases each query stage in BOTH CTAs;
//   warps 2-9  epilogue: tcgen05.ld of the accumulator (warp w reads TMEM
//              lane quarter w % 4, column half (w - 2) / 4), screen; the pairs
//              that pass go to
//   warp 10    the recheck, atomicMin of the packed (distance, index) word,
//              through a queue in shared memory, so that the loads of a pair's
//              rows (3 us on an epilogue warp) do not hold up the next tiles.
// Work: the items (key-tile pair, query tile), pair-major, are split into
// equal contiguous ranges, one per cluster; a run is the part of a range on
// one pair, and its key tile stays resident through the run (a pair split
// between two clusters is loaded by both). When the number of key tiles is odd
// the last pair's second tile lies past the table: that CTA multiplies the
// TMA's zero fill and its epilogue skips the run, so both CTAs still consume
// every query stage.
#include "internal.cuh"
#include "probe_common.cuh"
#include "tc_ptx.cuh"

namespace lc {
namespace {

constexpr int kBM = 128;              // queries per tile (MMA M)
constexpr int kMaxStages = 8;         // query ring depth limit (runtime count fills shared memory)
constexpr int kMaxChunks = 8;         // d_pad <= 256 (TF32), d <= 512 (FP16)
constexpr int kQStageBytes = kBM * 128;
constexpr int kQHalfBytes = kQStageBytes / 2;
#ifndef LC_EPI_WARPS
#define LC_EPI_WARPS 8
#endif
constexpr int kEpiWarps = LC_EPI_WARPS;  // 4 or 8: one or two per SM sub-partition
constexpr int kRecheckWarp = 2 + kEpiWarps;
constexpr int kThreads = 32 * (3 + kEpiWarps);
constexpr int kCluster = 2;
constexpr uint16_t kClusterMask = 0x3;
constexpr int kSmemBudget = 227 * 1024 - 1024;  // opt-in limit minus the alignment slack
constexpr long long kWaitLimit = 1LL << 31;     // ~1 s at GB300 clocks
constexpr int64_t kPairedReleaseItems = 64;     // items per cluster from which stages are released in pairs

struct TcArgs {
  int nst;       // query ring stages
  int qgroup;    // stages released together, 1 or 2 (the kernel instantiation; divides nst)
  int tau_staged;  // screen terms copied to shared memory per run (short runs), else read through L1
  int nch;       // 128-byte chunks per row
  int ksteps;    // MMAs of the last chunk that hold features (the others take four)
  int dpad;      // row stride of keys (and of qpad)
  int d, qvec;   // FP16: features of a query, its rows readable 16 bytes at a time
  int nq;        // query tiles
  int n_pairs;   // key-tile pairs
  int n_kt;      // key tiles (of BN) holding cache entries
  const float* kappa;
  const float* qscale;  // FP16: undoes the queries' scaling
  const float* q;       // recheck: padded FP32 queries (TF32), the caller's own (FP16)
  const float* keys;
  const float* tau;
  const float* rr;
  unsigned long long* best;
  ProbeOut out;
  DevStats* stats;
  int queue;        // candidates go to the recheck warp (ranges of several tiles)
  int debug_stall;  // test hook: the MMA issuer first waits on a barrier nothing arrives on
};

// Pairs on their way from the epilogue warps to the recheck warp (shared
// memory): pair number k is in slot k % kRecheckQ once seq there is k + 1.
// Without that warp (short ranges) each epilogue warp keeps its own kWarpQ of
// the slots and rechecks what they hold when they are full or its tiles are
// done: one round of loads instead of one per chunk (256 queries on 2,000
// entries, d = 64, 113 pairs: 19.4 us per chunk, 15.7 us so).
constexpr int kRecheckQ = 64;
constexpr int kWarpQ = kRecheckQ / kEpiWarps;
struct RecheckQueue {
  int n;      // slots reserved
  int taken;  // pairs rechecked (their slots are free)
  int done;   // epilogue warps past their last tile
  int pad;
  int2 pair[kRecheckQ];  // query row, key
  int seq[kRecheckQ];
};

template <int BN>
struct Layout {
  static constexpr int kKChunkBytes = BN * 128;
  static constexpr int kTmemCols = 2 * BN;
  static constexpr int kTauStaged = 4 * BN * 4;  // one private slice of screen terms per epilogue warp
  int nk, nst, tau_staged;  // nk: resident key chunks; tau_staged: the screen terms copied per run (else through L1)
  __device__ __host__ int kbytes() const { return nk * kKChunkBytes; }
  __device__ __host__ int qoff() const { return kbytes(); }
  __device__ __host__ int tauoff() const { return qoff() + nst * kQStageBytes; }
  __device__ __host__ int baroff() const { return tauoff() + (tau_staged ? kTauStaged : 0); }
  // barriers: full_k[nk], empty_k[nk], full_q[nst], empty_q[nst], acc_full[2], acc_empty[2], drain
  __device__ __host__ int nbar() const { return 2 * nk + 2 * nst + 5; }
  __device__ __host__ int miscoff() const { return (baroff() + 8 * nbar() + 15) / 16 * 16; }
  __device__ __host__ int rqoff() const { return miscoff() + 16; }
  __device__ __host__ int total() const { return rqoff() + (int)sizeof(RecheckQueue); }
  // deepest ring that fits the shared-memory budget
  static __host__ int stages_for(int nk, int tau_staged) {
    for (int n = kMaxStages; n >= 2; --n) {
      Layout<BN> L{nk, n, tau_staged};
      if (L.total() <= kSmemBudget) return n;
    }
    return 0;
  }
};

// The runs of one cluster: its range [it, end) of items (pair, query tile),
// pair-major; next() gives this CTA's key tile (of NH times BN keys) and the
// run's query tiles.
struct RunCursor {
  long long it, end;
  __device__ RunCursor(const TcArgs& a, int cluster_id, int n_clusters) {
    const long long T = (long long)a.n_pairs * a.nq;
    it = T * cluster_id / n_clusters;
    end = T * (cluster_id + 1) / n_clusters;
  }
  __device__ bool next(const TcArgs& a, uint32_t rank, int& kt, int& qt0, int& qt1) {
    if (it >= end) return false;
    const int pair = (int)(it / a.nq);
    qt0 = (int)(it - (long long)pair * a.nq);
    const long long run_end = min(end, (long long)(pair + 1) * a.nq);
    qt1 = qt0 + (int)(run_end - it);
    kt = pair * kCluster + (int)rank;
    it = run_end;
    return true;
  }
};

// MODE 0: short ranges (screen terms staged in shared memory, stages released
// one at a time); 1: long ranges (screen terms through L1), single releases;
// 2: long ranges, stages released in pairs.
// NH: key tiles of BN held side by side. With two (rows of at most two chunks,
// long ranges), every query stage is multiplied by both before it is released,
// half the stage writes, L2 reads and releases per MMA; the two accumulators
// then belong to the two halves.
template <int BN, int MODE, int KIND, int NH>
__global__ void __launch_bounds__(kThreads, 1)
    k_probe_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const TcArgs a) {
  constexpr int QG = MODE == 2 ? 2 : 1;  // query stages released together
  constexpr bool kTauStaged = MODE == 0;
  using Op = ScreenOp<KIND>;
  constexpr int kChunkF = Op::kChunk;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // 1024-byte alignment of the swizzled tiles
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int nk = NH * a.nch;
  const Layout<BN> L{nk, a.nst, a.tau_staged};
  const uint32_t s_base = ptx::smem_u32(smem);
  const uint32_t s_k = s_base;
  const uint32_t s_q = s_base + L.qoff();
  const uint32_t s_bar = s_base + L.baroff();
  const uint32_t full_k = s_bar, empty_k = s_bar + 8 * nk;
  const uint32_t full_q = s_bar + 16 * nk, empty_q = full_q + 8 * a.nst;
  const uint32_t acc_full = empty_q + 8 * a.nst, acc_empty = acc_full + 16, drain = acc_empty + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L.miscoff());
  volatile int* abort_s = reinterpret_cast<volatile int*>(smem + L.miscoff() + 4);
  RecheckQueue* rq = reinterpret_cast<RecheckQueue*>(smem + L.rqoff());

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  const int cluster_id = blockIdx.x / kCluster, n_clusters = gridDim.x / kCluster;

  if (threadIdx.x == 0) {
    for (int c = 0; c < nk; ++c) {
      ptx::mbar_init(full_k + 8 * c, 1);
      ptx::mbar_init(empty_k + 8 * c, 1);
    }
    for (int s = 0; s < a.nst; ++s) {
      ptx::mbar_init(full_q + 8 * s, 1);         // own arrival; bytes from both CTAs
      ptx::mbar_init(empty_q + 8 * s, kCluster); // released by the MMA of both CTAs
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(acc_full + 8 * b, 1);
      ptx::mbar_init(acc_empty + 8 * b, kEpiWarps);
    }
    ptx::mbar_init(drain, 1);
    *abort_s = 0;
    ptx::fence_mbar_init();
    ptx::tma_prefetch_desc(&tmQ);
    ptx::tma_prefetch_desc(&tmK);
  }
  if (warp == kRecheckWarp) {
    for (int k = lane; k < kRecheckQ; k += 32) rq->seq[k] = 0;
    if (lane == 0) rq->n = rq->taken = rq->done = 0;
  }
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_u32(tmem_slot), (uint32_t)Layout<BN>::kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  ptx::cluster_sync();  // the peer's barriers exist before any multicast reaches them
  ptx::wait_prerequisites();  // the prologue's queries, constants and reduction words
  const uint32_t tmem = *tmem_slot;

  const Recheck rck{a.q, KIND == kF16 ? a.d : a.dpad, KIND == kF16 ? a.qvec != 0 : true, a.keys, a.dpad, a.d, a.rr, a.best};
  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int qs = 0;
      uint32_t qph = 0;
      int i = 0;
      int last_k_par[kMaxChunks];
      uint32_t last_q_par[kMaxStages];
      bool q_used[kMaxStages];
      for (int c = 0; c < kMaxChunks; ++c) last_k_par[c] = -1;
      for (int s = 0; s < kMaxStages; ++s) {
        q_used[s] = false;
        last_q_par[s] = 0;
      }
      bool ok = true;
      RunCursor rc(a, cluster_id, n_clusters);
      int kt, qt0, qt1;
      for (; ok && rc.next(a, rank, kt, qt0, qt1); ++i) {
        for (int qt = qt0; qt < qt1 && ok; ++qt) {
          // key chunk c of half h of this run, as soon as the previous run's
          // last query tile has finished with it (past the table: zero fill)
          auto load_key = [&](int h, int c) {
            const int kc = h * a.nch + c;
            if (!ptx::mbar_wait(empty_k + 8 * kc, (uint32_t)(i & 1) ^ 1u, abort_s, kWaitLimit)) return false;
            ptx::mbar_expect_tx(full_k + 8 * kc, (uint32_t)Layout<BN>::kKChunkBytes);
            ptx::tma_load_2d(s_k + kc * Layout<BN>::kKChunkBytes, &tmK, c * kChunkF, (kt * NH + h) * BN, full_k + 8 * kc);
            last_k_par[kc] = i & 1;
            return true;
          };
          for (int c = 0; c < a.nch && ok; ++c) {
            if (qt == qt0) {
              ok = load_key(0, c);
              if (!ok) break;
            }
            // stage qs is free in both CTAs (its group was released); fetch
            // this CTA's half for both
            if (QG == 1 || (qs & 1) == 0) {
              ok = ptx::mbar_wait(empty_q + 8 * (qs >> (QG - 1)), qph ^ 1u, abort_s, kWaitLimit);
              if (!ok) break;
            }
            ptx::mbar_expect_tx(full_q + 8 * qs, (uint32_t)kQStageBytes);
            ptx::tma_load_2d_multicast(s_q + qs * kQStageBytes + rank * kQHalfBytes, &tmQ, c * kChunkF,
                                       qt * kBM + (int)rank * (kBM / 2), full_q + 8 * qs, kClusterMask);
            q_used[qs] = true;
            last_q_par[qs] = qph;
            if (++qs == a.nst) {
              qs = 0;
              qph ^= 1u;
            }
          }
          if (NH == 2 && qt == qt0)
            for (int c = 0; c < a.nch && ok; ++c) ok = load_key(1, c);
        }
      }
      // Let every copy into this CTA land before it can exit. (Bounded; a
      // phase that already completed returns at once.)
      volatile int never = 0;
      for (int s = 0; s < a.nst; ++s)
        if (q_used[s]) ptx::mbar_wait(full_q + 8 * s, last_q_par[s], &never, kWaitLimit);
      for (int c = 0; c < nk; ++c)
        if (last_k_par[c] >= 0) ptx::mbar_wait(full_k + 8 * c, (uint32_t)last_k_par[c], &never, kWaitLimit);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // The tensor pipe queues about one MMA ahead, so the issuing path has to be
    // short. The whole warp runs it converged (waits by vote, so the compiler
    // keeps descriptors and loop state in uniform registers, which the MMA
    // instruction reads) and one elected lane issues. Descriptors are advanced
    // by adding encoded offsets (the start-address field holds address >> 4, so
    // +32 bytes is +2 and never carries out of the field); the once-per-run key
    // waits and releases run in a separate edge path.
    {
      constexpr uint32_t idesc = Op::idesc(kBM, BN);
      const bool lead = ptx::elect_one();
      const uint64_t qdesc0 = ptx::sw128_kmajor_desc(s_q);
      const uint64_t kdesc0 = ptx::sw128_kmajor_desc(s_k);
      constexpr uint64_t kQStride = kQStageBytes >> 4;
      constexpr uint64_t kKStride = Layout<BN>::kKChunkBytes >> 4;
      const int nst = a.nst, nch = a.nch, ksl = a.ksteps;
      int qs = 0;
      uint32_t qph = 0;
      int t = 0, i = 0;
      // failure-detection test: no arrival ever completes this phase, so the
      // bounded wait expires and the kernel takes its abort path
      bool ok = !a.debug_stall || ptx::mbar_wait_warp(drain, 0, abort_s, kWaitLimit);
      RunCursor rc(a, cluster_id, n_clusters);
      int kt, qt0, qt1;
      for (; ok && rc.next(a, rank, kt, qt0, qt1); ++i) {
        for (int qt = qt0; qt < qt1 && ok; ++qt) {
          const bool first = qt == qt0, last = qt == qt1 - 1;
          const int qb = qs;  // first stage of the query tile and its phase
          const uint32_t qbph = qph;
#pragma unroll
          for (int h = 0; h < NH; ++h, ++t) {
            if (NH == 2 && h == 1) {
              qs = qb;
              qph = qbph;
            }
            const int buf = NH == 2 ? h : t & 1;
            if (!ptx::mbar_wait_warp(acc_empty + 8 * buf, (uint32_t)((t >> 1) & 1) ^ 1u, abort_s, kWaitLimit)) {
              ok = false;
              break;
            }
            const uint32_t d_tmem = tmem + (uint32_t)(buf * BN);
            uint64_t kd = kdesc0 + (uint64_t)(h * nch) * kKStride;
            for (int c = 0; c < nch; ++c, kd += kKStride) {
              if (first && !ptx::mbar_wait_warp(full_k + 8 * (h * nch + c), (uint32_t)(i & 1), abort_s, kWaitLimit)) {
                ok = false;
                break;
              }
              if (h == 0 && !ptx::mbar_wait_warp(full_q + 8 * qs, qph, abort_s, kWaitLimit)) {
                ok = false;
                break;
              }
              ptx::tc_fence_after();
              const uint64_t qd = qdesc0 + (uint64_t)qs * kQStride;
              const int steps = c == nch - 1 ? ksl : 4;
              if (lead) {
                Op::chunk(d_tmem, qd, kd, idesc, c != 0, steps);
                if (h == NH - 1 && (QG == 1 || (qs & 1)))
                  ptx::mma_commit_multicast(empty_q + 8 * (qs >> (QG - 1)), kClusterMask);
                if (last) ptx::mma_commit(empty_k + 8 * (h * nch + c));
                if (c == nch - 1) ptx::mma_commit(acc_full + 8 * buf);
              }
              if (++qs == nst) {
                qs = 0;
                qph ^= 1u;
              }
            }
            if (!ok) break;
          }
        }
      }
      // all issued MMAs complete before TMEM can be released
      if (lead) {
        volatile int never = 0;
        ptx::mma_commit(drain);
        ptx::mbar_wait(drain, 0, &never, kWaitLimit);
      }
    }
    __syncwarp();
  } else if (warp == kRecheckWarp) {
    // ------------------------------------------------------------ recheck
    // the pairs the epilogue warps hand over, as they come; ends once every
    // epilogue warp is done (each is, also after an abort) and none is left
    unsigned long long ncand = 0;
    volatile RecheckQueue* vq = rq;
    for (int k = 0; a.queue;) {
      const unsigned ready = __ballot_sync(0xffffffffu, vq->seq[(k + lane) % kRecheckQ] == k + lane + 1);
      const int m = ready == 0xffffffffu ? 32 : __ffs((int)~ready) - 1;
      if (m == 0) {
        if (__any_sync(0xffffffffu, vq->done == kEpiWarps)) {
          __threadfence_block();
          if (__all_sync(0xffffffffu, vq->n == k)) break;
          continue;
        }
        // (every look takes shared-memory cycles from the MMAs)
        __nanosleep(kTauStaged ? 250 : 1000);
        continue;
      }
      __threadfence_block();
      int row = 0, key = 0;
      if (lane < m) {
        row = vq->pair[(k + lane) % kRecheckQ].x;
        key = vq->pair[(k + lane) % kRecheckQ].y;
      }
      recheck_warp(rck, lane < m ? 1u : 0u, row, key, lane, ncand);
      k += m;
      __threadfence_block();
      __syncwarp();
      if (lane == 0) vq->taken = k;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ncand += __shfl_xor_sync(0xffffffffu, ncand, o);
    if (lane == 0 && ncand) atomicAdd(&a.stats->candidates, ncand);
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 2;
    const int quarter = warp & 3;         // TMEM lane quarter this warp may access
    const int half = ew >> 2;             // column slice
    constexpr int kColsPerWarp = BN * 4 / kEpiWarps;
    constexpr int kChunks = kColsPerWarp / 32;
    // this warp's private slice of the screen terms when they are staged
    float* my_tau = reinterpret_cast<float*>(smem + L.tauoff()) + ew * kColsPerWarp;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    int t = 0;
    bool ok = true;
    unsigned long long ncand = 0;
    int held = 0;  // pairs in this warp's own slots
    auto flush = [&]() {
      __syncwarp();
      int2 pr = make_int2(0, 0);
      if (lane < held) pr = rq->pair[ew * kWarpQ + lane];
      recheck_warp(rck, lane < held ? 1u : 0u, pr.x, pr.y, lane, ncand);
      held = 0;
      __syncwarp();
    };
    RunCursor rc(a, cluster_id, n_clusters);
    int kt, qt0, qt1;
    while (ok && rc.next(a, rank, kt, qt0, qt1)) {
      const int key0 = kt * (NH * BN) + half * kColsPerWarp;  // + h BN for half h of the key tile
      // the minimum of this warp's screen terms over each 32-key chunk of
      // the run's key tile. The per-pair test, which few chunks reach, reads
      // the terms themselves from a copy in shared memory made here when the
      // runs are short, else through L1 (the space goes to a deeper query
      // ring).
      if (kTauStaged) {
        __syncwarp();
        if (kt < a.n_kt)
          for (int v4 = lane; v4 < kColsPerWarp / 4; v4 += 32)
            reinterpret_cast<float4*>(my_tau)[v4] = __ldg(reinterpret_cast<const float4*>(a.tau + key0) + v4);
        __syncwarp();
      }
      float tmin[NH][kChunks];
#pragma unroll
      for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int ch = 0; ch < kChunks; ++ch) {
          float m = kt * NH + h >= a.n_kt ? INFINITY
                    : kTauStaged          ? my_tau[ch * 32 + lane]
                                          : __ldg(a.tau + key0 + h * BN + ch * 32 + lane);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
          tmin[h][ch] = m;
        }
      float kap = row_kappa(a.kappa, qt0 * kBM + quarter * 32 + lane, a.out.B);
      float scl = KIND == kF16 ? __ldg(a.qscale + qt0 * kBM + quarter * 32 + lane) : 1.f;
      for (int qt = qt0; qt < qt1 && ok; ++qt) {
        const int row = qt * kBM + quarter * 32 + lane;
        // next tile's screen constant, fetched while this accumulator is produced
        const float kap_next = (qt + 1 < qt1) ? row_kappa(a.kappa, row + kBM, a.out.B) : 0.f;
        const float scl_next = (KIND == kF16 && qt + 1 < qt1) ? __ldg(a.qscale + row + kBM) : 1.f;
#pragma unroll
        for (int h = 0; h < NH; ++h, ++t) {
        const int buf = t & 1;
        const bool live = kt * NH + h < a.n_kt;
        const float* __restrict__ tau_g = a.tau + key0 + h * BN;
        ok = ptx::mbar_wait(acc_full + 8 * buf, (uint32_t)((t >> 1) & 1), abort_s, kWaitLimit);
        ok = __all_sync(0xffffffffu, ok);  // warp-uniform before the aligned TMEM loads
        if (!ok) break;
        ptx::tc_fence_after();
        // Coarse test of each 32-key chunk: a_j - tau_j <= max_j a_j - min_j tau_j
        // exactly, and rounding is monotone, so a chunk whose value for (max a,
        // min tau) is below kappa holds no pair that passes. The TMEM load
        // itself reduces the products (tcgen05.ld.red): no instruction per
        // product, and an accumulator without a passing chunk is handed back
        // at once.
        const uint32_t tbase = tmem + lane_base + (uint32_t)(buf * BN + half * kColsPerWarp);
        uint32_t pass = 0;
#pragma unroll
        for (int ch = 0; ch < kChunks; ch += 2) {
          uint32_t va[32], vb[32];
          float amax[2];
          ptx::tmem_ld32_max(tbase + (uint32_t)(ch * 32), va, amax[0]);
          ptx::tmem_ld32_max(tbase + (uint32_t)(ch * 32 + 32), vb, amax[1]);
          ptx::tmem_wait_ld();
          ptx::hold32(va);
          ptx::hold32(vb);
#pragma unroll
          for (int u = 0; u < 2; ++u)
            pass |= (uint32_t)(screen_value<KIND>(amax[u], scl, tmin[h][ch + u]) >= kap) << (ch + u);
        }
        if (!live) pass = 0;
        // The chunks some row passes in, one copy of code for all (rarely run
        // code is fetched as it goes): the pairs that pass from the products,
        // the accumulator handed back once the last of those is loaded, then
        // the recheck.
        uint32_t chunks = __reduce_or_sync(0xffffffffu, pass);
        if (chunks == 0) {
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(acc_empty + 8 * buf);
        }
#pragma unroll 1
        while (chunks) {
          const int ch = __ffs((int)chunks) - 1;
          chunks &= chunks - 1;
          uint32_t v[32];
          ptx::tmem_ld32(tbase + (uint32_t)(ch * 32), v);
          ChunkTau ct;
          load_chunk_tau<!kTauStaged>(ct, (kTauStaged ? my_tau : tau_g) + ch * 32);
          ptx::tmem_wait_ld();
          if (chunks == 0) {
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(acc_empty + 8 * buf);
          }
          // with close keys and few features most passing chunks hold no pair
          // that passes (1.5 million keys x 1,909 queries like them, d = 24: 1005 us
          // with 32 loads, products and comparisons for each, 619 with this)
          const float least = screen_chunk<KIND>(v, ct, scl);
          const bool some = ((pass >> ch) & 1u) && least <= -kap;
          if (!__any_sync(0xffffffffu, some)) continue;
          uint32_t mask = 0;
#pragma unroll
          for (int j = 0; j < 32; ++j) mask |= (uint32_t)(__uint_as_float(v[j]) <= -kap) << j;
          mask = some ? mask : 0u;
          const int mine = __popc(mask);
          const int cnt = __reduce_add_sync(0xffffffffu, mine);
          const int first_key = key0 + h * BN + ch * 32;
          // to the recheck warp if there are tiles to go on with and its queue
          // has room, or to the warp's own slots, else here
          int base = -1;
          if (!a.queue) {
            if (held + cnt > kWarpQ && held) flush();
            if (cnt <= kWarpQ) {
              base = held;
              held += cnt;
            }
          } else if (lane == 0) {
            volatile RecheckQueue* vq = rq;
            for (int n = vq->n; n + cnt - vq->taken <= kRecheckQ;) {
              const int was = atomicCAS(&rq->n, n, n + cnt);
              if (was == n) {
                base = n;
                break;
              }
              n = was;
            }
          }
          base = __shfl_sync(0xffffffffu, base, 0);
          if (base < 0) {
            recheck_warp(rck, mask, row, first_key, lane, ncand);
            continue;
          }
          int at = mine;  // inclusive prefix of the lanes' counts
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += x;
          }
          for (at += base - mine; mask; mask &= mask - 1, ++at) {
            const int slot = a.queue ? at % kRecheckQ : ew * kWarpQ + at;
            rq->pair[slot] = make_int2(row, first_key + __ffs((int)mask) - 1);
            if (a.queue) {
              __threadfence_block();
              *(volatile int*)&rq->seq[slot] = at + 1;
            }
          }
          __syncwarp();
        }
        }
        kap = kap_next;
        scl = scl_next;
      }
    }
    if (held) flush();
    __syncwarp();
    if (lane == 0) {
      __threadfence_block();
      atomicAdd(&rq->done, 1);
    }
    // candidate count: one atomic per warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ncand += __shfl_xor_sync(0xffffffffu, ncand, o);
    if (lane == 0 && ncand) atomicAdd(&a.stats->candidates, ncand);
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_s) {
    // A role gave up: leave time for copies the peer may still be
    // multicasting into this CTA before the cluster retires.
    if (threadIdx.x == 0) {
      atomicAdd(&a.stats->errors, 1ull);
      atomicExch(&a.stats->abort_flag, kProbeAborted);
    }
    __nanosleep(50000);
  }
  ptx::cluster_sync();  // no remote arrival or copy can target an exited CTA
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, (uint32_t)Layout<BN>::kTmemCols);
  }
  finalize_last_cta(a.out, gridDim.x, abort_s + 1);
}

template <int BN, int KIND, int NH>
void launch_nh(lipcache* h, int64_t B, const ProbeBuffers& b, const ProbeOut& out, bool long_ranges, cudaStream_t s) {
  constexpr bool f16 = KIND == kF16;
  const int64_t Bpad = (B + kBM - 1) / kBM * kBM;
  lipcache::ProbeLaunch& pl = h->probe_launch[(BN == 256 ? 0 : 1) + (f16 ? 3 : 0)];
  const void* kbase = f16 ? static_cast<const void*>(h->table.keys16) : h->table.keys;
  if (pl.q_base != b.q || pl.q_rows != (uint64_t)Bpad) {
    encode_screen_map(h, &pl.tmQ, b.q, (uint64_t)Bpad, kBM / 2, f16);  // half a query tile per CTA of the pair
    pl.q_base = b.q;
    pl.q_rows = (uint64_t)Bpad;
  }
  if (pl.k_base != kbase || pl.k_rows != (uint64_t)h->table_rows) {
    encode_screen_map(h, &pl.tmK, kbase, (uint64_t)h->table_rows, BN, f16);
    pl.k_base = kbase;
    pl.k_rows = (uint64_t)h->table_rows;
  }
  TcArgs a;
  a.nch = f16 ? h->table.d16 / 64 : h->dpad / 32;
  a.ksteps = f16 ? (h->d - 64 * (a.nch - 1) + 15) / 16 : 4;
  // (the ring depth depends on whether the screen terms are staged: below)
  a.dpad = h->dpad;
  a.d = h->d;
  a.qvec = h->d % 4 == 0 && ((uintptr_t)b.Q & 15) == 0;
  a.nq = (int)(Bpad / kBM);
  const int64_t n_kt = (h->size + BN - 1) / BN;
  const int64_t n_pairs = (n_kt + NH * kCluster - 1) / (NH * kCluster);
  const int max_clusters = h->num_sms / kCluster;
  // Long ranges (many items per cluster, the large caches): the screen terms
  // are read through L1, the shared memory goes to the query ring, and the
  // stages are released two at a time (one commit per pair) when a tile's
  // stages pair up and the ring holds whole pairs. Short ranges keep the
  // staged screen terms and single releases, which measure faster there.
  a.tau_staged = long_ranges ? 0 : 1;
  a.nst = Layout<BN>::stages_for(NH * a.nch, a.tau_staged);
  // (two halves hold a whole query tile of stages while the next one loads)
  LC_REQUIRE(a.nst >= (NH == 2 ? a.nch + 2 : 2), LIPCACHE_E_INVALID, "key tile does not fit shared memory");
  a.qgroup = (long_ranges && a.nst % 2 == 0 && a.nst >= 4 && a.nch % 2 == 0) ? 2 : 1;
  LC_REQUIRE(n_pairs * a.nq < (1LL << 40), LIPCACHE_E_INVALID, "too many work items");
  a.n_pairs = (int)n_pairs;
  a.n_kt = (int)n_kt;
  a.kappa = b.kappa;
  a.qscale = b.scale;
  a.q = f16 ? b.Q : static_cast<const float*>(b.q);
  a.keys = h->table.keys;
  a.tau = h->probe_tau();
  a.rr = h->probe_rr();
  a.best = b.best;
  a.out = out;
  a.stats = h->stats;
  // With one to three tiles per cluster the recheck warp's turn would only come
  // at the end: 256 x 50,000 at d = 64 13.4 us without it, 15.0 with; 1,024 x
  // 50,000 at d = 128 (ten tiles) 22.1 without, 20.7 with. The line lies between
  // these two; nothing in between was measured.
  a.queue = n_pairs * a.nq >= 6 * (int64_t)max_clusters ? 1 : 0;
  a.debug_stall = (h->debug_flags & LIPCACHE_DEBUG_STALL_PROBE) ? 1 : 0;
  const Layout<BN> L{NH * a.nch, a.nst, a.tau_staged};
  const int smem = L.total() + 1024;
  // (two halves only run the long modes)
  constexpr int kM0 = NH == 2 ? 1 : 0;
  if (!pl.smem[NH - 1]) {
    // the attribute belongs to the kernel, not to this cache: set it to the
    // largest size any shape uses, so other caches' launches stay valid
    LC_CUDA(cudaFuncSetAttribute(k_probe_tc<BN, kM0, KIND, NH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmemBudget + 1024));
    LC_CUDA(cudaFuncSetAttribute(k_probe_tc<BN, 1, KIND, NH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmemBudget + 1024));
    LC_CUDA(cudaFuncSetAttribute(k_probe_tc<BN, 2, KIND, NH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmemBudget + 1024));
    pl.smem[NH - 1] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(max_clusters * kCluster));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // starts its setup behind the prologue kernel's last wave
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  // persistent grid: no more clusters than can be resident at once (asked for
  // with the most shared memory any launch uses)
  if (pl.resident == 0) {
    cfg.dynamicSmemBytes = (size_t)kSmemBudget + 1024;
    LC_CUDA(cudaOccupancyMaxActiveClusters(&pl.resident, k_probe_tc<BN, 1, KIND, NH>, &cfg));
    cfg.dynamicSmemBytes = (size_t)smem;
  }
  const int resident = pl.resident;
  LC_REQUIRE(resident >= 1, LIPCACHE_E_CUDA, "no CTA pair of the probe kernel fits on this device");
  int clusters = max_clusters < resident ? max_clusters : resident;
  if (n_pairs * a.nq < clusters) clusters = (int)(n_pairs * a.nq);  // one item per cluster at least
  cfg.gridDim = dim3((unsigned)(clusters * kCluster));
  h->last_grid = clusters * kCluster;
  h->last_cluster = kCluster;
  if (h->launch_event) LC_CUDA(cudaEventRecord(h->launch_event, s));
  void (*kern)(CUtensorMap, CUtensorMap, TcArgs) =
      a.tau_staged       ? k_probe_tc<BN, kM0, KIND, NH>
      : a.qgroup == 2 ? k_probe_tc<BN, 2, KIND, NH>
                      : k_probe_tc<BN, 1, KIND, NH>;
  cfg.numAttrs = 2;
  LC_CUDA(cudaLaunchKernelEx(&cfg, kern, pl.tmQ, pl.tmK, a));
  LC_LAUNCH_CHECK("k_probe_tc");
}

template <int BN, int KIND>
void launch(lipcache* h, int64_t B, const ProbeBuffers& b, const ProbeOut& out, cudaStream_t s) {
  const int max_clusters = h->num_sms / kCluster;
  LC_REQUIRE(max_clusters >= 1, LIPCACHE_E_CUDA, "device has fewer than two SMs");
  const int64_t nq = (B + kBM - 1) / kBM, n_kt = (h->size + BN - 1) / BN;
  const bool long_ranges = (n_kt + kCluster - 1) / kCluster * nq / max_clusters >= kPairedReleaseItems;
  if constexpr (KIND == kF16 && BN == 256) {
    // two key tiles side by side leave a ring of six stages or more
    if (long_ranges && h->table.d16 <= 128) return launch_nh<BN, KIND, 2>(h, B, b, out, true, s);
  }
  launch_nh<BN, KIND, 1>(h, B, b, out, long_ranges, s);
}

}  // namespace

// Rows of 128-byte boxes: FP32 rows of d_pad, or FP16 rows of d16 features.
void encode_screen_map(lipcache* h, CUtensorMap* map, const void* base, uint64_t rows, uint32_t box_rows, bool f16) {
  LC_REQUIRE(h->encode != nullptr, LIPCACHE_E_CUDA, "cuTensorMapEncodeTiled is unavailable from the driver");
  const cuuint64_t width = f16 ? (cuuint64_t)h->table.d16 : (cuuint64_t)h->dpad;
  const cuuint64_t dims[2] = {width, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {width * (f16 ? sizeof(__half) : sizeof(float))};
  const cuuint32_t box[2] = {f16 ? 64u : 32u, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = h->encode(map, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                               const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  LC_REQUIRE(r == CUDA_SUCCESS, LIPCACHE_E_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
}

int launch_probe_tc(lipcache* h, int64_t B, int path, bool f16, const ProbeBuffers& b, const ProbeOut& out,
                    cudaStream_t s) {
  LC_REQUIRE(f16 || tensor_path_supported(h->dpad), LIPCACHE_E_INVALID, "the tensor probe supports d <= 256");
  // A 256-key tile of up to four chunks (d <= 256 in FP16, 128 in TF32) stays
  // beside a deep query ring: single-CTA MMAs on all SMs. Longer rows would
  // force 128-key tiles, whose MMAs read shared memory at its whole bandwidth;
  // pair MMAs read a third less per flop and take those (clusters of four
  // leave some SMs idle).
  const bool short_rows = f16 ? h->table.d16 <= 256 : h->dpad <= 128;
  const bool pair = path == LIPCACHE_PROBE_TENSOR_PAIR || (path == LIPCACHE_PROBE_TENSOR && !short_rows);
  if (pair && probe_pair_clusters(h, f16) >= 1) {
    launch_probe_pair(h, B, f16, b, out, s);
    return LIPCACHE_PROBE_TENSOR_PAIR;
  }
  if (f16) {
    if (short_rows)
      launch<256, kF16>(h, B, b, out, s);
    else
      launch<128, kF16>(h, B, b, out, s);
  } else {
    if (short_rows)
      launch<256, kTf32>(h, B, b, out, s);
    else
      launch<128, kTf32>(h, B, b, out, s);
  }
  return LIPCACHE_PROBE_TENSOR_SINGLE;
}

}  // namespace lc
