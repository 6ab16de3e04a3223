// Spectral norm of the GuardNet head: sigma_max(W), the Lipschitz constant of
// f(z) = W z + b (Sec. 4.1, Eqs. 17-19; the bias cancels in logit
// differences). Algorithm 1 computes it once per cache, before any radius.
//
// Method: power iteration on A = X^T X in FP64, X = W or W^T, whichever has
// fewer columns (the singular values are the same). Power iteration alone needs
// about log(tol) / log(lambda_2/lambda_1) steps, which is thousands for the
// small spectral gaps of Gaussian heads, so the start vector is produced by
// `squarings` normalised squarings A_{k+1} = (A_k 2^-e)^2, 2^e <= tr A_k < 2^(e+1), i.e. by the
// power iteration with A^(2^k) (up to 2^40 steps for the default 40; it stops
// once A_k is a projector to FP64's resolution). The final
// iteration then runs on X itself (w = X v, theta = ||w||^2 = v^T A v,
// u = X^T w) until successive Rayleigh quotients agree to 1e-13 relative and
// ||A v - theta v|| <= 1e-10 theta.
//
// FP64 on this GPU: a dependent instruction takes ~64 cycles, and four warps of
// an SM together issue one every ~22 (measured), so the work is laid out for
// that pipe: one cooperative kernel (k_spectral) holds the whole method, four
// warps on each of as many SMs as the shape fills, a lane per output element.
#include "internal.cuh"

namespace lc {
namespace {

constexpr int kSpThreads = 128;            // one warp per SM sub-partition
constexpr int kSpWarps = kSpThreads / 32;
constexpr int kSpChunk = 128;              // summation steps staged in shared memory at a time
constexpr long long kSpWaitLimit = 1LL << 31;  // ~1 s at GB300 clocks
constexpr unsigned kSpAbort = 0x80000000u;

// Barrier of the whole (co-resident) grid; `target` arrivals in all. Bounded:
// on expiry the abort bit releases every CTA and all return false.
__device__ bool grid_barrier(unsigned* ctr, unsigned target) {
  __shared__ unsigned seen;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    unsigned v;
    const long long t0 = clock64();
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
      if (v >= target) break;
      if (clock64() - t0 > kSpWaitLimit) v = atomicOr(ctr, kSpAbort) | kSpAbort;
    }
    seen = v;
  }
  __syncthreads();
  return (seen & kSpAbort) == 0;
}

// Sum over 256 slots, slot l + 32 m in v[m] of lane l, in the order of a
// shared-memory tree (slot t += slot t + s for s = 128, 64, ..., 1); slots
// from n on are zero and are left out (adding +0 changes nothing). Every lane
// returns the sum.
__device__ double tree256(double (&v)[8], int n) {
#pragma unroll
  for (int s = 4; s > 0; s >>= 1)
#pragma unroll
    for (int m = 0; m < s; ++m)
      if (32 * (m + s) < n) v[m] = v[m] + v[m + s];
  double x = v[0];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = x + __shfl_down_sync(0xffffffffu, x, o);
  return __shfl_sync(0xffffffffu, x, 0);
}

// Sum of x(k)^2, k < n: slot t adds k = t, t + 256, ... in order.
template <typename F>
__device__ double sum_squares(int n, int lane, F x) {
  double v[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    v[m] = 0.0;
    for (int k = lane + 32 * m; k < n; k += 256) {
      const double e = x(k);
      v[m] = fma(e, e, v[m]);
    }
  }
  return tree256(v, n);
}

// One fused multiply-add chain sum_k col[k stride] x[k], k < n ascending, the
// loads of sixteen steps in flight while the sixteen before them are added.
__device__ double chain16(const double* col, size_t stride, const double* x, int n) {
  constexpr int N = 16;
  double acc = 0.0, cur[N], nxt[N];
#pragma unroll
  for (int u = 0; u < N; ++u) cur[u] = u < n ? __ldcg(col + (size_t)u * stride) : 0.0;
  for (int k = 0; k < n; k += N) {
#pragma unroll
    for (int u = 0; u < N; ++u) nxt[u] = k + N + u < n ? __ldcg(col + (size_t)(k + N + u) * stride) : 0.0;
#pragma unroll
    for (int u = 0; u < N; ++u)
      if (k + u < n) acc = fma(cur[u], x[k + u], acc);
#pragma unroll
    for (int u = 0; u < N; ++u) cur[u] = nxt[u];
  }
  return acc;
}

// X (m x n) is W (C x d) or its transpose.
struct SpectralArgs {
  const float* W;
  int m, n, mp, np;  // mp, np: m, n rounded up to 32
  int rs, cs;        // X(r, j) = W[r rs + j cs]
  int squarings, max_iter, n_tiles;
  double* A[2];    // n x np, blocked layout (columns from n on are never read into a result)
  double* X;       // m x np, blocked layout: X in FP64, zero past n
  double* XT;      // n x mp, zero past m
  double* w;       // segments(n) x mp: partial sums of X v
  double* u;       // segments(m) x np: partial sums of X^T w
  unsigned* ctr;   // grid barrier, zero at launch
  SpecResult* res;
};

// The iteration's products run in segments of kSeg steps, each a chain of its
// own on some warp of the grid, added in order afterwards: a chain's step takes
// 64 cycles, so whole chains took 5 to 8 us a product at 128 to 256 steps (the
// kernel at C = 200: d = 128 179 -> 162 us, d = 256 380 -> 356 us).
constexpr int kSeg = 32;
__host__ __device__ constexpr int segments(int n) { return (n + kSeg - 1) / kSeg; }
__device__ __forceinline__ double add_segments(const double* p, int stride, int n) {
  double s = 0.0;
  for (int g0 = 0; g0 < n; g0 += 8) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = g0 + u < n ? __ldcg(p + (size_t)(g0 + u) * stride) : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (g0 + u < n) s += v[u];
  }
  return s;
}

// Element (k, j) of a matrix with K rows in column blocks of 32: a block's
// rows are contiguous (a panel of 32 columns is one stream; rows of a
// power-of-two length apart cost 80 cycles a request at d = 256).
__device__ __forceinline__ size_t blk(int k, int j, int K) { return ((size_t)(j >> 5) * K + k) * 32 + (j & 31); }

// One warp: red[1] = tr S (blocked layout), red[0] = 2^-2e with 2^e <= tr S <
// 2^(e+1), the exact factor that normalises S^2, or 0 for a zero trace (W = 0).
__device__ void trace_scale(const double* S, int n, int lane, double* red) {
  double v[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int k = lane + 32 * m;
    v[m] = k < n ? __ldcg(S + blk(k, k, n)) : 0.0;
  }
  if (n > 256)
#pragma unroll
    for (int m = 0; m < 8; ++m)
      for (int k = lane + 32 * m + 256; k < n; k += 256) v[m] += __ldcg(S + blk(k, k, n));
  const double tr = tree256(v, n);
  if (lane == 0) {
    // tr W^T W of finite FP32 values has |e| < 350; the clamp is for NaN
    int e = (int)((__double_as_longlong(tr) >> 52) & 2047) - 1023;
    e = e < -500 ? -500 : (e > 500 ? 500 : e);
    red[0] = tr > 0.0 ? __longlong_as_double((long long)(1023 - 2 * e) << 52) : 0.0;
    red[1] = tr;
  }
}

// The symmetric product P_ij = sum_k S[k][i] S[k][j] (k < K ascending, one
// fused multiply-add chain per element) into B, with `scale` times the power
// of two that normalises S (taken on the result, so the panels need no
// products of their own: 1 / tr S on the panels, a division and up to 40
// multiplications per 128 steps of a warp, took 55 us of 435 at C = 200,
// d = 256 and 15 of 73 at C = 10, d = 64). S (K rows, blocked layout) is
// symmetric or is the operand itself, so one panel of columns and one of rows
// serve, and only i <= j is computed ((j, i) would add the same products in the same order). A tile is
// 32 columns (lanes) by 4 R rows (R chains per warp); tiles are numbered over
// the upper triangle.
template <int R>
__device__ void sym_product(const double* S, int K, bool scale, double* B, int d, int n_tiles, double* sm,
                            double* red) {
  constexpr int kRows = kSpWarps * R;
  double* cp = sm;                   // kSpChunk x 32
  double* rp = sm + kSpChunk * 32;   // kSpChunk x kRows
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int per = 32 / kRows;  // row blocks per 32 rows
  bool have_tr = !scale;
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    int cb = 0, rb = tile;  // column block cb has (cb + 1) * per row blocks
    while (rb >= (cb + 1) * per) {
      rb -= (cb + 1) * per;
      ++cb;
    }
    const int j0 = cb * 32, i0 = rb * kRows;
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0;
    for (int k0 = 0; k0 < K; k0 += kSpChunk) {
      const int kc = K - k0 < kSpChunk ? K - k0 : kSpChunk;
      __syncthreads();
      // every load of the panels is issued before the first is used (one L2
      // round trip per chunk)
      constexpr int NC = kSpChunk / kSpWarps, NR = kSpChunk * kRows / kSpThreads;
      double xc[NC], xr[NR];
      const double* sc = S + blk(k0, j0 + lane, K);
      const double* sr = S + blk(k0, i0 + tid % kRows, K);
#pragma unroll
      for (int u = 0; u < NC; ++u) {
        const int k = warp + u * kSpWarps;
        xc[u] = k < kc ? __ldcg(sc + k * 32) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < NR; ++u) {
        const int k = tid / kRows + u * (kSpThreads / kRows);
        xr[u] = k < kc ? __ldcg(sr + k * 32) : 0.0;
      }
      if (!have_tr) {
        // the trace, while the panels are on their way
        if (warp == 0) trace_scale(S, d, lane, red);
        have_tr = true;
      }
#pragma unroll
      for (int u = 0; u < NR; ++u) {
        const int k = tid / kRows + u * (kSpThreads / kRows);
        if (k < kc) rp[k * kRows + tid % kRows] = xr[u];
      }
#pragma unroll
      for (int u = 0; u < NC; ++u) {
        const int k = warp + u * kSpWarps;
        if (k < kc) cp[k * 32 + lane] = xc[u];
      }
      __syncthreads();
#pragma unroll 8
      for (int k = 0; k < kc; ++k) {
        const double c = cp[k * 32 + lane];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = fma(rp[k * kRows + warp * R + r], c, acc[r]);
      }
    }
    const double f = scale ? red[0] : 1.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = i0 + warp * R + r, j = j0 + lane;
      if (i <= j && j < d) {
        const double p = acc[r] * f;
        B[blk(i, j, d)] = p;
        if (i < j) B[blk(j, i, d)] = p;
      }
    }
  }
}

// The spectral norm of W by a co-resident grid: FP64 copies of X, A = X^T X,
// `squarings` steps A <- (A 2^-e)^2, then the power iteration on X. What
// bounds it: the FP64 pipe (four warps per SM: ~88 cycles per step of their
// chains); a squaring costs its n steps, the trace and one grid barrier.
template <int R>
__global__ void __launch_bounds__(kSpThreads) k_spectral(const SpectralArgs a) {
  __shared__ double sm[kSpChunk * 32 + kSpChunk * kSpWarps * R];
  __shared__ double red[2];
  static_assert(kSpChunk * 32 >= 2 * 1024 + 1024, "the iteration's vectors share the panels' space");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m = a.m, n = a.n, mp = a.mp;
  unsigned bar = 0;
  auto sync_grid = [&]() { return grid_barrier(a.ctr, bar += gridDim.x); };

  for (int e = blockIdx.x * kSpThreads + tid; e < m * a.np; e += gridDim.x * kSpThreads) {
    const int r = e / a.np, j = e - r * a.np;
    a.X[blk(r, j, m)] = j < n ? (double)a.W[(size_t)r * a.rs + (size_t)j * a.cs] : 0.0;
  }
  for (int e = blockIdx.x * kSpThreads + tid; e < n * mp; e += gridDim.x * kSpThreads) {
    const int j = e / mp, r = e - j * mp;
    a.XT[e] = r < m ? (double)a.W[(size_t)r * a.rs + (size_t)j * a.cs] : 0.0;
  }
  if (!sync_grid()) return;
  // A grid with fewer tiles than CTAs (units of the iteration): the spare CTAs
  // only follow the traces and meet the barriers.
  int cur = 0;
  if (a.squarings > 0) {
    // X^T X: products of FP32 values are exact in FP64
    sym_product<R>(a.X, m, false, a.A[0], n, a.n_tiles, sm, red);
    if (!sync_grid()) return;
    double s2 = 0.0;  // (tr A_k 2^-e)^2 of the matrix before
    for (int q = 0; q < a.squarings; ++q) {
      sym_product<R>(a.A[cur], n, true, a.A[cur ^ 1], n, a.n_tiles, sm, red);
      if ((int)blockIdx.x >= a.n_tiles) {  // a spare CTA follows the traces
        if (warp == 0) trace_scale(a.A[cur], n, lane, red);
        __syncthreads();
      }
      cur ^= 1;
      const double tr = red[1], f = red[0];  // of the matrix just squared
      if (!sync_grid()) return;
      // With unit trace, the matrix before is, from its purity t = tr / s2 = sum
      // l_i^2 (l_1 >= ... summing to 1), the projector on the dominant direction
      // up to (1 - t) / 2 relative; its square up to about the square of that,
      // and the one just formed below FP64's resolution. Gaussian heads take 10
      // to 14 steps; a (nearly) repeated largest singular value keeps t away
      // from 1 and takes them all.
      if (q > 0 && s2 - tr <= 1e-9 * s2) break;
      s2 = tr * tr * f;
    }
  }

  // Power iteration on X: every CTA keeps v and repeats the short sums; the
  // chains of w = X v and u = X^T w are spread over the grid.
  double* v = sm;
  double* w = sm + 1024;
  double* u = sm + 2048;
  __syncthreads();
  if (a.squarings > 0) {
    const double* A = a.A[cur];
    // the dominant column: the first largest diagonal entry
    if (warp == 0) {
      double best = -INFINITY;
      int at = 0x7fffffff;
      for (int k = lane; k < n; k += 32) {
        const double x = __ldcg(A + blk(k, k, n));
        if (x > best) {
          best = x;
          at = k;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oa = __shfl_xor_sync(0xffffffffu, at, o);
        if (ob > best || (ob == best && oa < at)) {
          best = ob;
          at = oa;
        }
      }
      if (lane == 0) red[0] = (double)(at < n ? at : 0);
    }
    __syncthreads();
    const int js = (int)red[0];
    for (int k = tid; k < n; k += kSpThreads) v[k] = __ldcg(A + blk(js, k, n));
  } else {
    for (int k = tid; k < n; k += kSpThreads) {
      unsigned x = (unsigned)k * 2654435761u;
      x ^= x >> 15;
      v[k] = 1.0 + 0.01 * (double)(x & 0xffff) / 65536.0;
    }
  }
  __syncthreads();
  double nv = sqrt(sum_squares(n, lane, [&](int k) { return v[k]; }));
  if (!(nv > 0.0)) {
    if (blockIdx.x == 0 && tid == 0) {
      a.res->sigma = 0.0;
      a.res->theta = 0.0;
      a.res->residual_rel = 0.0;
      a.res->iterations = 0;
      a.res->converged = 1;
      a.res->degenerate = 1;
    }
    return;
  }
  __syncthreads();
  for (int k = tid; k < n; k += kSpThreads) v[k] /= nv;
  __syncthreads();

  const int mu = mp / 32, nu32 = a.np / 32;  // 32-lane units of the two products, times their segments
  const int sv = segments(n), sw = segments(m);
  double theta = 0.0, theta_prev = -1.0, resid = INFINITY;
  int it = 0, converged = 0;
  for (it = 1; it <= a.max_iter; ++it) {
    for (int g = blockIdx.x + gridDim.x * warp; g < mu * sv; g += gridDim.x * kSpWarps) {
      const int r = g % mu * 32 + lane, k0 = g / mu * kSeg;
      a.w[(size_t)(g / mu) * mp + r] = chain16(a.XT + (size_t)k0 * mp + r, mp, v + k0, n - k0 < kSeg ? n - k0 : kSeg);
    }
    if (!sync_grid()) return;
    for (int r = tid; r < m; r += kSpThreads) w[r] = add_segments(a.w + r, mp, sv);
    __syncthreads();
    if (warp == kSpWarps - 1) {
      const double p = sum_squares(m, lane, [&](int r) { return w[r]; });
      if (lane == 0) red[0] = p;
    } else {
      for (int g = blockIdx.x + gridDim.x * warp; g < nu32 * sw; g += gridDim.x * (kSpWarps - 1)) {
        const int k = g % nu32 * 32 + lane, r0 = g / nu32 * kSeg;
        a.u[(size_t)(g / nu32) * a.np + k] = chain16(a.X + blk(r0, k, m), 32, w + r0, m - r0 < kSeg ? m - r0 : kSeg);
      }
    }
    if (!sync_grid()) return;
    theta = red[0];
    for (int k = tid; k < n; k += kSpThreads) u[k] = add_segments(a.u + k, a.np, sw);
    __syncthreads();
    if (warp == 0) {
      const double pr = sum_squares(n, lane, [&](int k) { return fma(-theta, v[k], u[k]); });
      if (lane == 0) red[0] = pr;
    } else if (warp == 1) {
      const double pu = sum_squares(n, lane, [&](int k) { return u[k]; });
      if (lane == 0) red[1] = pu;
    }
    __syncthreads();
    resid = sqrt(red[0]);
    const double nu = sqrt(red[1]);
    __syncthreads();
    if (!(nu > 0.0)) {  // v is in the null space of X: only possible for W = 0
      theta = 0.0;
      resid = 0.0;
      converged = 1;
      break;
    }
    for (int k = tid; k < n; k += kSpThreads) v[k] = u[k] / nu;
    __syncthreads();
    if (it >= 2 && fabs(theta - theta_prev) <= 1e-13 * theta && resid <= 1e-10 * theta) {
      converged = 1;
      break;
    }
    theta_prev = theta;
  }
  if (blockIdx.x == 0 && tid == 0) {
    a.res->theta = theta;
    a.res->sigma = sqrt(theta);
    a.res->residual_rel = theta > 0.0 ? resid / theta : 0.0;
    a.res->iterations = it > a.max_iter ? a.max_iter : it;
    a.res->converged = converged;
    a.res->degenerate = !(theta > 0.0);
  }
}

// ||W_c|| (rounded up) for every class and, for the tight radius, ||W_y - W_j|| for every
// pair (FP64; the differences of FP32 weights are exact, the sum of d squares
// is within gamma_d of the exact one) with its reciprocal, and FP32 brackets
// of the reciprocal (the FP64 value widened by 1e-12, far above its error,
// then rounded outward; +inf for coinciding rows, which the tight radius skips).
// One warp per unit (y, 32 classes j) of the upper triangle, a lane per pair;
// the mirrored pair squares the negated differences, the same sum. Bound by
// the FP64 pipe: two instructions per feature and 32 pairs.
// Feature k of class c is Wt[(c / 32) bs + k ks + c % 32].
__global__ void __launch_bounds__(kSpThreads) k_row_norms(const double* __restrict__ Wt, size_t bs, size_t ks, int C,
                                                          int Cp, int d,
                                                          float* __restrict__ Wnorm32,
                                                          double* __restrict__ pairnorm,
                                                          double* __restrict__ inv_pairnorm,
                                                          float* __restrict__ ipn_up32, float* __restrict__ ipn_dn32) {
  const int lane = threadIdx.x & 31;
  const int unit = blockIdx.x * kSpWarps + (threadIdx.x >> 5);
  const int nb = Cp / 32;
  if (unit < nb) {
    const int c = unit * 32 + lane;
    const double* wc = Wt + (size_t)unit * bs + lane;
    double n2 = 0.0;
#pragma unroll 8
    for (int k = 0; k < d; ++k) {
      const double x = wc[k * ks];
      n2 = fma(x, x, n2);
    }
    if (c < C) Wnorm32[c] = __double2float_ru(sqrt(n2) * (1.0 + 1e-15));
    return;
  }
  if (!pairnorm) return;
  int r = unit - nb, jb = 0;  // class block jb holds the units y < min(C, 32 (jb + 1))
  for (; jb < nb; ++jb) {
    const int ny = C < 32 * (jb + 1) ? C : 32 * (jb + 1);
    if (r < ny) break;
    r -= ny;
  }
  if (jb >= nb) return;
  const int y = r, j = jb * 32 + lane;
  const double* wy = Wt + (size_t)(y >> 5) * bs + (y & 31);
  const double* wj = Wt + (size_t)jb * bs + lane;
  double acc = 0.0;
#pragma unroll 8
  for (int k = 0; k < d; ++k) {
    const double e = wy[k * ks] - wj[k * ks];
    acc = fma(e, e, acc);
  }
  if (j >= C || j < y) return;
  const double pn = sqrt(acc);
  const double ipn = acc > 0.0 ? 1.0 / sqrt(acc) : 0.0;
  const float up = acc > 0.0 ? __double2float_ru(ipn * (1.0 + 1e-12)) : INFINITY;
  const float dn = acc > 0.0 ? __double2float_rd(ipn * (1.0 - 1e-12)) : INFINITY;
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    const size_t at = m ? (size_t)j * C + y : (size_t)y * C + j;
    pairnorm[at] = pn;
    inv_pairnorm[at] = ipn;
    ipn_up32[at] = up;
    ipn_dn32[at] = dn;
  }
}

// Bounds of a whole row of the bracket tables, which the tensor certify
// kernel's tight-radius screen uses in place of the tables:
// ipn_min32[y] <= 1 / ||W_y - W_j|| for every j with W_j != W_y (the minimum of
// the FP32 lower brackets; 0 when every other row equals W_y) and
// ipn_max32[y] >= 1 / ||W_y - W_j|| for every j != y (+inf when some W_j = W_y).
__global__ void __launch_bounds__(128) k_ipn_min(const double* __restrict__ pairnorm, const float* __restrict__ ipn_dn32,
                                                 const float* __restrict__ ipn_up32, int C,
                                                 float* __restrict__ ipn_min32, float* __restrict__ ipn_max32) {
  const int y = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (y >= C) return;
  float m = INFINITY, mx = 0.f;
  for (int j = lane; j < C; j += 32) {
    if (j == y) continue;
    if (pairnorm[(size_t)y * C + j] > 0.0) m = fminf(m, ipn_dn32[(size_t)y * C + j]);
    mx = fmaxf(mx, ipn_up32[(size_t)y * C + j]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if (lane == 0) {
    ipn_min32[y] = m < INFINITY ? m : 0.f;
    ipn_max32[y] = mx;
  }
}

// Tiles of sym_product over the upper triangle of a d x d matrix.
int sym_tiles(int d, int R) {
  const int nb = (d + 31) / 32, per = 32 / (kSpWarps * R);
  return nb * (nb + 1) / 2 * per;
}

template <int R>
void launch_spectral(lipcache* h, SpectralArgs a, cudaStream_t s) {
  a.n_tiles = sym_tiles(a.n, R);
  const int units = (a.mp > a.np ? a.mp : a.np) / 32;
  int grid = a.n_tiles > units ? a.n_tiles : units;
  if (grid > h->num_sms) grid = h->num_sms;
  void* args[] = {&a};
  LC_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_spectral<R>), dim3((unsigned)grid),
                                      dim3(kSpThreads), args, 0, s));
  LC_LAUNCH_CHECK("k_spectral");
}

}  // namespace

size_t spectral_work_bytes(int d, int C) {
  const size_t Cp = (size_t)(C + 31) / 32 * 32;
  const size_t dp = (size_t)(d + 31) / 32 * 32;
  return sizeof(double) * (2 * dp * d + dp * C + Cp * d + segments(d) * Cp + segments(C) * dp) + 16;  // (either orientation)
}

void spectral_norm(lipcache* h, cudaStream_t s) {
  const int d = h->d, C = h->C;
  // The transpose of a head with fewer classes than features: a squaring's
  // chains and tiles shrink with the smaller dimension (the kernel, C = 10,
  // d = 64: 85 us on W, 58 on W^T; C = 200, d = 256: 441 and 380; both with whole
  // chains in the iteration). Without squarings the start
  // vector is fixed and the iteration stays on W.
  const bool tr = C < d && h->squarings > 0;
  SpectralArgs a;
  a.W = h->W;
  a.m = tr ? d : C;
  a.n = tr ? C : d;
  a.rs = tr ? 1 : d;
  a.cs = tr ? d : 1;
  a.mp = (a.m + 31) / 32 * 32;
  a.np = (a.n + 31) / 32 * 32;
  a.squarings = h->squarings;
  a.max_iter = h->max_iter;
  double* p = reinterpret_cast<double*>(h->spec_work);
  a.A[0] = p;
  a.A[1] = a.A[0] + (size_t)a.np * a.n;
  a.X = a.A[1] + (size_t)a.np * a.n;
  a.XT = a.X + (size_t)a.np * a.m;
  a.w = a.XT + (size_t)a.mp * a.n;
  a.u = a.w + (size_t)segments(a.n) * a.mp;
  a.ctr = reinterpret_cast<unsigned*>(a.u + (size_t)segments(a.m) * a.np);
  a.res = h->spec;
  LC_CUDA(cudaMemsetAsync(a.ctr, 0, sizeof(unsigned), s));
  // a barrier that expired leaves this in place: neither converged nor degenerate
  LC_CUDA(cudaMemsetAsync(h->spec, 0xff, sizeof(SpecResult), s));
  // Chains per warp: one while the tiles of one-row warps fit the SMs once
  // (n <= 160: 120 tiles); above, two do the same products per sub-partition
  // with half the panel loads (n = 256: 144 tiles).
  if (sym_tiles(a.n, 1) <= h->num_sms)
    launch_spectral<1>(h, a, s);
  else
    launch_spectral<2>(h, a, s);
  const int Cp = (C + 31) / 32 * 32;
  const bool tight = h->radius_mode == LIPCACHE_RADIUS_TIGHT;
  const int nb = Cp / 32;
  int units = nb;
  if (tight)
    for (int jb = 0; jb < nb; ++jb) units += C < 32 * (jb + 1) ? C : 32 * (jb + 1);
  k_row_norms<<<(units + kSpWarps - 1) / kSpWarps, kSpThreads, 0, s>>>(
      tr ? a.X : a.XT, tr ? (size_t)32 * d : 32, tr ? 32 : (size_t)Cp, C, Cp, d, h->Wnorm32, tight ? h->pairnorm : nullptr, tight ? h->inv_pairnorm : nullptr,
      tight ? h->ipn_up32 : nullptr, tight ? h->ipn_dn32 : nullptr);
  LC_LAUNCH_CHECK("k_row_norms");
  if (tight) {
    k_ipn_min<<<(C + 3) / 4, 128, 0, s>>>(h->pairnorm, h->ipn_dn32, h->ipn_up32, C, h->ipn_min32, h->ipn_max32);
    LC_LAUNCH_CHECK("k_ipn_min");
  }
}

}  // namespace lc
