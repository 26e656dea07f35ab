// FP64 Householder QR and one-sided Jacobi SVD, batched over independent
// problems of one shape.
//
// A matrix is split by rows over a thread-block cluster of 1-16 CTAs, kept in
// shared memory where it fits, and the CTAs exchange partial sums through
// distributed shared memory: the QR with one cluster barrier per Householder
// column, the SVD with one per round of the round-robin Jacobi schedule.  A tall
// QR that has the device to itself runs on every SM instead.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <cstdlib>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "linalg.cuh"

namespace cg = cooperative_groups;

namespace peps {
namespace {

constexpr int QR_THREADS = 512;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = threadIdx.x < nw ? red[threadIdx.x] : 0.0;
    s = warp_sum(s);
    if (threadIdx.x == 0) red[0] = s;
  }
  __syncthreads();
  s = red[0];
  __syncthreads();
  return s;
}

struct QrArgs {
  int m, n;
  TP A;         // per problem
  long long rs, cs;
  TP Q;
  long long qrs, qcs;
  TP R;         // absent: R not wanted
  double* W;    // work per problem (problem p at W + p * wst): what k_qr_cluster's shared memory
                // does not hold (wst / C per CTA), k_qr_house's m x n copy
  double* Qw;   // k_qr_house: m*k work per problem, column-major (+ p * qst)
  double* tau;  // k_qr_house: k per problem (+ p * tst)
  long long wst, qst, tst;
  // k_qr_cluster<true>, P CTAs per problem (absent otherwise), per problem:
  int P;
  double* gpart;     // [n][P] the CTAs' partial sums
  double* gsum;      // [n] their sums
  double* grow;      // [2][n] row j of the matrix
  double* gtri;      // M, packed columns
  unsigned* gcount;  // four words QRG_LINE apart, zero at launch: arrivals with partial sums, with sums and with
                     // the largest high word, and that word
  int* flag;
};
constexpr int QRG_LINE = 32;    // 128 bytes
constexpr int QRG_MAXP = 160;   // five partial sums per lane

// Grid = problems, one CTA each, everything in global memory: for matrices with
// more columns than k_qr_cluster's shared memory holds sums for.
__global__ void __launch_bounds__(QR_THREADS) k_qr_house(const QrArgs q) {
  __shared__ double red[32];
  __shared__ double s_tau, s_scale;
  const int m = q.m, n = q.n, k = min(m, n);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int pb = blockIdx.x;
  const double* A = q.A.d(pb);
  double* const Qo = q.Q.d(pb);
  double* const Ro = q.R.n ? q.R.d(pb) : nullptr;
  double* const tau_g = q.tau + pb * q.tst;
  double* W = q.W + pb * q.wst;
  for (long long e = tid; e < (long long)m * n; e += nt) {
    int i = int(e % m), j = int(e / m);
    W[e] = A[i * q.rs + j * q.cs];
  }
  __syncthreads();
  for (int j = 0; j < k; ++j) {
    double part = 0.0;
    for (int i = j + 1 + tid; i < m; i += nt) {
      double v = W[(long long)j * m + i];
      part += v * v;
    }
    const double sig = block_sum(part, red);
    if (tid == 0) {
      const double alpha = W[(long long)j * m + j];
      if (sig == 0.0) {
        s_tau = 0.0;
        s_scale = 0.0;
      } else {
        const double nrm = sqrt(alpha * alpha + sig);
        const double beta = alpha >= 0.0 ? -nrm : nrm;
        s_tau = (beta - alpha) / beta;
        s_scale = 1.0 / (alpha - beta);
        W[(long long)j * m + j] = beta;
      }
      tau_g[j] = s_tau;
    }
    __syncthreads();
    const double tau = s_tau, scale = s_scale;
    if (tau != 0.0) {
      for (int i = j + 1 + tid; i < m; i += nt) W[(long long)j * m + i] *= scale;
      __syncthreads();
      for (int c = j + 1 + warp; c < n; c += nw) {
        double w = 0.0;
        for (int i = j + 1 + lane; i < m; i += 32) w += W[(long long)j * m + i] * W[(long long)c * m + i];
        w = warp_sum(w) + W[(long long)c * m + j];
        w *= tau;
        if (lane == 0) W[(long long)c * m + j] -= w;
        for (int i = j + 1 + lane; i < m; i += 32) W[(long long)c * m + i] -= w * W[(long long)j * m + i];
      }
    }
    __syncthreads();
  }
  // Q = H_0 ... H_{k-1} [I_k; 0], accumulated backwards.
  double* Qw = q.Qw + pb * q.qst;
  for (long long e = tid; e < (long long)m * k; e += nt) {
    int i = int(e % m), j = int(e / m);
    Qw[e] = (i == j) ? 1.0 : 0.0;
  }
  __syncthreads();
  for (int j = k - 1; j >= 0; --j) {
    const double tau = tau_g[j];
    if (tau != 0.0) {
      for (int c = j + warp; c < k; c += nw) {
        double w = 0.0;
        for (int i = j + 1 + lane; i < m; i += 32) w += W[(long long)j * m + i] * Qw[(long long)c * m + i];
        w = warp_sum(w) + Qw[(long long)c * m + j];
        w *= tau;
        if (lane == 0) Qw[(long long)c * m + j] -= w;
        for (int i = j + 1 + lane; i < m; i += 32) Qw[(long long)c * m + i] -= w * W[(long long)j * m + i];
      }
    }
    __syncthreads();
  }
  for (long long e = tid; e < (long long)m * k; e += nt) {
    int i = int(e % m), j = int(e / m);
    Qo[i * q.qrs + j * q.qcs] = Qw[e];
  }
  if (Ro) {
    for (long long e = tid; e < (long long)k * n; e += nt) {
      int i = int(e / n), j = int(e % n);
      Ro[e] = (j >= i) ? W[(long long)j * m + i] : 0.0;
    }
  }
}


// Sum of one double over the cluster's CTAs, all remote loads issued first.
__device__ __forceinline__ double remote_sum(cg::cluster_group& cl, double* slot, int C) {
  double v[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) v[r] = r < C ? *cl.map_shared_rank(slot, r) : 0.0;
  double s = 0.0;
#pragma unroll
  for (int r = 0; r < 16; ++r) s += v[r];
  return s;
}

// ---------------------------------------------------------------------------
// Householder QR, one thread-block cluster of C = 1-16 CTAs per matrix, its
// rows split over the CTAs and kept in shared memory where they fit.
//
// What bounds it: GB300's FP64 pipe.  A warp's FP64 instruction holds the pipe
// of its SM quarter for 64 clocks whatever its active lanes, and a dependent
// one waits as long (an addition after a shuffle 110), so a column step costs
// its FP64 instructions: the fused update and inner products (2 per element),
// a few sums, and the scalar chain (1 / norm and one reciprocal, ~1,100 clocks).
// Barriers cost ~50 clocks for a CTA, ~450 for a cluster, a remote load ~400.
// Hence
//   * one pass per column: the update with reflector j and the inner products
//     with column j+1 (updated just before) read every element once;
//   * the reflector stays unscaled, x = (alpha - beta; a_ij): with s = |x_j|^2
//     over rows >= j, y = sgn(alpha) / sqrt(s), beta = -s y and
//     g = 1 / (s + |alpha| sqrt(s)), H = I - g x x^T.  For the inner product
//     f_c = sum_{i >= j} a_ij a_ic, row j of R is -y f_c and an updated entry
//     a_ic - w_c a_ij with w_c = g (f_c - beta a_jc);
//   * partial sums stay in their CTA's shared memory and are read from there
//     after the cluster barrier by four threads per column, all loads first;
//   * Q is formed from the reflectors at once and not one by one: the passes
//     also take the inner products x_a . x_j of the earlier reflectors (one
//     FMA per element), so X^T X is known when the last column is done, and
//     Q = E - X M with M = T X_1^T, where T^{-1} is upper triangular with
//     1 / g on the diagonal and X^T X above it (the UT transform: Joffrain,
//     Low, Quintana-Orti, van de Geijn & Van Zee, 2006).  Every column of M is
//     one back substitution in one warp, the columns dealt to the CTAs; the
//     product runs at the FP64 pipe's rate.  Against one barrier, one set of
//     sums and one pass per reflector (256x16 70 us, 512x32 158, 1024x64 441,
//     64x64 280) this takes 56, 136, 396 and 209 us.
// Measured (us, one matrix, with Q; before: scaled reflectors, update and inner
// products in two passes, sums by one thread per column, Q one reflector at a
// time): 256x16 117 -> 56, 512x32 236 -> 136, 1024x64 608 -> 396, 2304x64
// 824 -> 643, 1620x180 3637 -> 2897, 8192x128 (tall-skinny, four leaves)
// 3847 -> 2845; 16 of 36x36 270 -> 125 (those ran in global memory, one CTA
// each).  Orthogonality stays at 1e-15 to 7e-15; |A - QR| is 1 to 3 eps of a
// column's norm.  Shared memory holds the sums (88 bytes a column, to 2600
// columns), then the rows, M's columns and the triangle, each while it fits; the
// rest lies in global memory.  With M's columns in shared memory or nowhere,
// squares of more than 400 columns kept their rows in global memory and more
// than 592 columns ran on one CTA: 448x448 52.3 -> 7.3 ms, 640x600 120 -> 15.7,
// 1024x1024 475 -> 58.9, 9600x640 3009 -> 141.
//
// GRID: the rows of one matrix over every SM.  One cluster has 16 SMs, and of
// clusters of 16 only seven run at once, so that one matrix, or its leaves,
// left more than half of the chip idle.  The CTAs are no cluster here (a
// cooperative launch): the partial sums go through global memory in two steps,
// each counted -- every CTA publishes its n partial sums, one warp somewhere
// adds those of a column, and everyone reads the n sums.
// That costs a column about 5000 clocks more than one cluster's barrier and
// sums, so it pays where the rows of 16 CTAs cost more than that.
// Measured (us, one cluster or leaves -> every SM): 2304x64 643 -> 384,
// 1024x128 1155 -> 797, 4096x128 2110 -> 969, 8192x128 2845 -> 1250,
// 1620x180 2897 -> 1305, 8192x64 886 -> 501, three of 4096x128 2825 -> 1549.
// Clusters of 8, summed first within the cluster and then over 15 to 19 of
// them: 423, 776, 1010, 1362, 1602, 625, 1547.
// ---------------------------------------------------------------------------
constexpr int QRC_MAXT = 512;

// Per-CTA shared memory besides the rows, the columns of M and the triangle, in doubles.
__host__ __device__ inline long long qr_head(int n, int k) { return 7LL * n + 4LL * k + 4; }
// A CTA's columns of M.
__host__ __device__ inline long long qr_mc(int k, int c) { return (long long)((k + c - 1) / c) * k; }
// The triangle: X^T X, then M.
__host__ __device__ inline long long qr_tri(int k) { return (long long)k * (k + 1) / 2; }

// Sum over rows i, i + L, ... < r1 of x y.
__device__ __forceinline__ double qr_dot(const double* x, const double* y, int i, int L, int r1) {
  double acc = 0.0;
  for (; i + 3 * L < r1; i += 4 * L) {
    const int i1 = i + L, i2 = i1 + L, i3 = i2 + L;
    const double a0 = x[i], a1 = x[i1], a2 = x[i2], a3 = x[i3];
    const double b0 = y[i], b1 = y[i1], b2 = y[i2], b3 = y[i3];
    acc = fma(a0, b0, acc);
    acc = fma(a1, b1, acc);
    acc = fma(a2, b2, acc);
    acc = fma(a3, b3, acc);
  }
  for (; i < r1; i += L) acc = fma(x[i], y[i], acc);
  return acc;
}

// The same rows of one column: the update a -= w xj, and the sum of the
// results times xn.  The loads of four rows are issued before their arithmetic.
__device__ __forceinline__ double qr_update_dot(double* wc, const double* xj, const double* xn, double w, int i,
                                                int L, int r1) {
  double acc = 0.0;
  for (; i + 3 * L < r1; i += 4 * L) {
    const int i1 = i + L, i2 = i1 + L, i3 = i2 + L;
    const double a0 = wc[i], a1 = wc[i1], a2 = wc[i2], a3 = wc[i3];
    const double x0 = xj[i], x1 = xj[i1], x2 = xj[i2], x3 = xj[i3];
    const double n0 = xn[i], n1 = xn[i1], n2 = xn[i2], n3 = xn[i3];
    const double y0 = fma(-w, x0, a0), y1 = fma(-w, x1, a1), y2 = fma(-w, x2, a2), y3 = fma(-w, x3, a3);
    wc[i] = y0;
    wc[i1] = y1;
    wc[i2] = y2;
    wc[i3] = y3;
    acc = fma(y0, n0, acc);
    acc = fma(y1, n1, acc);
    acc = fma(y2, n2, acc);
    acc = fma(y3, n3, acc);
  }
  if (i + L < r1) {
    const int i1 = i + L;
    const double a0 = wc[i], a1 = wc[i1], x0 = xj[i], x1 = xj[i1], n0 = xn[i], n1 = xn[i1];
    const double y0 = fma(-w, x0, a0), y1 = fma(-w, x1, a1);
    wc[i] = y0;
    wc[i1] = y1;
    acc = fma(y0, n0, acc);
    acc = fma(y1, n1, acc);
    i += 2 * L;
  }
  if (i < r1) {
    const double y = fma(-w, xj[i], wc[i]);
    wc[i] = y;
    acc = fma(y, xn[i], acc);
  }
  return acc;
}

__device__ __forceinline__ void arrive_gpu(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ unsigned load_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Bounded wait for `target` arrivals: false, with the status word set, when it
// runs out.  About 2 s of SM clock between CTAs that are all running; the first
// wait of a launch, which also waits for the SMs that other kernels on the
// device still hold, gets a minute.
constexpr long long QRG_WAIT = 4000000000LL, QRG_FIRST_WAIT = 120000000000LL;
__device__ __forceinline__ bool wait_arrivals(const unsigned* p, unsigned target, int* flag,
                                              long long limit = QRG_WAIT) {
  const long long start = clock64();
  while (int(load_acquire_gpu(p) - target) < 0) {
    if (clock64() - start > limit) {
      atomicOr(flag, FLAG_TIMEOUT);
      return false;
    }
  }
  return true;
}

// lanes_log2: threads that share a column of the pass, 4 to 32: 128 threads
// are enough to keep the FP64 pipe busy, and each doubling adds an addition to
// every sum.
template <bool GRID>
__global__ void __launch_bounds__(QRC_MAXT) k_qr_cluster(const QrArgs q, int w_smem, int mc_smem, int tri_smem,
                                                         int ld, int lanes_log2) {
  extern __shared__ double qsm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = GRID ? q.P : int(cluster.num_blocks());   // CTAs of a problem
  const int pb = blockIdx.x / C;
  const int rank = GRID ? blockIdx.x - pb * C : int(cluster.block_rank());
  const double* A = q.A.d(pb);
  double* const Qo = q.Q.d(pb);
  double* const Ro = q.R.n ? q.R.d(pb) : nullptr;
  const int m = q.m, n = q.n, k = min(m, n);
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int chunk = (m + C - 1) / C;
  const int r0 = min(m, rank * chunk), r1 = min(m, r0 + chunk), rows = r1 - r0;
  const int mcols = (k + C - 1) / C;        // columns of M solved here: rank, rank + C, ...
  double* part = qsm;                       // [2][n] my partial sums (read by every CTA)
  double* rowv = part + 2 * n;              // [2][n] row j of the matrix (in the row's owner)
  double* dsum = rowv + 2 * n;              // [n] inner products of this step
  double* rowl = dsum + n;                  // [n] row j, local copy
  double* wfin = rowl + n;                  // [n] w_c of this step
  double* ys = wfin + n;                    // [k] y
  double* gs = ys + k;                      // [k] g
  double* nb = gs + k;                      // [k] -beta
  double* vs = nb + k;                      // [k] alpha - beta
  double* mc = vs + k + 4;                  // [mcols][k] my columns of X_1^T, then of M (read by every CTA)
  double* tri = mc + (mc_smem ? qr_mc(k, C) : 0); // packed columns: X^T X above the diagonal, then M
  double* W = tri + (tri_smem ? qr_tri(k) : 0);   // [n][ld], row i at i - r0
  double* const gpart = GRID ? q.gpart + (long long)pb * n * C : nullptr;
  double* const gsum = GRID ? q.gsum + (long long)pb * n : nullptr;
  double* const grow = GRID ? q.grow + (long long)pb * 2 * n : nullptr;
  unsigned* const cnt_part = GRID ? q.gcount + pb * 4 * QRG_LINE : nullptr;
  unsigned* const cnt_sum = cnt_part + QRG_LINE;
  unsigned* const cnt_top = cnt_sum + QRG_LINE;
  unsigned* const gtop = cnt_top + QRG_LINE;
  __shared__ unsigned s_warp[QRC_MAXT / 32], s_top;   // largest high word of a warp's loads, of my rows (read by every CTA)
  bool live = true;                         // GRID: no wait of this thread has run out
  if (!GRID) {                              // what shared memory does not hold
    double* g = q.W + pb * q.wst + rank * (q.wst / C);
    if (!mc_smem) {
      mc = g;
      g += qr_mc(k, C);
    }
    if (!tri_smem) {
      tri = g;
      g += qr_tri(k);
    }
    if (!w_smem) W = g;
  }
  auto cta_or_cluster_sync = [&]() {
    if (!GRID && C > 1)
      cluster.sync();
    else
      __syncthreads();
  };
  unsigned top = 0;
  if (q.cs == 1) {
    for (int e = tid; e < rows * n; e += nt) {
      const int li = e / n, j = e - li * n;
      const double v = A[(r0 + li) * q.rs + j];
      W[j * ld + li] = v;
      top = max(top, high_word(v));
    }
  } else {
    for (int e = tid; e < rows * n; e += nt) {
      const int j = e / rows, li = e - j * rows;
      const double v = A[(r0 + li) * q.rs + j * q.cs];
      W[j * ld + li] = v;
      top = max(top, high_word(v));
    }
  }
  top = __reduce_max_sync(0xffffffffu, top);
  if (lane == 0) s_warp[tid >> 5] = top;
  __syncthreads();
  // A matrix far from order one is brought there by an exact power of two (and
  // R back): a column whose squares underflow would get no reflector.
  top = __reduce_max_sync(0xffffffffu, lane < nt >> 5 ? s_warp[lane] : 0u);
  if (GRID) {
    if (tid == 0) {
      atomicMax(gtop, top);
      arrive_gpu(cnt_top);
      live = wait_arrivals(cnt_top, unsigned(C), q.flag, QRG_FIRST_WAIT);
      s_top = __ldcg(gtop);
    }
    __syncthreads();
    top = s_top;
  } else if (C > 1) {
    if (tid == 0) s_top = top;
    cluster.sync();
    top = __reduce_max_sync(0xffffffffu, lane < C ? *cluster.map_shared_rank(&s_top, lane) : 0u);
  }
  const int shift = order_one(top);                   // the same in every CTA
  if (shift != 0) {
    for (int e = tid; e < rows * n; e += nt) {
      const int c = e / rows, li = e - c * rows;
      W[c * ld + li] *= pow2(shift);
    }
    __syncthreads();
  }
  // One pass over the columns: the update with reflector column j (w from
  // wfin; j < 0: none) for c > jn, then the inner products with column jn
  // (final already) over rows >= jn for c > jn, over rows > jn otherwise.  The
  // owner of row jn publishes it.
  const int sh = lanes_log2, L = 1 << sh;
  auto pass = [&](int j, int jn, int b) {
    const double* xj = W + max(j, 0) * ld - r0;
    const double* xn = W + jn * ld - r0;
    const bool own = jn >= r0 && jn < r1;
    for (int t0 = tid - lane; t0 < n << sh; t0 += nt) {
      const int c = (t0 + lane) >> sh, l = lane & (L - 1);
      double acc = 0.0;
      double* wc = W + min(c, n - 1) * ld - r0;
      const int i0 = max(r0, c > jn ? jn : jn + 1) + l;
      if (c < n) {
        if (j >= 0 && c > jn)
          acc = qr_update_dot(wc, xj, xn, wfin[c], i0, L, r1);
        else
          acc = qr_dot(wc, xn, i0, L, r1);
      }
      for (int o = L >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (c < n && l == 0) {
        if (GRID)
          __stcg(gpart + c * C + rank, acc);
        else
          part[b * n + c] = acc;
        if (own) {
          if (GRID)
            __stcg(grow + b * n + c, wc[jn]);
          else
            rowv[b * n + c] = wc[jn];
        }
      }
    }
  };
  // Sum over the cluster of one partial sum, by four neighbouring lanes (l: which of them).
  auto cluster_sum = [&](double* slot, int l) {
    const double v0 = l < C ? *cluster.map_shared_rank(slot, l) : 0.0;
    const double v1 = l + 4 < C ? *cluster.map_shared_rank(slot, l + 4) : 0.0;
    const double v2 = l + 8 < C ? *cluster.map_shared_rank(slot, l + 8) : 0.0;
    const double v3 = l + 12 < C ? *cluster.map_shared_rank(slot, l + 12) : 0.0;
    double s = v0;
    if (C > 4) s += v1;
    if (C > 8) s = (s + v2) + v3;
    if (C > 2) s += __shfl_xor_sync(0xffffffffu, s, 2);
    return s + __shfl_xor_sync(0xffffffffu, s, 1);
  };
  pass(-1, 0, 0);
  for (int j = 0; j < k; ++j) {
    const int b = j & 1, owner = j / chunk;
    cta_or_cluster_sync();                            // column j: inner products and row j visible
    if (GRID) {
      // The next partial sums are written after these sums were awaited, the
      // next sums after every CTA has arrived with new partial sums, row j
      // alternates between two buffers: nothing is overwritten before its readers are done.
      if (tid == 0) arrive_gpu(cnt_part);
      for (int c = rank + (tid >> 5) * C; c < n; c += (nt >> 5) * C) {   // my columns, one warp each
        if (lane == 0 && live) live = wait_arrivals(cnt_part, unsigned(j + 1) * C, q.flag);
        __syncwarp();
        double v[QRG_MAXP / 32];
#pragma unroll
        for (int i = 0; i < QRG_MAXP / 32; ++i) v[i] = 32 * i + lane < C ? __ldcg(gpart + c * C + 32 * i + lane) : 0.0;
        double s = v[0];
#pragma unroll
        for (int i = 1; i < QRG_MAXP / 32; ++i)
          if (32 * i < C) s += v[i];
        s = warp_sum(s);
        if (lane == 0) {
          __stcg(gsum + c, s);
          arrive_gpu(cnt_sum);
        }
      }
      if (tid == nt - 32 && live) live = wait_arrivals(cnt_sum, unsigned(j + 1) * n, q.flag);
      __syncthreads();
    }
    // row j, local copy: the threads that do not sum start at the far end
    for (int c = nt - 1 - tid; c < n; c += nt)
      rowl[c] = GRID    ? __ldcg(grow + b * n + c)
                : C > 1 ? *cluster.map_shared_rank(rowv + b * n + c, owner)
                        : rowv[b * n + c];
    // sums over the CTAs, four threads per column (GRID: read by one), column j first
    constexpr int SPREAD = GRID ? 0 : 2;
    for (int t0 = tid - lane; t0 < n << SPREAD; t0 += nt) {
      const int ci = (t0 + lane) >> SPREAD, l = lane & ((1 << SPREAD) - 1);
      int c = min(ci, n - 1) + j;
      if (c >= n) c -= n;
      double* slot = part + b * n + c;
      double alpha = 0.0, s;
      if (GRID) {
        s = __ldcg(gsum + c);
        if (ci == 0) alpha = __ldcg(grow + b * n + j);
      } else if (C == 1) {
        s = *slot;
        if (ci == 0) alpha = rowv[b * n + j];
      } else {
        if (ci == 0) alpha = *cluster.map_shared_rank(rowv + b * n + j, owner);
        s = cluster_sum(slot, l);
      }
      if (ci >= n || l != 0) continue;
      if (ci > 0) {
        dsum[c] = s;
        continue;
      }
      // scalars of reflector j (thread 0): a column that is zero below the
      // diagonal, or whose squares underflow, has no reflector.  Tests on the
      // bits: an FP64 compare costs as much as an FMA.
      const double ss = fma(alpha, alpha, s);
      double y = 0.0, g = 0.0, h = 0.0;
      if (__double_as_longlong(s) << 1 != 0 && (__double2hiint(ss) >> 20 & 0x7ff) >= 23) {
        const double r = rsqrt(ss), e = fma(fabs(alpha), r, 1.0);
        g = r * r * __drcp_rn(e);
        y = copysign(r, alpha);
        h = copysign(ss * r, alpha);
      }
      ys[j] = y;
      gs[j] = g;
      nb[j] = h;
      vs[j] = alpha;
    }
    __syncthreads();
    const double y = ys[j], g = gs[j], h = nb[j];
    double* wj = W + j * ld - r0;
    if (j + 1 < n) {
      // column j+1 first: the pass takes inner products with its new values
      const double w1 = g * fma(h, rowl[j + 1], dsum[j + 1]);
      double* w1c = W + (j + 1) * ld - r0;
      for (int i = max(r0, j + 1) + tid; i < r1; i += nt) w1c[i] = fma(-w1, wj[i], w1c[i]);
    }
    for (int c = nt - 1 - tid; c < n; c += nt) {
      if (c > j + 1) {
        wfin[c] = g * fma(h, rowl[c], dsum[c]);
      } else if (c < j) {                             // x_c . x_j
        tri[j * (j - 1) / 2 + c] = fma(rowl[j] + h, rowl[c], dsum[c]);
      }
      if (j % C == rank && c <= j) mc[(j / C) * k + c] = rowl[c];
    }
    if (j >= r0 && j < r1 && __double_as_longlong(g) != 0) {   // row j of R
      for (int c = j + 1 + (nt - 1 - tid); c < n; c += nt) W[c * ld + (j - r0)] = -y * dsum[c];
      if (tid == 0) wj[j] = -h;
    }
    __syncthreads();
    if (j + 1 < k) pass(j, j + 1, 1 - b);
  }
  if (Ro) {
    for (int e = tid; e < rows * n; e += nt) {
      const int li = e / n, j = e - li * n, i = r0 + li;
      if (i >= k) continue;
      const double v = (j >= i) ? W[j * ld + li] : 0.0;
      Ro[(long long)i * n + j] = shift != 0 ? v * pow2(-shift) : v;
    }
  }
  for (int j = tid; j < k; j += nt) vs[j] = vs[j] + nb[j];
  __syncthreads();
  // X: zero above the diagonal (where R was), alpha - beta on it
  for (int e = tid; e < rows * k; e += nt) {
    const int c = e / rows, li = e - c * rows;
    if (r0 + li <= c) W[c * ld + li] = r0 + li == c ? vs[c] : 0.0;
  }
  // M, my columns, one warp each: T^{-1} M = X_1^T from the bottom up
  for (int cc = tid >> 5; cc < mcols; cc += nt >> 5) {
    const int c = rank + cc * C;
    if (c >= k) break;
    double* x = mc + cc * k;
    if (lane == 0) x[c] = vs[c];
    __syncwarp();
    for (int j = c; j >= 0; --j) {
      const double* t = tri + j * (j - 1) / 2;
      const double v = gs[j] * x[j];
      __syncwarp();
      for (int i = lane; i < j; i += 32) x[i] = fma(-t[i], v, x[i]);
      if (lane == 0) x[j] = v;
      __syncwarp();
    }
  }
  double* const gtri = GRID ? q.gtri + (long long)pb * qr_tri(k) : nullptr;
  if (GRID) {
    __syncthreads();
    for (int c = rank + (tid >> 5) * C; c < k; c += (nt >> 5) * C)
      for (int i = lane; i <= c; i += 32) __stcg(gtri + c * (c + 1) / 2 + i, mc[c / C * k + i]);
  }
  cta_or_cluster_sync();                              // every column of M visible
  if (GRID) {
    if (tid == 0) {
      arrive_gpu(cnt_part);
      if (live) wait_arrivals(cnt_part, unsigned(k + 1) * C, q.flag);
    }
    __syncthreads();
    for (int i = tid; i < qr_tri(k); i += nt) tri[i] = __ldcg(gtri + i);
  } else {
    for (int c = tid >> 5; c < k; c += nt >> 5) {
      double* src = mc + (c / C) * k;
      if (!mc_smem) {
        const double* g = src + (c % C - rank) * (q.wst / C);
        for (int i = lane; i <= c; i += 32) tri[c * (c + 1) / 2 + i] = __ldcg(g + i);
        continue;
      }
      if (C > 1) src = cluster.map_shared_rank(src, c % C);
      for (int i = lane; i <= c; i += 32) tri[c * (c + 1) / 2 + i] = src[i];
    }
  }
  __syncthreads();
  // Q = E - X M on my rows, one entry per thread at a time, lanes along rows
  for (int e = tid; e < rows * k; e += nt) {
    const int c = e / rows, li = e - c * rows;
    const double* t = tri + c * (c + 1) / 2;
    const double* x = W + li;
    double acc = r0 + li == c ? 1.0 : 0.0;
    int a = 0;
    for (; a + 3 <= c; a += 4) {
      const double x0 = x[a * ld], x1 = x[(a + 1) * ld], x2 = x[(a + 2) * ld], x3 = x[(a + 3) * ld];
      const double t0 = t[a], t1 = t[a + 1], t2 = t[a + 2], t3 = t[a + 3];
      acc = fma(-x0, t0, acc);
      acc = fma(-x1, t1, acc);
      acc = fma(-x2, t2, acc);
      acc = fma(-x3, t3, acc);
    }
    for (; a <= c; ++a) acc = fma(-x[a * ld], t[a], acc);
    Qo[(r0 + li) * q.qrs + c * q.qcs] = acc;
  }
  if (!GRID && C > 1) cluster.sync();   // no CTA leaves while others may still read its shared memory
}

struct SvdArgs {
  int p, q;          // G is p x q (p >= q), G(i, j) = A[i*rs + j*cs]
  TP A;              // per problem
  long long rs, cs;
  int trans;         // 1: the SVD of G^T is wanted, else that of G
  double* work;      // rows of G and V where shared memory does not hold them
  long long wst;     // doubles of work per problem
  int kk;
  TP US;             // (trans ? q : p) x kk row-major
  TP Vt;             // kk x (trans ? p : q) row-major
  int* flag;
  int max_sweeps;    // sweep cap (PEPS_ECONVERGE when reached)
};

// ---------------------------------------------------------------------------
// One-sided Jacobi (Hestenes) on a thread-block cluster of C = 1-16 CTAs: the
// rows of the working matrix G (p x q) and of V (q x q) are split over the
// CTAs and kept in shared memory where they fit.  A round of the round-robin
// schedule rotates q / 2 disjoint column pairs.
//
// What bounds it: the FP64 pipe (64 clocks per warp instruction and SM
// quarter) and, for the matrices of a boundary fit, the chain of one round --
// inner products, cluster barrier, sums, rotation scalars, rotation.  So
//   * one inner product per pair and round: squared column norms are exact at
//     the start of a sweep and follow the rotations inside it
//     (alpha' = alpha - t gamma, beta' = beta + t gamma); a sweep without
//     rotations, the one that ends the iteration, has tested exact norms;
//   * the angle's tangent t = g / (|d| + sqrt(d^2 + g^2)), d = beta - alpha and
//     g = 2 gamma, from one reciprocal root and one reciprocal, and its cosine
//     from another root (taken from FP32 values, t leaves 1e-7 of the inner
//     product to the next sweep: 3 to 10% faster, and less orthogonal where no
//     further sweep came, graded 5x40 3e-14 against 9e-16);
//   * scaled rotations (fast Givens): columns are kept as G = G' diag(d), and
//     a rotation is one FMA per element, g_a' -= t d_b / d_a g_b',
//     g_b' += t d_a / d_b g_a' (old values), d *= c; d goes back into the
//     columns every 64 rounds;
//   * partial sums stay in their CTA and are read after the barrier.
// Same threshold, ordering and output rules as LAPACK's one-sided Jacobi: a
// pair is orthogonal once |gamma| <= tol sqrt(alpha beta) with
// tol = 4 p eps (rounding alone leaves p eps).
// Measured (us; before: plain rotations and three inner products per pair and
// round, rows in global memory; now: with the preconditioning of svd_trunc):
// random 16x16 582 -> 360, 32 of 64x64 6193 -> 3285, 180x180 42224 -> 12897,
// graded 180x180 27740 -> 8278.  A round of 180x180 takes about 14,000 clocks:
// the rotations half of it, the scalars a third.
// ---------------------------------------------------------------------------
constexpr int SVC_MAXT = 512;
constexpr int SVC_RESCALE = 64;

__host__ __device__ inline long long svd_head(int q) {
  const long long npair = (q + 1) / 2;
  return 4 * npair + 3LL * q + 2 * npair + q + (q + 1) / 2 + 2;
}
__host__ __device__ inline int svd_ld(int rows) { return rows | 1; }   // odd: no bank conflicts across columns

// Slots (a, b) of pair pr in a round of the circle schedule over qq slots: slot 0 fixed, the others rotate.
__device__ __forceinline__ void jacobi_pair(int pr, int round, int qq, int& a, int& b) {
  const int w = qq - 1;
  int u = pr - 1 + round, v = qq - 2 - pr + round;
  u -= u >= w ? w : 0;
  v -= v >= w ? w : 0;
  a = pr == 0 ? 0 : 1 + u;
  b = 1 + v;
  if (a > b) {
    const int t = a;
    a = b;
    b = t;
  }
}

// x * 2^k by the exponent bits; 0 below the normal range.
__device__ __forceinline__ double scale2(double x, int k) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  if (ex == 0 || ex + k <= 0) return 0.0;
  return __hiloint2double(hi + k * (1 << 20), __double2loint(x));
}

__global__ void __launch_bounds__(SVC_MAXT) k_svd_cluster(const SvdArgs s, int head_smem, int rows_smem, int lanes_log2) {
  extern __shared__ double ssm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = int(cluster.num_blocks()), rank = int(cluster.block_rank());
  const int pb = blockIdx.x / C;
  const int p = s.p, q = s.q, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int qq = q + (q & 1), npair = qq / 2;
  const int cp = (p + C - 1) / C, cv = (q + C - 1) / C;
  const int g0 = min(p, rank * cp), gr = min(p, g0 + cp) - g0;            // my rows of G
  const int v0 = min(q, rank * cv), vr = min(q, v0 + cv) - v0;            // my rows of V
  const int ld = svd_ld(cp + cv);             // a column: my rows of G, then (at cp) my rows of V
  double* const work = s.work + pb * s.wst + rank * (s.wst / C);
  double* part = head_smem ? ssm : work;      // [2][2 npair] my partial sums (read by every CTA)
  double* al = part + 4 * npair;              // [q] squared norms
  double* ds = al + q;                        // [q] column scales
  double* es = ds + q;                        // [q] their reciprocals
  double* ta = es + q;                        // [npair] this round's rotations: t d_b / d_a
  double* tb = ta + npair;                    // [npair] t d_a / d_b
  double* nrm = tb + npair;                   // [q]
  int* order = reinterpret_cast<int*>(nrm + q);   // [q]
  __shared__ int s_rot;
  __shared__ unsigned s_top, s_all;
  double* G = rows_smem ? ssm + svd_head(q) : work + (head_smem ? 0 : svd_head(q));
  const double* A = s.A.d(pb);
  const bool rows_first = s.rs < s.cs;
  if (tid == 0) s_top = s_all = 0;
  __syncthreads();
  unsigned top = 0;
  for (long long e = tid; e < (long long)gr * q; e += nt) {
    const int j = int(rows_first ? e / gr : e % q), li = int(rows_first ? e % gr : e / q);
    const double v = A[(g0 + li) * s.rs + j * s.cs];
    G[(long long)j * ld + li] = v;
    top = max(top, high_word(v));
  }
  top = __reduce_max_sync(0xffffffffu, top);
  if (lane == 0) atomicMax(&s_top, top);
  for (int j = warp; j < q; j += nw)
    for (int li = lane; li < vr; li += 32) G[(long long)j * ld + cp + li] = (v0 + li == j) ? 1.0 : 0.0;
  for (int j = tid; j < q; j += nt) {
    ds[j] = 1.0;
    es[j] = 1.0;
  }
  auto cta_or_cluster_sync = [&]() {
    if (C > 1)
      cluster.sync();
    else
      __syncthreads();
  };
  auto sum_parts = [&](double* slot) { return C > 1 ? remote_sum(cluster, slot, C) : *slot; };
  // A matrix far from order one is brought there by an exact power of two (and
  // its singular values back): the norms are squares and the rotation test
  // compares their products.
  cta_or_cluster_sync();
  if (tid < C) atomicMax(&s_all, C > 1 ? *cluster.map_shared_rank(&s_top, tid) : s_top);
  __syncthreads();
  const int shift = order_one(s_all);
  if (shift != 0)
    for (int j = warp; j < q; j += nw)
      for (int li = lane; li < gr; li += 32) G[(long long)j * ld + li] *= pow2(shift);
  const double unscale = pow2(-shift);
  // the scales into the columns (after a barrier; followed by one)
  auto rescale = [&]() {
    for (int j = warp; j < q; j += nw) {
      const double d = ds[j];
      double* x = G + (long long)j * ld;
      for (int li = lane; li < cp + vr; li += 32)
        if (li < gr || li >= cp) x[li] *= d;
    }
    __syncthreads();
    for (int j = tid; j < q; j += nt) {
      ds[j] = 1.0;
      es[j] = 1.0;
    }
  };
  int buf = 0;   // double-buffer index of part: advances with every exchange
  // exact squared norms of the columns into al
  auto norms = [&]() {
    for (int j = warp; j < q; j += nw) {
      const double* x = G + (long long)j * ld;
      double v = 0.0;
      for (int li = lane; li < gr; li += 32) v = fma(x[li], x[li], v);
      v = warp_sum(v);
      if (lane == 0) part[buf * 2 * npair + j] = v;
    }
    cta_or_cluster_sync();
    for (int j = tid; j < q; j += nt) al[j] = sum_parts(part + buf * 2 * npair + j);
    buf ^= 1;
    __syncthreads();
  };
  const double tol = fmax(1e-15, 4.0 * double(p) * 2.220446049250313e-16);
  const int sh = lanes_log2, L = 1 << sh;   // threads per inner product
  const int W = cp + vr > 16 ? 32 : (cp + vr > 8 ? 16 : 8);   // lanes per rotated pair
  __syncthreads();
  int sweep = 0;
  for (; sweep < s.max_sweeps; ++sweep) {
    rescale();
    if (tid == 0) s_rot = 0;
    __syncthreads();
    norms();
    int rotated = 0;
    for (int round = 0; round < qq - 1; ++round) {
      if (round % SVC_RESCALE == SVC_RESCALE - 1) {
        rescale();
        __syncthreads();
      }
      for (int t0 = tid - lane; t0 < npair << sh; t0 += nt) {
        const int pr = (t0 + lane) >> sh, l = lane & (L - 1);
        int a, b;
        jacobi_pair(pr, round, qq, a, b);
        double ga = 0.0;
        if (pr < npair && b < q) {
          const double* xa = G + (long long)a * ld;
          const double* xb = G + (long long)b * ld;
#pragma unroll 4
          for (int li = l; li < gr; li += L) ga = fma(xa[li], xb[li], ga);
        }
        for (int o = L >> 1; o > 0; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
        if (pr < npair && l == 0) part[buf * 2 * npair + pr] = ga;
      }
      cta_or_cluster_sync();
      for (int pr = tid; pr < npair; pr += nt) {
        int a, b;
        jacobi_pair(pr, round, qq, a, b);
        double x = 0.0, y = 0.0;
        if (b < q) {
          const double da = ds[a], db = ds[b], A2 = al[a], B2 = al[b];
          const double ga = sum_parts(part + buf * 2 * npair + pr) * da * db;
          // gamma^2 > tol^2 alpha beta, tested on the sign of the difference,
          // everything scaled by the larger norm's exponent (fourth powers of
          // a small column would underflow); no rotation where a norm is no
          // finite number
          const double dl = B2 - A2;
          const int k = 1023 - ((max(__double2hiint(A2), __double2hiint(B2)) >> 20) & 0x7ff);
          const double g1 = scale2(ga, k);
          const double over = fma(-(tol * scale2(A2, k)), tol * scale2(B2, k), g1 * g1);
          if (k > -1024 && (__double2hiint(over) > 0 || (__double2hiint(over) == 0 && __double2loint(over) != 0))) {
            const double d1 = scale2(dl, k), g2 = d1 >= 0.0 ? 2.0 * g1 : -2.0 * g1;
            const double r = rsqrt(fma(d1, d1, g2 * g2)), t = g2 * r * __drcp_rn(fma(fabs(d1), r, 1.0));
            const double w = fma(t, t, 1.0), c = rsqrt(w), ic = w * c;
            x = t * (db * es[a]);
            y = t * (da * es[b]);
            al[a] = fma(-t, ga, A2);
            al[b] = fma(t, ga, B2);
            ds[a] = da * c;
            ds[b] = db * c;
            es[a] *= ic;
            es[b] *= ic;
            rotated = 1;
          }
        }
        ta[pr] = x;
        tb[pr] = y;
      }
      buf ^= 1;
      __syncthreads();
      // rotate my rows of G and V
      const int sub = lane / W, per = 32 / W;
      for (int pr = warp * per + sub; pr < npair; pr += nw * per) {
        const double x = ta[pr], y = tb[pr];
        if (__double_as_longlong(x) << 1 == 0 && __double_as_longlong(y) << 1 == 0) continue;
        int a, b;
        jacobi_pair(pr, round, qq, a, b);
        double* xa = G + (long long)a * ld;
        double* xb = G + (long long)b * ld;
        for (int li = lane & (W - 1); li < cp + vr; li += W) {
          if (li >= gr && li < cp) continue;
          const double u = xa[li], v = xb[li];
          xa[li] = fma(-x, v, u);
          xb[li] = fma(y, u, v);
        }
      }
      __syncthreads();
    }
    if (rotated) s_rot = 1;   // benign race: every writer stores 1
    __syncthreads();
    const int rot = s_rot;
    __syncthreads();
    if (!rot) break;          // identical in every CTA (same sums, same decisions)
  }
  if (sweep >= s.max_sweeps && tid == 0 && rank == 0) atomicOr(s.flag, FLAG_SVD_NOCONV);
  // column norms of G over all rows, then a stable descending order
  rescale();
  __syncthreads();
  norms();
  for (int j = tid; j < q; j += nt) nrm[j] = sqrt(al[j]);
  __syncthreads();
  for (int j = tid; j < q; j += nt) {
    const double vj = nrm[j];
    int r = 0;
    for (int i = 0; i < q; ++i) {
      const double vi = nrm[i];
      r += (vi > vj) || (vi == vj && i < j);
    }
    order[r] = j;
  }
  __syncthreads();
  const int kk = s.kk;
  double* const US = s.US.d(pb);
  double* const Vt = s.Vt.d(pb);
  const int n = s.trans ? p : q;
  // G0 V = G: G0 = G V^T, G0^T = V G^T
  if (!s.trans) {
    // US[i][r] = G(i, order[r]) for my G rows; Vt[r][j] = V(j, order[r]) for my V rows
    for (int e = tid; e < gr * kk; e += nt) {
      const int li = e / kk, r = e % kk;
      US[(long long)(g0 + li) * kk + r] = (r < q) ? G[(long long)order[r] * ld + li] * unscale : 0.0;
    }
    for (int e = tid; e < vr * kk; e += nt) {
      const int r = e / vr, li = e % vr;
      Vt[(long long)r * n + (v0 + li)] = (r < q) ? G[(long long)order[r] * ld + cp + li] : 0.0;
    }
  } else {
    // US[i][r] = V(i, order[r]) * nrm for my V rows; Vt[r][j] = G(j, order[r]) / nrm for my G rows
    for (int e = tid; e < vr * kk; e += nt) {
      const int li = e / kk, r = e % kk;
      US[(long long)(v0 + li) * kk + r] = (r < q) ? G[(long long)order[r] * ld + cp + li] * (nrm[order[r]] * unscale) : 0.0;
    }
    for (int e = tid; e < gr * kk; e += nt) {
      const int r = e / gr, li = e % gr;
      const double nr = (r < q) ? nrm[order[r]] : 0.0;
      Vt[(long long)r * n + (g0 + li)] = (r < q && nr > 0.0) ? G[(long long)order[r] * ld + li] / nr : 0.0;
    }
  }
  if (C > 1) cluster.sync();   // no CTA leaves while others may still read its shared memory
}

}  // namespace

namespace {
// Clusters of c CTAs of `kern` with `smem` bytes of dynamic shared memory per
// CTA that run at once; 0 if they cannot be launched.  Cached per kernel,
// device, threads, size (in 4 KB steps) and c; sets the kernel's attributes.
template <class K>
int active_clusters(K kern, int threads, size_t smem, int c) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, int, int, size_t, int>, int> cache;
  static std::map<std::pair<const void*, int>, bool> attrs;
  int dev = 0;
  PEPS_CUDA(cudaGetDevice(&dev));
  const void* id = reinterpret_cast<const void*>(kern);
  const size_t key = (smem + 4095) / 4096 * 4096;
  std::lock_guard<std::mutex> g(mu);
  const auto k = std::make_tuple(id, dev, threads, key, c);
  const auto it = cache.find(k);
  if (it != cache.end()) return it->second;
  auto at_it = attrs.find({id, dev});
  if (at_it == attrs.end()) {
    const bool ok =
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024) == cudaSuccess;
    cudaGetLastError();
    at_it = attrs.emplace(std::make_pair(id, dev), ok).first;
  }
  int n = 0;
  if (at_it->second) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = key;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
    if (std::getenv("PEPS_VERBOSE"))
      std::fprintf(stderr, "[peps] cluster %d threads %d smem %zu: %s, %d active clusters\n", c, threads, key,
                   cudaGetErrorString(e), n);
    cudaGetLastError();
    if (e != cudaSuccess) n = 0;
  }
  cache[k] = n;
  return n;
}

}  // namespace

namespace {

// Largest dynamic shared memory of the cluster kernels (227 KB per CTA on sm_103).
constexpr size_t kQrSmemMax = 224 * 1024;

int qr_ld(int m, int c) { return (((m + c - 1) / c) + 7) / 8 * 8 + 4; }   // = 4 mod 8: no bank conflicts
size_t qr_head_bytes(int m, int n) { return sizeof(double) * size_t(qr_head(n, std::min(m, n))); }
size_t qr_mc_bytes(int m, int n, int c) { return sizeof(double) * size_t(qr_mc(std::min(m, n), c)); }
// Shared memory per CTA of an m x n factorisation with its rows split over c
// CTAs and kept there (the columns of M and the triangle too where they still fit).
size_t qr_smem(int m, int n, int c) {
  return qr_head_bytes(m, n) + sizeof(double) * size_t(qr_ld(m, c)) * size_t(n);
}
// One warp per SM quarter at least; four threads per column while that is no more than 512.
int qr_threads(int n) { return std::max(128, std::min(QRC_MAXT, (4 * n + 31) / 32 * 32)); }

int qr_lanes_log2(int n) { return n > 16 ? 2 : n > 8 ? 3 : n > 4 ? 4 : 5; }

size_t qr_tri_bytes(int m, int n) { return sizeof(double) * size_t(qr_tri(std::min(m, n))); }

// A launch on clusters of c CTAs.
struct ClusterLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  ClusterLaunch(int ctas, int threads, size_t smem, int c, cudaStream_t st) {
    cfg.gridDim = dim3(ctas, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
};

// Estimated clocks of np factorisations on clusters of c CTAs, fitted to
// measured times of shapes from 16x16 to 2304x64 on 1 to 16 CTAs (within 20%;
// 180x180 to 676x338 on 16 come out so as well):
// a column costs its barriers, sums and scalars, its share of the back
// substitutions, and the FP64 pipe 24 clocks per warp instruction and SM (19
// at best), two per row and column; the pass leaves a quarter of that idle
// where a column's warp has an SM quarter to itself, and a triangle in global
// memory costs a fifth more.  Clusters beyond those that run at once wait:
// only a few of 16 CTAs do (8192x128 in 8 leaves takes 3.7 ms, in 4 2.9 ms).
double qr_clocks(int m, int n, int c, int np) {
  const double k = std::min(m, n), rows = std::ceil(double(m) / c);
  const double warps = qr_threads(n) / 32;
  const size_t rows_b = qr_smem(m, n, c), mc_b = rows_b + qr_mc_bytes(m, n, c), all_b = mc_b + qr_tri_bytes(m, n);
  const bool tri = all_b <= kQrSmemMax;
  const int at_once = active_clusters(k_qr_cluster<false>, qr_threads(n),
                                      tri ? all_b : mc_b <= kQrSmemMax ? mc_b : rows_b, c);
  if (at_once == 0) return 1e300;
  const double step = (c == 1 ? 3800.0 : 5600.0) + 180.0 * std::ceil(std::ceil(k / c) / warps);
  const double fp = 24.0 * rows * 2.0 * n / 32.0 * (n < 64 ? 1.3 : 1.0);
  const double waves = std::ceil(double(np) / at_once);
  const double per_sm = std::ceil(std::min<double>(np, at_once) * c / num_sms());
  return 10000.0 + waves * k * (step + per_sm * fp) * (tri ? 1.0 : 1.2);
}

// dst[b][i*qrs + j*qcs] = src[b][i*n + j]
__global__ void k_copy_strided(const TP src, const TP dst, int m, int n, long long qrs, long long qcs) {
  const double* s = src.d(blockIdx.y);
  double* d = dst.d(blockIdx.y);
  const long long total = (long long)m * n;
  const bool rows_fast = qrs < qcs;   // write along whichever index is contiguous in dst
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long i = rows_fast ? e % m : e / n, j = rows_fast ? e / m : e % n;
    d[i * qrs + j * qcs] = s[i * n + j];
  }
}

// Largest c (a power of two) up to cmax whose rows fit in shared memory with
// the least estimated time; 0 if none fits.
int qr_best_cluster(int m, int n, int np, int cmax, double* clocks) {
  int best = 0;
  *clocks = 1e300;
  for (int c = 1; c <= cmax; c *= 2) {
    if (qr_smem(m, n, c) > kQrSmemMax) continue;
    const double t = qr_clocks(m, n, c, np);
    if (t < *clocks * 1.02) {   // a tie goes to more CTAs
      *clocks = t;
      best = c;
    }
  }
  return best;
}

// How one factorisation runs on k_qr_cluster: cluster size (0: k_qr_house),
// what is in shared memory, and how much of it.
struct QrPlan {
  int C = 0;
  bool w_smem = false, mc_smem = false, tri_smem = false;
  size_t bytes = 0;
};

// The cluster size with the least estimated time among those whose rows fit in
// shared memory; rows in global memory, on the largest cluster of 32 rows per
// CTA or more that still holds the partial sums, where none fits.  Kept per
// shape (a few integers each): the choice costs several occupancy look-ups.
QrPlan qr_plan(int m, int n, int np, int qr_cmax) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, int, int>, QrPlan> cache;
  int dev = 0;
  PEPS_CUDA(cudaGetDevice(&dev));
  const auto key = std::make_tuple(dev, m, n, np, qr_cmax);
  {
    std::lock_guard<std::mutex> g(mu);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
  }
  const int lim = qr_cmax > 0 ? std::min(qr_cmax, 16) : 16;
  double clocks;
  QrPlan p;
  p.C = qr_best_cluster(m, n, np, lim, &clocks);
  p.w_smem = p.C > 0;
  // (entries are indexed with 32 bits)
  auto holds = [&](int c) { return qr_head_bytes(m, n) <= kQrSmemMax && (long long)qr_ld(m, c) * n < (1LL << 31); };
  if (!p.w_smem)
    for (int c = 1; c <= std::min(lim, std::max(1, m / 32)); c *= 2)
      if (holds(c)) p.C = c;
  // rows, columns of M and triangle: each in shared memory where it still fits
  auto settle = [&] {
    auto add = [&](size_t b) {
      const bool fits = p.bytes + b <= kQrSmemMax;
      if (fits) p.bytes += b;
      return fits;
    };
    p.bytes = p.w_smem ? qr_smem(m, n, p.C) : qr_head_bytes(m, n);
    p.mc_smem = add(qr_mc_bytes(m, n, p.C));
    p.tri_smem = add(qr_tri_bytes(m, n));
  };
  while (p.C > 0) {
    settle();
    if (active_clusters(k_qr_cluster<false>, qr_threads(n), p.bytes, p.C) > 0) break;
    p.C /= 2;   // clusters of this size cannot be launched here
    p.w_smem = p.C > 0 && qr_smem(m, n, p.C) <= kQrSmemMax;
    if (p.C > 0 && !holds(p.C)) p.C = 0;
  }
  std::lock_guard<std::mutex> g(mu);
  return cache.emplace(key, p).first->second;
}

// Leaves of a tall-skinny QR: a power of two L >= 2 that divides m, leaves of
// at least n rows (and 32 per CTA of a 16-CTA cluster) that fit in shared
// memory; the one with the least estimated time, 0 if none fits.
int tsqr_leaves(int m, int n, int np, double* clocks) {
  int best = 0;
  *clocks = 1e300;
  for (int L = 2; L <= 16; L *= 2) {
    if (m % L || np * L > MAXB) break;
    const int ml = m / L;
    if (ml < n || ml < 16 * 32) break;
    double t1, t2;
    if (!qr_best_cluster(ml, n, np * L, 16, &t1) || !qr_best_cluster(L * n, n, np, 16, &t2)) continue;
    const double t = t1 + t2 + 2.0 * double(np) * m * n * n / num_sms() / 3.0 + 20000.0;   // + the Q combine
    if (t < *clocks) {
      *clocks = t;
      best = L;
    }
  }
  return best;
}

// How a matrix with m >= 1024 rows is factored: by P CTAs that are no cluster
// (P > 0), in L leaves (L > 0), or like any other.
struct TallPlan {
  int L = 0;
  int P = 0;
  size_t bytes = 0;
};

// k_qr_cluster<true> on every SM (P = 0: it does not fit, rows and triangle in
// shared memory), with qr_clocks' terms and two waits for the other CTAs in a
// column: 10500 clocks where one cluster has 5600 (the shapes above come out
// within 15%).
TallPlan qr_grid(int m, int n, int np, double* clocks) {
  TallPlan p;
  *clocks = 1e300;
  const int c = std::min(QRG_MAXP, num_sms() / np);
  if (c < 2) return p;
  const size_t b = qr_smem(m, n, c) + qr_mc_bytes(m, n, c) + qr_tri_bytes(m, n);
  if (b > kQrSmemMax || active_clusters(k_qr_cluster<true>, qr_threads(n), b, 1) < c * np) return p;
  const double rows = std::ceil(double(m) / c);
  *clocks = 14000.0 + n * (10500.0 + 24.0 * rows * 2.0 * n / 32.0 * (n < 64 ? 1.3 : 1.0));
  p.P = c;
  p.bytes = b;
  return p;
}

// Kept per shape.
TallPlan tall_plan(int m, int n, int np, bool whole) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, int, bool>, TallPlan> cache;
  int dev = 0;
  PEPS_CUDA(cudaGetDevice(&dev));
  const auto key = std::make_tuple(dev, m, n, np, whole);
  std::lock_guard<std::mutex> g(mu);
  const auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  double direct, leaves, grid = 1e300;
  qr_best_cluster(m, n, np, 16, &direct);
  TallPlan p, w;
  p.L = tsqr_leaves(m, n, np, &leaves);
  if (whole) w = qr_grid(m, n, np, &grid);
  // the estimates are no better than a tenth
  if (!(p.L > 1 && leaves < 0.9 * direct)) p.L = 0;
  if (w.P > 0 && grid < 0.9 * (p.L ? leaves : direct)) p = w;
  return cache.emplace(key, p).first->second;
}

}  // namespace

void qr_direct(Ctx& cx, int m, int n, const TP& A, long long rs, long long cs, const TP& Q, long long qrs,
               long long qcs, const TP& R, double counted_flops);

// Algorithmic flops of one thin QR (the count used for rooflines): 2mn^2 - 2n^3/3.
double qr_flops(int m, int n) {
  const double k = std::min(m, n);
  return 2.0 * m * double(n) * k - 2.0 / 3.0 * k * k * k;
}

// Tall-skinny QR (Demmel, Grigori, Hoemmen & Langou): the rows are split into
// L leaves factored together as one batched cluster QR (rows in shared
// memory), the L stacked R factors are factored once more, and each leaf's Q
// is its own Q times its block of the second Q (one batched FP64 GEMM).  Q is
// the Householder Q of A up to the sign of each column; R likewise.
void qr_tsqr(Ctx& cx, int m, int n, int L, const TP& A, long long rs, long long cs, const TP& Q, long long qrs,
             long long qcs, const TP& R, int np) {
  const int ml = m / L;
  const size_t qn = size_t(ml) * n, rn = size_t(n) * n;
  double* qleaf = cx.ws->dalloc(size_t(np) * L * qn);
  double* rstack = cx.ws->dalloc(size_t(np) * L * rn);
  double* qtree = cx.ws->dalloc(size_t(np) * L * rn);
  TP Al, Ql, Rl, Bt, Ct, At, Qt;
  Al.n = Ql.n = Rl.n = Bt.n = Ct.n = np * L;
  At.n = Qt.n = np;
  const bool direct_out = (qrs == n && qcs == 1);
  double* qout = direct_out ? nullptr : cx.ws->dalloc(size_t(np) * m * n);
  for (int b = 0; b < np; ++b) {
    At.p[b] = rstack + size_t(b) * L * rn;
    Qt.p[b] = qtree + size_t(b) * L * rn;
    for (int i = 0; i < L; ++i) {
      const int j = b * L + i;
      Al.p[j] = A.d(b) + (long long)i * ml * rs;
      Ql.p[j] = qleaf + size_t(j) * qn;
      Rl.p[j] = rstack + size_t(j) * rn;
      Bt.p[j] = qtree + size_t(j) * rn;
      Ct.p[j] = direct_out ? Q.d(b) + size_t(i) * qn : qout + size_t(b) * m * n + size_t(i) * qn;
    }
  }
  // The three steps are charged to the QR class, with the algorithmic flops of
  // the whole factorisation counted once.
  qr_direct(cx, ml, n, Al, rs, cs, Ql, n, 1, Rl, qr_flops(m, n) * np);
  qr_direct(cx, L * n, n, At, n, 1, Qt, n, 1, R, 0.0);
  cx.f64_class = K_QR;
  cx.f64_flops = false;
  ein(cx, "ik,kj->ij", Ql, {ml, n}, Bt, {n, n}, Ct);
  cx.f64_class = -1;
  cx.f64_flops = true;
  if (!direct_out) {
    TP src;
    src.n = np;
    for (int b = 0; b < np; ++b) src.p[b] = qout + size_t(b) * m * n;
    Launch Lc(K_QR, cx.st);
    k_copy_strided<<<dim3(unsigned(std::min<long long>(4096, ((long long)m * n + 255) / 256)), np), 256, 0, cx.st>>>(
        src, Q.all(np), m, n, qrs, qcs);
    PEPS_CHECK_LAUNCH();
  }
}

// One QR on the whole device.  Cooperative: its CTAs wait for one another and
// have to be resident together.
void qr_whole(Ctx& cx, int m, int n, const TallPlan& p, const TP& A, long long rs, long long cs, const TP& Q,
              long long qrs, long long qcs, const TP& R, int np) {
  QrArgs a;
  std::memset(static_cast<void*>(&a), 0, sizeof(a));
  a.m = m;
  a.n = n;
  a.A = A.all(np);
  a.rs = rs;
  a.cs = cs;
  a.Q = Q.all(np);
  a.qrs = qrs;
  a.qcs = qcs;
  a.R = R.all(np);
  a.P = p.P;
  a.flag = cx.flag;
  const size_t b = size_t(np), count = b * 2 * QRG_LINE, part = b * n * p.P, tri = b * qr_tri(n);
  double* w = cx.scratch(count + part + tri + b * 3 * n);
  a.gcount = reinterpret_cast<unsigned*>(w);
  a.gpart = w + count;
  a.gtri = a.gpart + part;
  a.gsum = a.gtri + tri;
  a.grow = a.gsum + b * n;
  PEPS_CUDA(cudaMemsetAsync(a.gcount, 0, count * sizeof(double), cx.st));
  if (std::getenv("PEPS_VERBOSE")) std::fprintf(stderr, "[peps] qr %dx%d x%d: %d CTAs\n", m, n, np, p.P);
  Launch L(K_QR, cx.st, qr_flops(m, n) * np, 0);
  int w_smem = 1, mc_smem = 1, tri_smem = 1, ld = qr_ld(m, p.P), lanes = qr_lanes_log2(n);
  void* args[] = {&a, &w_smem, &mc_smem, &tri_smem, &ld, &lanes};
  PEPS_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_qr_cluster<true>), dim3(p.P * np),
                                        dim3(qr_threads(n)), args, p.bytes, cx.st));
  PEPS_CHECK_LAUNCH();
}

void qr_thin(Ctx& cx, int m, int n, const TP& A, long long rs, long long cs, const TP& Q, long long qrs,
             long long qcs, const TP& R) {
  PEPS_REQUIRE(m > 0 && n > 0, "qr of an empty matrix");
  const int np = problems({&A, &Q, &R});
  PEPS_REQUIRE(!A.null() && Q.n == np && (R.null() || R.n == np), "internal: qr operands");
  // Tall-skinny QR over leaves on more SMs than one cluster has, where the rows
  // do not fit in the shared memory of one cluster or the leaves are estimated
  // to be faster.
  if (m >= 1024 && m >= n && cx.qr_cmax <= 0) {
    const TallPlan p = tall_plan(m, n, np, cx.qr_whole);
    if (p.L > 0) {
      qr_tsqr(cx, m, n, p.L, A, rs, cs, Q, qrs, qcs, R, np);
      return;
    }
    if (p.P > 0) {
      qr_whole(cx, m, n, p, A, rs, cs, Q, qrs, qcs, R, np);
      return;
    }
  }
  qr_direct(cx, m, n, A, rs, cs, Q, qrs, qcs, R, qr_flops(m, n) * np);
}

void qr_direct(Ctx& cx, int m, int n, const TP& A, long long rs, long long cs, const TP& Q, long long qrs,
               long long qcs, const TP& R, double counted_flops) {
  const int np = problems({&A, &Q, &R});
  const int k = std::min(m, n);
  const QrPlan pl = qr_plan(m, n, np, cx.qr_cmax);
  const int C = pl.C;
  if (std::getenv("PEPS_VERBOSE")) std::fprintf(stderr, "[peps] qr %dx%d x%d: cluster %d\n", m, n, np, C);
  QrArgs a;
  std::memset(static_cast<void*>(&a), 0, sizeof(a));
  a.m = m;
  a.n = n;
  a.A = A.all(np);
  a.rs = rs;
  a.cs = cs;
  a.Q = Q.all(np);
  a.qrs = qrs;
  a.qcs = qcs;
  a.R = R.all(np);
  const int ld = qr_ld(m, std::max(C, 1));
  const long long tri = qr_tri(k);
  if (C == 0) {
    a.wst = (long long)m * n;
    a.qst = (long long)m * k;
    a.tst = k;
  } else if (!pl.w_smem || !pl.mc_smem || !pl.tri_smem) {
    a.wst = C * ((pl.mc_smem ? 0 : qr_mc(k, C)) + (pl.tri_smem ? 0 : tri) + (pl.w_smem ? 0 : (long long)ld * n));
  }
  if (a.wst) {
    double* w = cx.scratch(size_t(np) * (a.wst + a.qst + a.tst) + 64);
    a.W = w;
    a.Qw = w + size_t(np) * a.wst;
    a.tau = a.Qw + size_t(np) * a.qst;
  }
  Launch L(K_QR, cx.st, counted_flops, 0);
  if (C == 0) {
    k_qr_house<<<np, QR_THREADS, 0, cx.st>>>(a);
  } else {
    ClusterLaunch c(C * np, qr_threads(n), pl.bytes, C, cx.st);
    PEPS_CUDA(cudaLaunchKernelEx(&c.cfg, k_qr_cluster<false>, a, pl.w_smem ? 1 : 0, pl.mc_smem ? 1 : 0,
                                 pl.tri_smem ? 1 : 0, ld, qr_lanes_log2(n)));
  }
  PEPS_CHECK_LAUNCH();
}

// Jacobi SVD of G (or G^T), see SvdArgs.
void svd_jacobi(Ctx& cx, int p, int q, const TP& A, long long rs, long long cs, int trans, int kk, const TP& US,
                const TP& Vt, int np) {
  SvdArgs s;
  std::memset(static_cast<void*>(&s), 0, sizeof(s));
  s.p = p;
  s.q = q;
  s.A = A.all(np);
  s.rs = rs;
  s.cs = cs;
  s.trans = trans;
  s.kk = kk;
  s.US = US.all(np);
  s.Vt = Vt.all(np);
  s.flag = cx.flag;
  s.max_sweeps = std::max(1, cx.svd_cap);
  // Cluster size: the least estimated time.  A round costs its barriers, sums
  // and scalars, and the FP64 pipe's share of 3 p + 2 q FMAs per pair; clusters
  // beyond those that run at once wait, several CTAs on an SM share its pipe.
  const int npair = (s.q + 1) / 2, nt = npair > 64 ? 512 : npair > 32 ? 256 : 128;
  const size_t head = sizeof(double) * size_t(svd_head(s.q));
  auto rows_of = [&](int c) { return size_t(svd_ld((s.p + c - 1) / c + (s.q + c - 1) / c)) * s.q; };
  int C = 1;
  bool head_smem = false, rows_smem = false;
  double best = 1e300;
  for (int c = 1; c <= 16 && head <= kQrSmemMax; c *= 2) {
    const bool fits = head + sizeof(double) * rows_of(c) <= kQrSmemMax;
    const size_t smem = head + (fits ? sizeof(double) * rows_of(c) : 0);
    if (c > 1 && s.p / c < 2) break;
    const int at_once = active_clusters(k_svd_cluster, nt, smem, c);
    if (at_once == 0) continue;
    const double per_sm = std::max(1.0, double(std::min(np, at_once)) * c / num_sms());
    const double round = (c == 1 ? 2400.0 : 3600.0 + 70.0 * c) +
                         per_sm * (fits ? 1.0 : 2.0) * npair * (3.0 * s.p + 2.0 * s.q) / (1.4 * c);
    const double t = std::ceil(double(np) / at_once) * round;
    if (t < best) {
      best = t;
      C = c;
      head_smem = true;
      rows_smem = fits;
    }
  }
  // (a matrix too wide for even its sums in shared memory runs on one CTA from global memory)
  if (!head_smem || !rows_smem) {
    s.wst = C * ((head_smem ? 0 : svd_head(s.q)) + (rows_smem ? 0 : (long long)rows_of(C)));
    s.work = cx.scratch(size_t(np) * s.wst + 64);
  }
  const int rows = (s.p + C - 1) / C;
  int lanes = 0;   // threads per inner product: up to 8, while each has four rows and a thread to itself
  while (lanes < 3 && (npair << (lanes + 1)) <= nt && (rows >> (lanes + 1)) >= 4) ++lanes;
  Launch L(K_SVD, cx.st, 0, 0);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C * np, 1, 1);
  cfg.blockDim = dim3(nt, 1, 1);
  cfg.dynamicSmemBytes = (head_smem ? head : 0) + (rows_smem ? sizeof(double) * rows_of(C) : 0);
  cfg.stream = cx.st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  PEPS_CUDA(cudaLaunchKernelEx(&cfg, k_svd_cluster, s, head_smem ? 1 : 0, rows_smem ? 1 : 0, lanes));
  PEPS_CHECK_LAUNCH();
}

// From this width on the iteration runs on a matrix preconditioned by two QR
// factorisations (Drmac & Veselic, without pivoting): G = Q1 R1, R1^T = Q2 R2,
// so G = Q1 R2^T Q2^T, and R2^T is close to diagonal.  The centre matrices of
// a boundary, whose singular values fall by 10 to 20 orders, take 14 to 40
// sweeps as they are and 7 or 8 so (180x180: 28 and 40 sweeps -> 8); random ones
// 10 and 8.  Below, the four extra launches cost what the sweeps do.
constexpr int SVD_PRECOND = 12;

void svd_trunc(Ctx& cx, int m, int n, const TP& A, int kk, const TP& US, const TP& Vt) {
  PEPS_REQUIRE(m > 0 && n > 0 && kk > 0, "svd of an empty matrix");
  const int np = problems({&A, &US, &Vt});
  PEPS_REQUIRE(!A.null() && US.n == np && Vt.n == np, "internal: svd operands");
  const int trans = m < n ? 1 : 0, p = trans ? n : m, q = trans ? m : n;
  const long long rs = trans ? 1 : n, cs = trans ? n : 1;
  {
    Launch count(K_SVD, cx.st, 8.0 * 4.0 * double(p) * q * q * np, 0);   // the flops, once; launches count themselves
    count.more(-1);
  }
  if (q < SVD_PRECOND || kk > q) {
    svd_jacobi(cx, p, q, A, rs, cs, trans, kk, US, Vt, np);
    return;
  }
  const size_t qq = size_t(q) * q, pq = size_t(p) * q, qk = size_t(q) * kk;
  auto up = [](size_t x) { return (x + 31) / 32 * 32; };
  Arena tmp(cx.st, sizeof(double) * np * (up(pq) + 3 * up(qq) + 2 * up(qk)));
  auto blk = [&](size_t per) { return strided(tmp.dalloc(up(per) * np), np, per); };
  const TP Q1 = blk(pq), R1 = blk(qq), Q2 = blk(qq), R2 = blk(qq), u = blk(qk), v = blk(qk);
  qr_thin(cx, p, q, A, rs, cs, Q1, q, 1, R1);
  qr_thin(cx, q, q, R1, 1, q, Q2, q, 1, R2);
  svd_jacobi(cx, q, q, R2, 1, q, trans, kk, u, v, np);
  // G = Q1 (u v) Q2^T, G^T = Q2 (u v) Q1^T
  cx.f64_class = K_SVD;
  cx.f64_flops = false;
  ein(cx, "iq,qk->ik", trans ? Q2 : Q1, {trans ? q : p, q}, u, {q, kk}, US);
  ein(cx, "kq,iq->ki", v, {kk, q}, trans ? Q1 : Q2, {trans ? p : q, q}, Vt);
  cx.f64_class = -1;
  cx.f64_flops = true;
}

}  // namespace peps
