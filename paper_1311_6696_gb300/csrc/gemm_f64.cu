// FP64 gather-GEMM: C[m,n] = alpha * sum_k A[m,k] B[k,n] + beta * C[m,n]
// where m, n, k (and a batch index) are each a group of tensor indices with
// arbitrary strides.  A pairwise tensor contraction therefore runs without
// any permutation copy: each CTA decomposes the row, column and k indices of
// its tile into element offsets once, keeps them in shared memory and
// gathers the operands through them.
//
// What bounds it: the FP64 pipe takes at most 2 FMA per clock and SM (one warp
// instruction in 64 clocks and SM quarter; 1.26 TFLOP/s for the chip at 2070
// MHz, of which torch's DGEMM of 8192^3 reaches 1.10), so slow that a tile of any size keeps it busy -- a 16x16 tile
// needs 2 loaded doubles per 16 FMA -- and what decides the time is that every
// SM gets the same share of the multiply-adds.  A contraction of 1M FMA on
// 64x64 tiles occupies 16 SMs for 20 us; on 16x16 tiles, K split over a
// cluster where the tiles are still too few, all of them for 2.  So tiles are
// 32x32 or 16x16, and the CTAs of a thread-block cluster share one tile's K
// and add up their partial tiles through distributed shared memory, in rank
// order: no partials in global memory, no second launch, and results are
// deterministic.  The index arithmetic is 32-bit with precomputed reciprocals
// (64-bit divisions of every row, column and k index took longer than the
// multiply-adds of a small contraction).
// Measured (us; before: 64x64-output tiles, split K with a second kernel):
// 64x64 outputs, K 64 24.7 -> 6; 1024 outputs, K 64 78 -> 6.3; 256x256, K 16
// 24.7 -> 6.3; 256x16, K 256 85 -> 10; 512x512, K 32 43 -> 23; 147456 outputs,
// K 2304 801 -> 590 (1.15 TFLOP/s).
// Independent problems of one shape (TP pointer sets) share a launch.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <map>

#include "ein.cuh"

namespace cg = cooperative_groups;

namespace peps {

namespace {

constexpr int MAXG = 8;

// A group of indices, extents > 1 only, adjacent ones merged where their
// strides allow it.  mul / shr: x / dim = umulhi(x, mul) >> shr for x < 2^31.
struct Grp {
  int n;
  int dim[MAXG];
  unsigned mul[MAXG];
  int shr[MAXG];
  long long sa[MAXG], sb[MAXG], sc[MAXG];
};

struct GemmArgs {
  TP A, B, C;        // per problem
  int nprob;
  Grp gm, gn, gk, gb;
  long long M, N, K, NB;
  long long kchunk;  // K per CTA of a cluster
  int wide;          // an extent reaches 2^31: 64-bit index arithmetic
  int a_kfast, b_kfast;   // the operand's unit stride lies in the K group
  int plain;         // alpha = 1, beta = 0 (an FP64 compare on the device costs as much as an FMA)
  double alpha, beta;
};

__device__ __forceinline__ void decomp(const Grp& g, int wide, long long idx, long long& oa, long long& ob,
                                       long long& oc) {
  oa = ob = oc = 0;
  if (wide) {
    for (int i = g.n - 1; i >= 0; --i) {
      const long long q = idx / g.dim[i], r = idx - q * g.dim[i];
      idx = q;
      oa += r * g.sa[i];
      ob += r * g.sb[i];
      oc += r * g.sc[i];
    }
    return;
  }
  unsigned x = unsigned(idx);
  for (int i = g.n - 1; i >= 0; --i) {
    unsigned r = x;
    if (i > 0) {
      const unsigned q = __umulhi(x, g.mul[i]) >> g.shr[i];
      r = x - q * unsigned(g.dim[i]);
      x = q;
    }
    oa += r * g.sa[i];
    ob += r * g.sb[i];
    oc += r * g.sc[i];
  }
}

// Grid = (tiles x S, batch x problems); the S CTAs of a cluster share a tile.
// Every thread owns TM x TN outputs, interleaved so that its shared-memory
// reads are conflict-free; the next k tile is loaded into registers while the
// current one is multiplied.
template <int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN)) k_gemm_f64(const __grid_constant__ GemmArgs g) {
  constexpr int TX = BN / TN, TY = BM / TM, NT = TX * TY;
  constexpr int LA = BM * BK / NT, LB = BN * BK / NT;
  static_assert(LA * NT == BM * BK && LB * NT == BN * BK && BM <= NT && BN <= NT && BK <= NT, "tile shape");
  constexpr int TILE = BK * (BM + 1) + BK * (BN + 1), RED = BM * BN;
  __shared__ double sm[TILE > RED ? TILE : RED];
  double(*As)[BM + 1] = reinterpret_cast<double(*)[BM + 1]>(sm);
  double(*Bs)[BN + 1] = reinterpret_cast<double(*)[BN + 1]>(sm + BK * (BM + 1));
  __shared__ long long oAm[BM], oCm[BM], oBn[BN], oCn[BN], oAk[2][BK], oBk[2][BK];
  __shared__ long long bA, bB, bC;
  cg::cluster_group cluster = cg::this_cluster();
  const int S = int(cluster.num_blocks());

  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const long long tiles_n = (g.N + BN - 1) / BN;
  const long long tile = blockIdx.x / S;
  const int split = int(blockIdx.x % S);
  const long long m0 = (tile / tiles_n) * BM, n0 = (tile % tiles_n) * BN;
  const int bi = int(blockIdx.y % g.NB), pb = int(blockIdx.y / g.NB);
  const double* __restrict__ Ap = static_cast<const double*>(g.A.p[pb]);
  const double* __restrict__ Bp = static_cast<const double*>(g.B.p[pb]);
  const long long kbeg = min(g.K, split * g.kchunk), kend = min(g.K, kbeg + g.kchunk);

  auto k_offsets = [&](long long k0, int buf) {
    if (tid < BK) {
      long long k = k0 + tid, a = -1, b = -1, c;
      if (k < kend) decomp(g.gk, g.wide, k, a, b, c);
      oAk[buf][tid] = a;
      oBk[buf][tid] = b;
    }
  };
  if (tid == NT - 1) {
    long long a = 0, b = 0, c = 0;
    if (g.NB > 1) decomp(g.gb, 0, bi, a, b, c);
    bA = a;
    bB = b;
    bC = c;
  }
  if (tid < BM) {
    long long a = -1, b, c = -1;
    if (m0 + tid < g.M) decomp(g.gm, g.wide, m0 + tid, a, b, c);
    oAm[tid] = a;
    oCm[tid] = c;
  }
  if (NT - 1 - tid < BN) {
    const int i = NT - 1 - tid;
    long long a, b = -1, c = -1;
    if (n0 + i < g.N) decomp(g.gn, g.wide, n0 + i, a, b, c);
    oBn[i] = b;
    oCn[i] = c;
  }
  k_offsets(kbeg, 0);
  __syncthreads();

  double ra[LA], rb[LB];
  auto load = [&](int buf) {
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int e = tid + NT * i;
      const int mm = g.a_kfast ? e / BK : e % BM, kk = g.a_kfast ? e % BK : e / BM;
      const long long om = oAm[mm], ok = oAk[buf][kk];
      ra[i] = (om >= 0 && ok >= 0) ? Ap[bA + om + ok] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int e = tid + NT * i;
      const int nn = g.b_kfast ? e / BK : e % BN, kk = g.b_kfast ? e % BK : e / BN;
      const long long on = oBn[nn], ok = oBk[buf][kk];
      rb[i] = (on >= 0 && ok >= 0) ? Bp[bB + on + ok] : 0.0;
    }
  };
  double acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;

  if (kbeg < kend) load(0);
  int buf = 0;
  for (long long k0 = kbeg; k0 < kend; k0 += BK) {
    const bool more = k0 + BK < kend;
    if (more) k_offsets(k0 + BK, buf ^ 1);
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int e = tid + NT * i;
      const int mm = g.a_kfast ? e / BK : e % BM, kk = g.a_kfast ? e % BK : e / BM;
      As[kk][mm] = ra[i];
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int e = tid + NT * i;
      const int nn = g.b_kfast ? e / BK : e % BN, kk = g.b_kfast ? e % BK : e / BN;
      Bs[kk][nn] = rb[i];
    }
    __syncthreads();
    buf ^= 1;
    if (more) load(buf);
    const int kn = int(min((long long)BK, kend - k0));   // no FMAs for K beyond the end
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
      double a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + TY * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + TX * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }

  auto put = [&](int r, int c, double sum) {
    if (oCm[r] < 0 || oCn[c] < 0) return;
    double* p = static_cast<double*>(g.C.p[pb]) + bC + oCm[r] + oCn[c];
    *p = g.plain ? sum : g.alpha * sum + (g.beta != 0.0 ? g.beta * *p : 0.0);
  };
  if (S == 1) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) put(ty + TY * i, tx + TX * j, acc[i][j]);
    return;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) sm[(ty + TY * i) * BN + tx + TX * j] = acc[i][j];
  cluster.sync();
  const int per = (RED + S - 1) / S, e1 = min(RED, (split + 1) * per);
  for (int e = split * per + tid; e < e1; e += NT) {
    double v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = r < S ? *cluster.map_shared_rank(sm + e, r) : 0.0;
    double sum = v[0];
#pragma unroll
    for (int r = 1; r < 8; ++r)
      if (r < S) sum += v[r];
    put(e / BN, e % BN, sum);
  }
  cluster.sync();   // no CTA leaves while others may still read its shared memory
}

// Few outputs, long K (density matrices, scalars): each block reduces one K
// chunk for every output at once; partials are summed in a fixed order.
constexpr int DOT_MAXP = 16;

// Grid = (K chunks, problems).
__global__ void __launch_bounds__(256) k_dot_partial(const GemmArgs g, long long kchunk, double* part) {
  __shared__ long long oa[DOT_MAXP], ob[DOT_MAXP];
  __shared__ double red[8][DOT_MAXP];
  const int P = int(g.M * g.N * g.NB);
  const int tid = threadIdx.x;
  const int pb = blockIdx.y;
  const double* __restrict__ Ap = static_cast<const double*>(g.A.p[pb]);
  const double* __restrict__ Bp = static_cast<const double*>(g.B.p[pb]);
  if (tid < P) {
    const long long bi = tid / (g.M * g.N), mn = tid % (g.M * g.N), m = mn / g.N, n = mn % g.N;
    long long a0, b0, c0, a1, b1, c1, a2, b2, c2;
    decomp(g.gb, g.wide, bi, a0, b0, c0);
    decomp(g.gm, g.wide, m, a1, b1, c1);
    decomp(g.gn, g.wide, n, a2, b2, c2);
    oa[tid] = a0 + a1;
    ob[tid] = b0 + b2;
  }
  __syncthreads();
  double acc[DOT_MAXP];
#pragma unroll
  for (int p = 0; p < DOT_MAXP; ++p) acc[p] = 0.0;
  const long long k0 = blockIdx.x * kchunk, k1 = min(g.K, k0 + kchunk);
  for (long long k = k0 + tid; k < k1; k += blockDim.x) {
    long long ka, kb, kc;
    decomp(g.gk, g.wide, k, ka, kb, kc);
#pragma unroll
    for (int p = 0; p < DOT_MAXP; ++p)
      if (p < P) acc[p] = fma(Ap[oa[p] + ka], Bp[ob[p] + kb], acc[p]);
  }
  const int lane = tid & 31, w = tid >> 5;
#pragma unroll
  for (int p = 0; p < DOT_MAXP; ++p) {
    if (p >= P) break;
    double v = acc[p];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[w][p] = v;
  }
  __syncthreads();
  if (tid < P) {
    double v = 0.0;
    for (int i = 0; i < int(blockDim.x >> 5); ++i) v += red[i][tid];
    part[((long long)pb * gridDim.x + blockIdx.x) * DOT_MAXP + tid] = v;
  }
}

// Grid = problems.
__global__ void k_dot_finish(const GemmArgs g, int nblk, const double* part) {
  const int P = int(g.M * g.N * g.NB);
  const int p = threadIdx.x;
  const int pb = blockIdx.x;
  if (p >= P) return;
  double v = 0.0;
  for (int b = 0; b < nblk; ++b) v += part[((long long)pb * nblk + b) * DOT_MAXP + p];
  const long long bi = p / (g.M * g.N), mn = p % (g.M * g.N), m = mn / g.N, n = mn % g.N;
  long long a, b, c0, c1, c2;
  decomp(g.gb, g.wide, bi, a, b, c0);
  decomp(g.gm, g.wide, m, a, b, c1);
  decomp(g.gn, g.wide, n, a, b, c2);
  double* out = static_cast<double*>(g.C.p[pb]) + c0 + c1 + c2;
  double r = g.alpha * v;
  if (g.beta != 0.0) r += g.beta * *out;
  *out = r;
}

struct Parsed {
  std::string a, b, c;
};

Parsed parse(const char* spec) {
  std::string s(spec);
  auto comma = s.find(',');
  auto arrow = s.find("->");
  PEPS_REQUIRE(comma != std::string::npos && arrow != std::string::npos && comma < arrow,
               std::string("bad contraction spec ") + spec);
  return {s.substr(0, comma), s.substr(comma + 1, arrow - comma - 1), s.substr(arrow + 2)};
}

std::vector<long long> strides_of(const Dims& d) {
  std::vector<long long> s(d.size());
  long long acc = 1;
  for (int i = int(d.size()) - 1; i >= 0; --i) {
    s[i] = acc;
    acc *= d[i];
  }
  return s;
}

}  // namespace

int num_sms() {
  static std::atomic<int> known[64];
  int dev = 0, n = 0;
  PEPS_CUDA(cudaGetDevice(&dev));
  if (dev < 64) n = known[dev].load(std::memory_order_relaxed);
  if (n > 0) return n;
  PEPS_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
  if (dev < 64) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

Dims ein_dims(const char* spec, const Dims& ad, const Dims& bd) {
  Parsed p = parse(spec);
  PEPS_REQUIRE(p.a.size() == ad.size() && p.b.size() == bd.size(),
               std::string("operand rank mismatch in ") + spec);
  Dims out;
  for (char ch : p.c) {
    auto ia = p.a.find(ch);
    auto ib = p.b.find(ch);
    PEPS_REQUIRE(ia != std::string::npos || ib != std::string::npos,
                 std::string("output index not in operands: ") + spec);
    out.push_back(ia != std::string::npos ? ad[ia] : bd[ib]);
  }
  return out;
}

TP strided(double* base, int count, size_t per) {
  TP t;
  t.n = count;
  const size_t stride = (per + 31) / 32 * 32;
  for (int b = 0; b < count; ++b) t.p[b] = base + b * stride;
  return t;
}

int problems(std::initializer_list<const TP*> args) {
  int B = 1;
  for (const TP* t : args) B = std::max(B, t->n);
  for (const TP* t : args) PEPS_REQUIRE(t->n <= 1 || t->n == B, "internal: problem counts differ");
  PEPS_REQUIRE(B <= MAXB, "internal: too many problems in one launch");
  return B;
}

void ein(Ctx& cx, const char* spec, const TP& A, const Dims& ad, const TP& B,
         const Dims& bd, const TP& C, double alpha, double beta) {
  Parsed p = parse(spec);
  Dims cd = ein_dims(spec, ad, bd);
  auto sa = strides_of(ad), sb = strides_of(bd), sc = strides_of(cd);
  const int np = problems({&A, &B, &C});
  PEPS_REQUIRE(!A.null() && !B.null() && C.n == np, "internal: contraction operands");
  GemmArgs g;
  std::memset(static_cast<void*>(&g), 0, sizeof(g));
  g.A = A.all(np);
  g.B = B.all(np);
  g.C = C.all(np);
  g.nprob = np;
  g.alpha = alpha;
  g.beta = beta;
  g.plain = alpha == 1.0 && beta == 0.0 ? 1 : 0;
  bool empty = false, empty_k = false;
  auto push = [&](Grp& gr, int dim, long long a, long long b, long long c) {
    if (dim == 0) empty = true;
    if (dim <= 1) return;
    const int i = gr.n - 1;   // merge with the index before it where every tensor's strides allow it
    if (i >= 0 && gr.sa[i] == a * dim && gr.sb[i] == b * dim && gr.sc[i] == c * dim &&
        (long long)gr.dim[i] * dim < (1LL << 31)) {
      gr.dim[i] *= dim;
      gr.sa[i] = a;
      gr.sb[i] = b;
      gr.sc[i] = c;
      return;
    }
    PEPS_REQUIRE(gr.n < MAXG, std::string("too many indices in one group: ") + spec);
    gr.dim[gr.n] = dim;
    gr.sa[gr.n] = a;
    gr.sb[gr.n] = b;
    gr.sc[gr.n] = c;
    gr.n++;
  };
  // M, N and batch groups in C's order (so the fastest C index is last).
  for (size_t i = 0; i < p.c.size(); ++i) {
    char ch = p.c[i];
    auto ia = p.a.find(ch), ib = p.b.find(ch);
    bool inA = ia != std::string::npos, inB = ib != std::string::npos;
    if (inA && inB) {
      PEPS_REQUIRE(ad[ia] == bd[ib], std::string("dim mismatch in ") + spec);
      push(g.gb, cd[i], sa[ia], sb[ib], sc[i]);
    } else if (inA) {
      push(g.gm, cd[i], sa[ia], 0, sc[i]);
    } else {
      push(g.gn, cd[i], 0, sb[ib], sc[i]);
    }
  }
  const bool empty_c = empty;
  // K group in A's order.  An index summed in one operand only has stride 0 in
  // the other (sum_e A[..e..] B = (sum_e A) B).
  for (size_t i = 0; i < p.a.size(); ++i) {
    char ch = p.a[i];
    if (p.c.find(ch) != std::string::npos) continue;
    auto ib = p.b.find(ch);
    if (ib != std::string::npos) {
      PEPS_REQUIRE(ad[i] == bd[ib], std::string("dim mismatch in ") + spec);
      push(g.gk, ad[i], sa[i], sb[ib], 0);
    } else {
      push(g.gk, ad[i], sa[i], 0, 0);
    }
  }
  for (size_t i = 0; i < p.b.size(); ++i) {
    char ch = p.b[i];
    if (p.c.find(ch) == std::string::npos && p.a.find(ch) == std::string::npos) push(g.gk, bd[i], 0, sb[i], 0);
  }
  empty_k = empty && !empty_c;
  auto finish = [](Grp& gr) {
    long long n = 1;
    for (int i = 0; i < gr.n; ++i) {
      n *= gr.dim[i];
      int l = 1;   // ceil(log2 dim)
      while ((1LL << l) < gr.dim[i]) ++l;
      const unsigned long long d = unsigned(gr.dim[i]);
      gr.mul[i] = unsigned(((1ULL << (31 + l)) + d - 1) / d);
      gr.shr[i] = l - 1;
    }
    return n;
  };
  if (empty_c) return;
  if (empty_k) {
    PEPS_REQUIRE(false, "empty contraction dimension");
  }
  // the operand that holds C's last index is B: its columns are written along
  if (!p.c.empty() && p.a.find(p.c.back()) != std::string::npos && p.b.find(p.c.back()) == std::string::npos) {
    std::swap(g.A, g.B);
    std::swap(g.gm, g.gn);
    for (Grp* gr : {&g.gm, &g.gn, &g.gk, &g.gb})
      for (int i = 0; i < gr->n; ++i) std::swap(gr->sa[i], gr->sb[i]);
  }
  g.M = finish(g.gm);
  g.N = finish(g.gn);
  g.K = finish(g.gk);
  g.NB = finish(g.gb);
  g.wide = std::max({g.M, g.N, g.K}) >= (1LL << 31) ? 1 : 0;
  auto inner = [](const Grp& gr, bool a) {
    long long s = 1LL << 62;
    for (int i = 0; i < gr.n; ++i) s = std::min(s, a ? gr.sa[i] : gr.sb[i]);
    return s;
  };
  g.a_kfast = inner(g.gk, true) < inner(g.gm, true) ? 1 : 0;
  g.b_kfast = inner(g.gk, false) < inner(g.gn, false) ? 1 : 0;
  PEPS_REQUIRE(g.NB * np <= 65535, "batch too large");

  if (g.M * g.N * g.NB <= DOT_MAXP && g.K >= 1024) {
    const long long kchunk = 2048;
    const int nblk = int(std::max<long long>(1, std::min<long long>((g.K + kchunk - 1) / kchunk, 4 * num_sms() / np)));
    const long long kc = (g.K + nblk - 1) / nblk;
    double* part = cx.scratch(size_t(nblk) * np * DOT_MAXP);
    Launch L(cx.f64_class >= 0 ? KClass(cx.f64_class) : K_GEMM_F64, cx.st,
             cx.f64_flops ? 2.0 * double(g.M * g.N * g.NB) * double(g.K) * np : 0.0, 0);
    k_dot_partial<<<dim3(nblk, np), 256, 0, cx.st>>>(g, kc, part);
    k_dot_finish<<<np, 32, 0, cx.st>>>(g, nblk, part);
    L.more();
    PEPS_CHECK_LAUNCH();
    return;
  }
  // Tile and cluster: the least estimated time.  The FP64 pipe of an SM takes
  // its CTAs' padded multiply-adds at 1.7 per clock on average, of the 2 it
  // could, whatever the tile (64x64, 64x32 and 64x16 measured no better than
  // these two); a launch, its index set-up and first loads cost ~4,000 clocks,
  // a CTA's own ~300, a further k tile a load latency that co-resident CTAs
  // hide, and a cluster's exchange ~2,000, likewise.
  struct Shape {
    int bm, bn, bk, nt;
  };
  static const Shape shapes[] = {{32, 32, 32, 128}, {16, 16, 64, 128}};
  const double sms = num_sms();
  int best = 0, S = 1;
  double bestt = 1e300;
  for (int t = 0; t < 2; ++t) {
    const Shape& h = shapes[t];
    const double tiles = double((g.M + h.bm - 1) / h.bm) * double((g.N + h.bn - 1) / h.bn) * double(g.NB) * np;
    for (int c = 1; c <= 8; c *= 2) {
      const double kc = std::ceil(double(g.K) / c);
      if (c > 1 && kc < 8) break;
      double per_sm = tiles * c / sms;
      if (per_sm < 8) per_sm = std::ceil(per_sm);
      const double hidden = std::max(1.0, per_sm / 4.0);
      const double busy = std::min(1.0, 0.5 + 0.125 * per_sm);   // one CTA leaves the pipe idle at its loads
      const double est = 4000.0 + (c > 1 ? 2000.0 * hidden : 0.0) + per_sm * (300.0 + h.bm * h.bn * kc / (1.7 * busy)) +
                         hidden * (std::ceil(kc / h.bk) - 1.0) * 700.0;
      if (est < bestt) {
        bestt = est;
        best = t;
        S = c;
      }
    }
  }
  const Shape& h = shapes[best];
  const long long tiles = ((g.M + h.bm - 1) / h.bm) * ((g.N + h.bn - 1) / h.bn);
  g.kchunk = (g.K + S - 1) / S;
  PEPS_REQUIRE(tiles * S < (1LL << 31), "too many tiles");
  const double flops = 2.0 * double(g.M) * double(g.N) * double(g.K) * double(g.NB) * np;
  Launch L(cx.f64_class >= 0 ? KClass(cx.f64_class) : K_GEMM_F64, cx.st, cx.f64_flops ? flops : 0.0, 0);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(tiles * S), unsigned(g.NB * np), 1);
  cfg.blockDim = dim3(h.nt, 1, 1);
  cfg.stream = cx.st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = S;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (best == 0)
    PEPS_CUDA(cudaLaunchKernelEx(&cfg, k_gemm_f64<32, 32, 32, 2, 4>, g));
  else
    PEPS_CUDA(cudaLaunchKernelEx(&cfg, k_gemm_f64<16, 16, 64, 1, 2>, g));
  PEPS_CHECK_LAUNCH();
}

}  // namespace peps
