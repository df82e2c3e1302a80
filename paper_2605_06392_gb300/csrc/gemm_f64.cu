// FP64 dense tile contractions for the BTA sweeps (sm_103a).
//
// On GB300 the FP64 rate is about two DFMA per clock per SM (a DFMA-chain
// probe reaches ~1.19 TFLOP/s over 152 SMs, while mma.sync .f64 reaches only
// ~1.05), so these kernels are FP64-pipe bound at any reasonable tiling: the
// design goal is to keep every SM's FP64 pipe fed (many resident CTAs, no
// idle tails), not to save bandwidth.  A 16x16 thread grid computes a
// BM x BN tile with DFMA from shared-memory stages of BK = 16, prefetching
// the next stage into registers while the current one is consumed.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdlib>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "common.cuh"

namespace bta {

int64_t g_launches = 0;
int g_launch_priority = 0;

int highest_priority() {
  int least = 0, greatest = 0;
  if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) return 0;
  return greatest;
}

namespace {

constexpr int BK = 16;
constexpr int NT = 256;

// Kernel parameters: shared shape and flags, per-problem pointers indexed by
// blockIdx.z (a batch of same-shaped products in one launch).
struct GemmDev {
  int M, N, K;
  int lda, transA, triA;
  int ldb, transB, triB;
  int ldc, ldcin;
  double alpha, beta;
  int out_lower;
  const double* A[kMaxBatch];
  const double* B[kMaxBatch];
  double* C[kMaxBatch];
  const double* Cin[kMaxBatch];
  int kb[kMaxBatch], ke[kMaxBatch];   // K range of problem z (split-K chunks)
};

__device__ __forceinline__ bool a_zero(int tri, int m, int k) {
  return (tri == TRI_LOWER && k > m) || (tri == TRI_UPPER && k < m);
}
// op(B) is K x N; lower means nonzero only for k >= n.
__device__ __forceinline__ bool b_zero(int tri, int k, int n) {
  return (tri == TRI_LOWER && n > k) || (tri == TRI_UPPER && k > n);
}

template <int BM, int BN>
__global__ void __launch_bounds__(NT) gemm_f64_kernel(GemmDev g) {
  constexpr int TM = BM / 16, TN = BN / 16;
  constexpr int LA = BM * BK / NT;   // A elements loaded per thread per stage
  constexpr int LB = BN * BK / NT;
  __shared__ double As[BK][BM + 1];
  __shared__ double Bs[BK][BN + 1];

  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  if (g.out_lower && n0 > m0 + BM - 1) return;
  const double* __restrict__ A = g.A[blockIdx.z];
  const double* __restrict__ B = g.B[blockIdx.z];
  double* C = g.C[blockIdx.z];
  const double* Cin = g.Cin[blockIdx.z];

  // K range that can hold nonzeros for this tile (absolute k).
  int kbeg = g.kb[blockIdx.z], kend = g.ke[blockIdx.z];
  if (g.triA == TRI_LOWER) kend = min(kend, m0 + BM);
  if (g.triA == TRI_UPPER) kbeg = max(kbeg, m0);
  if (g.triB == TRI_LOWER) kbeg = max(kbeg, n0);
  if (g.triB == TRI_UPPER) kend = min(kend, n0 + BN);
  const int kfirst = kbeg;   // masked loads below start at the chunk start exactly
  kbeg = kbeg / BK * BK;

  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  double acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;

  double ra[LA], rb[LB];
  auto load = [&](int k0) {
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      int idx = tid + NT * r;
      int m, k;
      if (!g.transA) { m = idx % BM; k = idx / BM; } else { k = idx % BK; m = idx / BK; }
      int gm = m0 + m, gk = k0 + k;
      double v = 0.0;
      if (gm < g.M && gk >= kfirst && gk < kend && !a_zero(g.triA, gm, gk))
        v = g.transA ? A[gk + (int64_t)gm * g.lda] : A[gm + (int64_t)gk * g.lda];
      ra[r] = v;
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      int idx = tid + NT * r;
      int n, k;
      if (!g.transB) { k = idx % BK; n = idx / BK; } else { n = idx % BN; k = idx / BN; }
      int gn = n0 + n, gk = k0 + k;
      double v = 0.0;
      if (gn < g.N && gk >= kfirst && gk < kend && !b_zero(g.triB, gk, gn))
        v = g.transB ? B[gn + (int64_t)gk * g.ldb] : B[gk + (int64_t)gn * g.ldb];
      rb[r] = v;
    }
  };
  auto store = [&]() {
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      int idx = tid + NT * r;
      int m, k;
      if (!g.transA) { m = idx % BM; k = idx / BM; } else { k = idx % BK; m = idx / BK; }
      As[k][m] = ra[r];
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      int idx = tid + NT * r;
      int n, k;
      if (!g.transB) { k = idx % BK; n = idx / BK; } else { n = idx % BN; k = idx / BN; }
      Bs[k][n] = rb[r];
    }
  };

  if (kbeg < kend) {
    load(kbeg);
    for (int k0 = kbeg; k0 < kend; k0 += BK) {
      __syncthreads();
      store();
      __syncthreads();
      if (k0 + BK < kend) load(k0 + BK);
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        double av[TM], bv[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) av[i] = As[kk][tx + 16 * i];
#pragma unroll
        for (int j = 0; j < TN; ++j) bv[j] = Bs[kk][ty + 16 * j];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
      }
    }
  }

#pragma unroll
  for (int j = 0; j < TN; ++j) {
    int gn = n0 + ty + 16 * j;
    if (gn >= g.N) continue;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      int gm = m0 + tx + 16 * i;
      if (gm >= g.M) continue;
      if (g.out_lower && gm < gn) continue;
      double v = g.alpha * acc[i][j];
      if (g.beta != 0.0) v = fma(g.beta, Cin[gm + (int64_t)gn * g.ldcin], v);
      C[gm + (int64_t)gn * g.ldc] = v;
    }
  }
}

// ----------------------------------------------------------------------------
// GEMV with a deterministic split over K.
// ----------------------------------------------------------------------------
// C_z = alpha * sum_s part_z[s] + beta * Cin_z over an M x N output (fixed
// order over s, so results do not depend on scheduling).
struct SplitDev {
  int M, N, S, ldc, ldcin;
  double alpha, beta;
  const double* part[kMaxBatch];
  double* C[kMaxBatch];
  const double* Cin[kMaxBatch];
};

__global__ void splitk_reduce(SplitDev d) {
  const int z = blockIdx.y;
  const int64_t mn = (int64_t)d.M * d.N;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < mn;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int m = (int)(e % d.M), n = (int)(e / d.M);
    double acc = 0.0;
    for (int s = 0; s < d.S; ++s) acc += d.part[z][(int64_t)s * mn + e];
    double v = d.alpha * acc;
    if (d.beta != 0.0) v = fma(d.beta, d.Cin[z][m + (int64_t)n * d.ldcin], v);
    d.C[z][m + (int64_t)n * d.ldc] = v;
  }
}

struct GemvDev {
  int M, K, lda, triA, K2, lda2;
  double alpha, beta;
  const double* A[kMaxBatch];
  const double* x[kMaxBatch];
  double* y[kMaxBatch];
  const double* yin[kMaxBatch];
  const double* A2[kMaxBatch];
  const double* x2[kMaxBatch];
};

// y = alpha A x + beta yin.  A matrix-vector product is FP64-pipe bound on one SM
// long before its bytes matter (one 32-lane FMA per 64 clocks and sub-partition),
// so it is spread thinly: a cluster of 8 CTAs owns 32 rows (lane = row, coalesced
// columns), its 64 warps take every 64th column, and the CTAs' partial sums meet in
// the first one's registers through distributed shared memory, in a fixed order: one
// launch, no workspace.  1024 x 1024: 20 us and a second launch before (one warp per
// 32 rows and 64 columns, dependent FMAs), 12 us now (cold cache).
constexpr int kGemvThreads = 256;
constexpr int kGemvCluster = 8;
__global__ void __cluster_dims__(kGemvCluster, 1, 1) __launch_bounds__(kGemvThreads)
    gemv_n_kernel(GemvDev g) {
  namespace cg = cooperative_groups;
  const cg::cluster_group cl = cg::this_cluster();
  const int z = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = (int)cl.block_rank();
  const double* __restrict__ A = g.A[z];
  const double* __restrict__ x = g.x[z];
  const int m0 = (int)(blockIdx.x / kGemvCluster) * 32, m = m0 + lane;
  int kb = 0, ke = g.K;
  if (g.triA == TRI_LOWER) ke = min(ke, m0 + 32);
  if (g.triA == TRI_UPPER) kb = m0;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  const int first = kb + rank * (kGemvThreads / 32) + warp;
  constexpr int kStep = kGemvCluster * kGemvThreads / 32;
  if (m < g.M) {
    for (int k = first; k < ke; k += 4 * kStep) {
      double a[4], v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int kq = k + q * kStep;
        const bool in = kq < ke && !(g.triA == TRI_LOWER && kq > m) &&
                        !(g.triA == TRI_UPPER && kq < m);
        a[q] = in ? A[m + (int64_t)kq * g.lda] : 0.0;
        v[q] = in ? x[kq] : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) s[q] = fma(a[q], v[q], s[q]);
    }
  }
  __shared__ double part[kGemvThreads / 32][32];
  part[warp][lane] = (s[0] + s[1]) + (s[2] + s[3]);
  __syncthreads();
  if (warp == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kGemvThreads / 32; ++w) t += part[w][lane];
    part[0][lane] = t;
  }
  cl.sync();
  if (rank == 0 && warp == 0) {
    double p[kGemvCluster];
#pragma unroll
    for (int r = 0; r < kGemvCluster; ++r) p[r] = cl.map_shared_rank(&part[0][0], r)[lane];
    double t = 0.0;
#pragma unroll
    for (int r = 0; r < kGemvCluster; ++r) t += p[r];
    if (m < g.M) {
      double v = g.alpha * t;
      if (g.beta != 0.0) v = fma(g.beta, g.yin[z][m], v);
      g.y[z][m] = v;
    }
  }
  cl.sync();   // the parts stay until they have been read
}

// y = alpha (A^T x + A2^T x2) + beta yin (A2 optional): one warp per output, lanes
// over K.
__global__ void __launch_bounds__(kGemvThreads) gemv_t_kernel(GemvDev g) {
  const int z = blockIdx.y;
  const double* __restrict__ A = g.A[z];
  const double* __restrict__ x = g.x[z];
  const int m = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (m >= g.M) return;
  int kb = 0, ke = g.K;
  // op(A)[m,k] = A[k,m]; op(A) lower -> zero for k > m
  if (g.triA == TRI_LOWER) ke = min(ke, m + 1);
  if (g.triA == TRI_UPPER) kb = m;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  for (int k = kb + lane; k < ke; k += 128) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int kq = k + 32 * q;
      if (kq < ke) s[q] = fma(A[kq + (int64_t)m * g.lda], x[kq], s[q]);
    }
  }
  for (int k = lane; k < g.K2; k += 32)
    s[0] = fma(g.A2[z][k + (int64_t)m * g.lda2], g.x2[z][k], s[0]);
  double t = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
  for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) {
    double v = g.alpha * t;
    if (g.beta != 0.0) v = fma(g.beta, g.yin[z][m], v);
    g.y[z][m] = v;
  }
}

// The arrow's share of a block (Gram).  A 16 x 64 tile of gemm_f64 took K serial steps of
// mostly padding on one SM's FP64 pipe (a = 9, K = 192: 48 us), and split over K it needed
// a second launch.  Here a cluster of 8 CTAs shares K: a warp reads columns of C, R rows
// of it to a lane group (R = 8 or 16, so 4 or 2 columns at once), and lane m of a group
// accumulates row m of C C^T against the other rows, shuffled in, so that little but real
// products reach the FP64 pipe.  The 64 warps' sums meet in shared memory and through the
// cluster's in a fixed order.  a = 9, K = 192: 9.1 us; a = 12, K = 4800: 255 us in three
// launches with C x before, 45 now.
struct GramDev {
  int a, K;
  const double* C[kMaxBatch];
  double* T[kMaxBatch];
  const double* x[kMaxBatch];
  double* y[kMaxBatch];
};
template <int R>
__global__ void __cluster_dims__(kGemvCluster, 1, 1) __launch_bounds__(kGemvThreads)
    gram_kernel(GramDev g) {
  namespace cg = cooperative_groups;
  const cg::cluster_group cl = cg::this_cluster();
  constexpr int kCols = 32 / R, kWarps = kGemvThreads / 32;
  const int z = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = (int)cl.block_rank(), a = g.a;
  const int m = lane % R, h = lane / R;
  const double* __restrict__ C = g.C[z];
  const double* __restrict__ x = g.x[z];
  double acc[R + 1];   // row m of C C^T, then of C x
#pragma unroll
  for (int n = 0; n <= R; ++n) acc[n] = 0.0;
  constexpr int kStep = kCols * kGemvCluster * kWarps;
  const int first = (rank * kWarps + warp) * kCols + h;
  for (int k0 = first - h; k0 < g.K; k0 += 4 * kStep) {   // one trip count for the warp
    double c[4], v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + h + q * kStep;
      const bool in = k < g.K;
      c[q] = in && m < a ? C[m + (int64_t)k * a] : 0.0;
      v[q] = in && x ? x[k] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (k0 + q * kStep >= g.K) break;   // the same in all lanes
#pragma unroll
      for (int n = 0; n < R; ++n)
        if (n < a) acc[n] = fma(c[q], __shfl_sync(0xffffffffu, c[q], h * R + n), acc[n]);
      if (x) acc[R] = fma(c[q], v[q], acc[R]);
    }
  }
  __shared__ double part[kWarps][R + 1][R], sum[R + 1][R];
#pragma unroll
  for (int n = 0; n <= R; ++n) {
    double t = acc[n];
#pragma unroll
    for (int o = R; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (h == 0) part[warp][n][m] = t;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < (R + 1) * R; e += kGemvThreads) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += part[w][e / R][e % R];
    sum[e / R][e % R] = t;
  }
  cl.sync();
  if (rank == 0) {
    for (int e = threadIdx.x; e < (R + 1) * R; e += kGemvThreads) {
      const int n = e / R, i = e % R;
      double p[kGemvCluster];
#pragma unroll
      for (int r = 0; r < kGemvCluster; ++r) p[r] = cl.map_shared_rank(&sum[0][0], r)[e];
      double t = 0.0;
#pragma unroll
      for (int r = 0; r < kGemvCluster; ++r) t += p[r];
      if (i >= a) continue;
      if (n < a) g.T[z][i + n * a] -= t;
      else if (n == R && x) g.y[z][i] += t;
    }
  }
  cl.sync();   // the sums stay until they have been read
}

// ---- measured tile choice ---------------------------------------------------
// A product's tile shape is timed once per (shape, layout, problems in the
// launch) on scratch buffers and the fastest kept; untimed products use the
// time model.  Timing runs only where a TuneScope is open (the eager first
// evaluation before a graph is captured) and never inside stream capture.
// The tile does not change a product's bits: every tile sums K in the same
// order and the ranges it skips hold exact zeros.
// The measured choices form a process-wide cache (a table of hardware
// timings, keyed by device, guarded by a mutex); the scratch operands of a
// timing are allocated on the stream for that timing alone.
using TuneKey = std::tuple<int, int, int, int, int, int, int, int, int, int, int, int>;
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tuned;
thread_local int g_tune_depth = 0;

bool autotune_on() {
  static const bool v = [] {
    const char* e = getenv("BTA_GEMM_AUTOTUNE");
    return e ? atoi(e) != 0 : true;
  }();
  return v;
}

}  // namespace

TuneScope::TuneScope() { ++g_tune_depth; }
TuneScope::~TuneScope() { --g_tune_depth; }

bta_status gemm_f64(const Gemm& g, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return BTA_OK;
  if (g.Ab ? !(g.Bb && g.Cb) : (g.batch != 1 || !g.A || !g.B || !g.C)) return BTA_ERR_ARG;
  if (g.blocked()) return BTA_ERR_ARG;   // block operands: emulated products only
  const int nb = g.batch;
  const int K = g.K > 0 ? g.K : 0;
  // Tile choice.  Every tile is FP64-pipe bound and the hardware spreads
  // tiles evenly over the SMs, so an op takes about
  // ceil(tiles / SMs) x (BM x BN x K) / rate: pick the shape minimising that
  // (16 x 16 tiles pay ~5 % more for their shared-memory traffic per FMA).
  const int kSMs = sm_count();
  auto units = [&](int bm, int bn, int count) -> int64_t {
    const int tm = cdiv(g.M, bm), tn = cdiv(g.N, bn);
    int64_t u = 0;
    if (!g.out_lower) {
      u = (int64_t)tm * tn;
    } else {
      for (int r = 0; r < tm; ++r) u += std::min(tn, (r * bm + bm - 1) / bn + 1);
    }
    return u * count;
  };
  auto pick = [&](int count) {
    auto cost = [&](int bm, int bn, double pen) {
      const int64_t u = units(bm, bn, count);
      return (double)((u + kSMs - 1) / kSMs) * bm * bn * (1.0 + pen);
    };
    const double c16 = cost(16, 16, 0.05);
    // one row of tiles: 16 x 64 (0) only where its tiles fill the SMs as well (16 x 64 x
    // 64: 18.4 us as one 16 x 64 tile, 7.8 as four)
    if (g.M <= 16) return c16 < cost(16, 64, 0.0) ? 16 : 0;
    const double c64 = cost(64, 64, 0.0), c32 = cost(32, 32, 0.0);
    int bm = 64;
    double best = c64;
    if (c32 < best) { bm = 32; best = c32; }
    if (c16 < best) { bm = 16; best = c16; }
    return bm;
  };
  // Split-K for products with too few output tiles to fill the GPU (the
  // skinny arrow products, a x b by b x b): S chunks of K write partial
  // products to the caller's workspace, then one pass sums them in order.
  int bm = pick(nb);
  int S = 1;
  const bool have_ws = g.sk_ws || g.sk_wsb;
  if (have_ws && !g.out_lower && K >= 256) {
    // a fixed reference tile (not the chosen one): the split, and so the
    // bits of the result, never depend on tile selection
    const int bmn = g.M <= 16 ? 16 : 32, bnn = g.M <= 16 ? 64 : 32;
    // decided per problem (not per batch) so that a product gives the same
    // bits whether it runs alone or inside a batch
    const int64_t u = units(bmn, bnn, 1);
    if (u < kSMs) {
      S = (int)std::min<int64_t>((2 * kSMs + u - 1) / u, std::min(16, K / 64));
      while (S > 1 && (size_t)S * g.M * g.N > g.sk_cap) --S;
    }
  }
  struct Prob { const double *A, *B; double* C; const double* Cin; int kb, ke; };
  std::vector<Prob> probs;
  probs.reserve((size_t)nb * S);
  const int chunk = S > 1 ? (cdiv(K, S) + 15) / 16 * 16 : K;
  for (int z = 0; z < nb; ++z) {
    const double* A = g.Ab ? g.Ab[z] : g.A;
    const double* B = g.Ab ? g.Bb[z] : g.B;
    double* C = g.Ab ? g.Cb[z] : g.C;
    const double* Cin = g.Ab ? (g.Cinb ? g.Cinb[z] : g.Cb[z]) : (g.Cin ? g.Cin : g.C);
    if (S == 1) {
      probs.push_back({A, B, C, Cin, 0, K});
    } else {
      double* ws = g.Ab ? g.sk_wsb[z] : g.sk_ws;
      for (int c = 0; c < S; ++c) {
        const int kb = c * chunk, ke = std::min(K, kb + chunk);
        probs.push_back({A, B, ws + (size_t)c * g.M * g.N, nullptr, kb, std::max(kb, ke)});
      }
    }
  }
  if (S > 1) bm = pick(nb * S);
  const int np = (int)probs.size();
  auto launch = [&](int tbm, const std::vector<Prob>& P) -> bta_status {
    GemmDev d;
    d.M = g.M; d.N = g.N; d.K = K;
    d.lda = g.lda; d.transA = g.transA; d.triA = g.triA;
    d.ldb = g.ldb; d.transB = g.transB; d.triB = g.triB;
    d.ldc = S > 1 ? g.M : g.ldc;
    d.ldcin = S > 1 ? g.M : (g.Cin || g.Cinb ? g.ldcin : g.ldc);
    d.alpha = S > 1 ? 1.0 : g.alpha;
    d.beta = S > 1 ? 0.0 : g.beta;
    d.out_lower = g.out_lower;
    for (int z0 = 0; z0 < np; z0 += kMaxBatch) {
      const int cnt = std::min(kMaxBatch, np - z0);
      for (int z = 0; z < cnt; ++z) {
        const Prob& q = P[z0 + z];
        d.A[z] = q.A; d.B[z] = q.B; d.C[z] = q.C; d.Cin[z] = q.Cin ? q.Cin : q.C;
        d.kb[z] = q.kb; d.ke[z] = q.ke;
      }
      if (tbm == 0) {
        dim3 grid(cdiv(g.M, 16), cdiv(g.N, 64), cnt);
        launch_prio(gemm_f64_kernel<16, 64>, grid, dim3(NT), s, d);
      } else if (tbm == 64) {
        dim3 grid(cdiv(g.M, 64), cdiv(g.N, 64), cnt);
        launch_prio(gemm_f64_kernel<64, 64>, grid, dim3(NT), s, d);
      } else if (tbm == 32) {
        dim3 grid(cdiv(g.M, 32), cdiv(g.N, 32), cnt);
        launch_prio(gemm_f64_kernel<32, 32>, grid, dim3(NT), s, d);
      } else {
        dim3 grid(cdiv(g.M, 16), cdiv(g.N, 16), cnt);
        launch_prio(gemm_f64_kernel<16, 16>, grid, dim3(NT), s, d);
      }
      BTA_LAUNCHED();
    }
    return BTA_OK;
  };
  if (g.M > 16 && autotune_on()) {
    int dev = 0;
    BTA_CUDA_TRY(cudaGetDevice(&dev));
    const TuneKey key{dev, g.M, g.N, K, g.lda, g.ldb, g.transA, g.transB, g.triA, g.triB,
                      g.out_lower, np};
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tuned.find(key);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (it == g_tuned.end() && g_tune_depth > 0 && cudaStreamIsCapturing(s, &cap) == cudaSuccess &&
        cap == cudaStreamCaptureStatusNone) {
      // scratch operands with the product's strides; every problem of the
      // launch points at them (the scratch results are discarded)
      const size_t fa = (size_t)g.lda * (g.transA ? g.M : std::max(K, 1));
      const size_t fb = (size_t)g.ldb * (g.transB ? std::max(K, 1) : g.N);
      const size_t fc = std::max((size_t)g.ldc * g.N, (size_t)g.M * g.N);
      const size_t need = fa + fb + fc;
      double* scratch = nullptr;
      BTA_CUDA_TRY(cudaMallocAsync(&scratch, need * sizeof(double), s));
      BTA_CUDA_TRY(cudaMemsetAsync(scratch, 0, need * sizeof(double), s));
      std::vector<Prob> P(probs);
      for (Prob& q : P) {
        q.A = scratch;
        q.B = scratch + fa;
        q.C = scratch + fa + fb;
        q.Cin = q.Cin ? q.C : nullptr;
      }
      cudaEvent_t e0, e1;
      BTA_CUDA_TRY(cudaEventCreate(&e0));
      BTA_CUDA_TRY(cudaEventCreate(&e1));
      int best = bm;
      float best_ms = 1e30f;
      for (int cand : {64, 32, 16}) {
        float t = 1e30f;
        for (int rep = 0; rep < 3; ++rep) {
          BTA_CUDA_TRY(cudaEventRecord(e0, s));
          BTA_TRY(launch(cand, P));
          BTA_CUDA_TRY(cudaEventRecord(e1, s));
          BTA_CUDA_TRY(cudaEventSynchronize(e1));
          float ms = 0.f;
          BTA_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
          if (rep > 0) t = std::min(t, ms);   // the first run warms up
        }
        if (t < best_ms) { best_ms = t; best = cand; }
      }
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      BTA_CUDA_TRY(cudaFreeAsync(scratch, s));
      it = g_tuned.emplace(key, best).first;
    }
    if (it != g_tuned.end()) bm = it->second;
  }
  BTA_TRY(launch(bm, probs));
  if (S > 1) {
    SplitDev r;
    r.M = g.M; r.N = g.N; r.S = S; r.ldc = g.ldc;
    r.ldcin = g.Cin || g.Cinb ? g.ldcin : g.ldc;
    r.alpha = g.alpha; r.beta = g.beta;
    for (int z0 = 0; z0 < nb; z0 += kMaxBatch) {
      const int cnt = std::min(kMaxBatch, nb - z0);
      for (int z = 0; z < cnt; ++z) {
        const int zz = z0 + z;
        r.part[z] = g.Ab ? g.sk_wsb[zz] : g.sk_ws;
        r.C[z] = g.Ab ? g.Cb[zz] : g.C;
        r.Cin[z] = g.Ab ? (g.Cinb ? g.Cinb[zz] : g.Cb[zz]) : (g.Cin ? g.Cin : g.C);
      }
      const int64_t mn = (int64_t)g.M * g.N;
      const int gx = (int)std::min<int64_t>(cdiv(mn, 256), 608);
      launch_prio(splitk_reduce, dim3(gx, cnt), dim3(256), s, r);
      BTA_LAUNCHED();
    }
  }
  return BTA_OK;
}

bta_status gemv_f64(const Gemv& g, cudaStream_t s) {
  if (g.M <= 0 || g.batch <= 0) return BTA_OK;
  if (g.Ab ? !(g.xb && g.yb) : (g.batch != 1 || !g.A || !g.x || !g.y)) return BTA_ERR_ARG;
  if (g.K2 > 0 && (!g.transA || (g.Ab ? !(g.A2b && g.x2b) : !(g.A2 && g.x2)))) return BTA_ERR_ARG;
  GemvDev d;
  d.M = g.M; d.K = std::max(g.K, 0); d.lda = g.lda; d.triA = g.triA;
  d.K2 = std::max(g.K2, 0); d.lda2 = g.lda2;
  d.alpha = g.alpha; d.beta = g.beta;
  for (int z0 = 0; z0 < g.batch; z0 += kMaxBatch) {
    const int cnt = std::min(kMaxBatch, g.batch - z0);
    for (int z = 0; z < cnt; ++z) {
      const int q = z0 + z;
      d.A[z] = g.Ab ? g.Ab[q] : g.A;
      d.x[z] = g.Ab ? g.xb[q] : g.x;
      d.y[z] = g.Ab ? g.yb[q] : g.y;
      const double* yin = g.Ab ? (g.yinb ? g.yinb[q] : nullptr) : g.yin;
      d.yin[z] = yin ? yin : d.y[z];
      d.A2[z] = g.K2 > 0 ? (g.Ab ? g.A2b[q] : g.A2) : nullptr;
      d.x2[z] = g.K2 > 0 ? (g.Ab ? g.x2b[q] : g.x2) : nullptr;
      // an output is written while others still read x
      if (d.x[z] == d.y[z] || (d.x2[z] && d.x2[z] == d.y[z])) return BTA_ERR_ARG;
    }
    if (!g.transA)
      gemv_n_kernel<<<dim3(kGemvCluster * cdiv(g.M, 32), cnt), kGemvThreads, 0, s>>>(d);
    else
      gemv_t_kernel<<<dim3(cdiv((int64_t)g.M * 32, kGemvThreads), cnt), kGemvThreads, 0, s>>>(d);
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

bta_status gram_f64(const Gram& g, cudaStream_t s) {
  if (g.batch <= 0) return BTA_OK;
  if (g.a < 1 || g.a > kGramRows || !g.C || !g.T) return BTA_ERR_ARG;
  GramDev d;
  d.a = g.a; d.K = std::max(g.K, 0);
  for (int z0 = 0; z0 < g.batch; z0 += kMaxBatch) {
    const int cnt = std::min(kMaxBatch, g.batch - z0);
    for (int z = 0; z < cnt; ++z) {
      d.C[z] = g.C[z0 + z];
      d.T[z] = g.T[z0 + z];
      d.x[z] = g.x ? g.x[z0 + z] : nullptr;
      d.y[z] = g.y ? g.y[z0 + z] : nullptr;
      if (d.x[z] && !d.y[z]) return BTA_ERR_ARG;
    }
    const dim3 grid(kGemvCluster, cnt);
    if (g.a <= 8) gram_kernel<8><<<grid, kGemvThreads, 0, s>>>(d);
    else gram_kernel<16><<<grid, kGemvThreads, 0, s>>>(d);
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

}  // namespace bta
