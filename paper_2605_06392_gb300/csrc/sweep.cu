// The three block sweeps over a BTA matrix (FP64):
//   factor_sweep  -- Algorithm 1, fused block Cholesky + lower solve
//   upper_solve   -- Eqs. 3-5
//   selinv_sweep  -- selected inversion with the Eq. 7 traces fused in
// Each step is a handful of tile-parallel products on the whole GPU; the
// diagonal factor is kept as L_Di^{-1} (see potrf.cu).
#include <algorithm>
#include <cmath>
#include <vector>

#include "sweep.cuh"

// Phase marks of the sweeps for timeline measurements: compile-time empty in
// the library.  A measurement build defines BTA_SWEEP_MARK(stream, tag, block)
// to stamp the time at which the stream's work reaches that point.  Tags:
// 0 / 3 a factor step's start / end, 1 / 2 around its diagonal factor, 4 / 5 a
// selected-inversion step's start / end.
#ifndef BTA_SWEEP_MARK
#define BTA_SWEEP_MARK(s, tag, i) ((void)0)
#endif

namespace bta {
namespace {

// Tip block (a x a, a <= kMaxTip) in one CTA: Cholesky, solves, inverse.
constexpr int kMaxTip = 32;

// One CTA of 128 threads.  FP64 latency (72 clocks an operation, several hundred a
// division or square root) bounds it, so the columns of an update go to different
// threads.  The solves divide by their pivots: products with reciprocals would round twice
// (and save 6 us of a b = 64 gradient's 0.46 ms).  Measured a = 9, mode 0: 35 us with one
// thread, 23 us.
// mode 0: factor T in place (lower L_T, upper zeroed), logdet slot, and if
//         r != null: z_T = L_T^{-1} (r_T - v_T)  (written to r); T2, vT2 (or null):
//         another leg's shares, added to T and v_T
// mode 1: x_T = L_T^{-T} z_T in place (z)
// mode 2: T <- Z_T = L_T^{-T} L_T^{-1} (full)
constexpr int kTipThreads = 128;
__global__ void __launch_bounds__(kTipThreads)
    tip_kernel(int mode, int a, double* T, double* r, const double* vT, const double* T2,
               const double* vT2, double* logdet_slot, int32_t* fail, int32_t fail_code) {
  __shared__ double L[kMaxTip][kMaxTip + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < a * a; e += kTipThreads)
    L[e % a][e / a] = T2 ? T[e] + T2[e] : T[e];
  __syncthreads();
  if (mode == 0) {
    bool bad = false;
    double ld = 0.0;   // lane j of warp 0: log of pivot j
    for (int j = 0; j < a; ++j) {
      double d = L[j][j];
      if (!(d > 0.0) || !isfinite(d)) { bad = true; d = 1.0; }
      const double piv = sqrt(d);   // every thread: the same value
      __syncthreads();
      if (tid < a - j) L[j + tid][j] = tid == 0 ? piv : L[j + tid][j] / piv;
      if (warp == 0 && lane == j) ld = log(piv);
      __syncthreads();
      for (int k = j + 1 + warp; k < a; k += kTipThreads / 32)   // column k, lane = row
        if (lane >= k && lane < a) L[lane][k] = fma(-L[lane][j], L[k][j], L[lane][k]);
      __syncthreads();
    }
    for (int e = tid; e < a * a; e += kTipThreads)
      T[e] = e % a >= e / a ? L[e % a][e / a] : 0.0;
    if (warp == 0) {
#pragma unroll
      for (int o = 16; o; o >>= 1) ld += __shfl_xor_sync(0xffffffffu, ld, o);
      if (lane == 0) {
        *logdet_slot = 2.0 * ld;
        if (bad) atomicCAS(fail, -1, fail_code);
      }
      if (r) {   // lane = row
        double s = lane < a ? r[lane] - vT[lane] : 0.0;
        if (vT2 && lane < a) s -= vT2[lane];
        for (int k = 0; k < a; ++k) {
          const double v = __shfl_sync(0xffffffffu, s, k) / L[k][k];
          if (lane == k) s = v;
          else if (lane > k && lane < a) s = fma(-L[lane][k], v, s);
        }
        if (lane < a) r[lane] = s;
      }
    }
    return;
  }
  if (mode == 1) {
    if (warp == 0) {
      double s = lane < a ? r[lane] : 0.0;
      for (int k = a - 1; k >= 0; --k) {
        const double v = __shfl_sync(0xffffffffu, s, k) / L[k][k];
        if (lane == k) s = v;
        else if (lane < k) s = fma(-L[k][lane], v, s);
      }
      if (lane < a) r[lane] = s;
    }
    return;
  }
  // W = L^{-1} (lower): thread = column; then Z = W^T W
  __shared__ double W[kMaxTip][kMaxTip + 1];
  if (tid < a) {
    for (int i = 0; i < a; ++i) W[i][tid] = i == tid ? 1.0 / L[i][i] : 0.0;
    for (int i = tid + 1; i < a; ++i) {
      double s = 0.0;
      for (int k = tid; k < i; ++k) s = fma(L[i][k], W[k][tid], s);
      W[i][tid] = -s / L[i][i];
    }
  }
  __syncthreads();
  for (int e = tid; e < a * a; e += kTipThreads) {
    const int i = e % a, j = e / a;
    double s = 0.0;
    for (int k = i > j ? i : j; k < a; ++k) s = fma(W[k][i], W[k][j], s);
    T[e] = s;
  }
}

struct CopyDev {
  int lds, ldd, rows, cols;
  double alpha;
  const double* src[kMaxBatch];
  double* dst[kMaxBatch];
};

__global__ void copy_batch_kernel(CopyDev d) {
  const double* __restrict__ src = d.src[blockIdx.y];
  double* __restrict__ dst = d.dst[blockIdx.y];
  const int64_t n = (int64_t)d.rows * d.cols;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    int i = (int)(e % d.rows), j = (int)(e / d.rows);
    dst[i + (int64_t)j * d.ldd] = d.alpha * src[i + (int64_t)j * d.lds];
  }
}

// A pair of 32 x 32 tiles (bi, bj) and (bj, bi), bi >= bj, per CTA: the lower one is read
// once, coalesced, and its transpose written through shared memory (src == dst: only
// the upper triangle is written).
__global__ void __launch_bounds__(256) mirror_kernel(CopyDev d) {
  const int bi = blockIdx.x, bj = blockIdx.y;
  if (bi < bj) return;
  const double* src = d.src[blockIdx.z];
  double* dst = d.dst[blockIdx.z];
  __shared__ double t[32][33];   // t[column][row]
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = bi * 32 + x, c = bj * 32 + y + 8 * q;
    if (r < d.rows && c < d.rows) t[y + 8 * q][x] = src[r + (int64_t)c * d.lds];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = y + 8 * q;
    int r = bi * 32 + x, c = bj * 32 + k;
    if (src != dst && r >= c && r < d.rows && c < d.rows) dst[r + (int64_t)c * d.ldd] = t[k][x];
    // element (c2, r2) of the upper triangle = (r2, c2) of the lower one
    r = bj * 32 + x;
    c = bi * 32 + k;
    if (r < c && c < d.rows) dst[r + (int64_t)c * d.ldd] = t[x][k];
  }
}

__global__ void sum_kernel(const double* parts, int n, double* out, int acc) {
  if (threadIdx.x || blockIdx.x) return;
  double s = 0.0;
  for (int i = 0; i < n; ++i) s += parts[i];
  *out = acc ? *out + s : s;
}

}  // namespace

int sm_count() {
  static int cache[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    dev = 0;
  }
  int* slot = dev >= 0 && dev < 64 ? &cache[dev] : nullptr;
  if (slot && *slot > 0) return *slot;
  int v = 0;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) {
    cudaGetLastError();
    v = 1;
  }
  if (slot) *slot = v;
  return v;
}

bta_status copy_block_batch(int count, const double* const* src, int lds, double* const* dst,
                            int ldd, int rows, int cols, double alpha, cudaStream_t s) {
  const int64_t n = (int64_t)rows * cols;
  if (n <= 0 || count <= 0) return BTA_OK;
  CopyDev d;
  d.lds = lds; d.ldd = ldd; d.rows = rows; d.cols = cols; d.alpha = alpha;
  for (int z0 = 0; z0 < count; z0 += kMaxBatch) {
    const int cnt = std::min(kMaxBatch, count - z0);
    for (int z = 0; z < cnt; ++z) {
      d.src[z] = src[z0 + z];
      d.dst[z] = dst[z0 + z];
    }
    int gx = (int)std::min<int64_t>(cdiv(n, 256), std::max(1, 32 * sm_count() / cnt));
    copy_batch_kernel<<<dim3(gx, cnt), 256, 0, s>>>(d);
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

bta_status copy_block(const double* src, int lds, double* dst, int ldd, int rows, int cols,
                      double alpha, cudaStream_t s) {
  return copy_block_batch(1, &src, lds, &dst, ldd, rows, cols, alpha, s);
}

bta_status mirror_batch(int count, const double* const* src, int lds, double* const* dst, int ldd,
                        int n, cudaStream_t s) {
  if (n <= 0 || count <= 0) return BTA_OK;
  CopyDev d;
  d.lds = lds; d.ldd = ldd; d.rows = n; d.cols = n; d.alpha = 1.0;
  for (int z0 = 0; z0 < count; z0 += kMaxBatch) {
    const int cnt = std::min(kMaxBatch, count - z0);
    for (int z = 0; z < cnt; ++z) {
      d.src[z] = src[z0 + z];
      d.dst[z] = dst[z0 + z];
    }
    mirror_kernel<<<dim3(cdiv(n, 32), cdiv(n, 32), cnt), 256, 0, s>>>(d);
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

bta_status sum_slots(const double* parts, int nparts, double* out, int accumulate,
                     cudaStream_t s) {
  sum_kernel<<<1, 32, 0, s>>>(parts, nparts, out, accumulate);
  BTA_LAUNCHED();
  return BTA_OK;
}

size_t SweepWs::bytes(int ld, int a) {
  size_t m = (size_t)ld * ld;
  // a multiple of 256 bytes: a second workspace carved right after this one
  // keeps its blocks aligned for vector access
  const size_t d = 3 * m + (size_t)a * ld + (size_t)ld + a + 64;
  return sizeof(double) * ((d + 31) / 32 * 32);
}

void SweepWs::carve(double* base, int ld, int a) {
  size_t m = (size_t)ld * ld;
  W1 = base;
  W2 = W1 + m;
  W3 = W2 + m;
  Wc1 = W3 + m;
  gv = Wc1 + (size_t)a * ld;
  vT = gv + ld;
}

int logdet_slots(int n, int ld) { return n * potrf_inv_slots(ld) + 1; }

bool arrow_fused(int ld, int a, int precision) {
  return precision == 2 && a > 0 && ld + a <= kOzakiMaxK;
}

size_t sweep_tc_ws_bytes(int ld, int a, int precision, int group) {
  const int e = a > 0 && ld + a <= kOzakiMaxK ? a : 0;
  const size_t big = precision == 1      ? tc_gemm_ws_bytes(ld, ld, ld)
                     : ld <= kOzakiMaxK ? ozaki_ws_bytes(ld + e, ld, ld + e, group)
                                         : 0;
  return std::max(big, potrf_tc_ws_bytes(ld));
}


namespace {

// Index groups of a set: all items, items with an arrow (grouped by a),
// items with a vector.
struct Groups {
  std::vector<int> all;
  std::vector<std::vector<int>> arrow;   // one group per distinct a > 0
  std::vector<int> vec;
};

Groups make_groups(const SweepItem* it, int m) {
  Groups g;
  for (int z = 0; z < m; ++z) {
    g.all.push_back(z);
    if (it[z].vec) g.vec.push_back(z);
    if (it[z].q.a > 0) {
      bool placed = false;
      for (auto& grp : g.arrow)
        if (it[grp[0]].q.a == it[z].q.a) { grp.push_back(z); placed = true; break; }
      if (!placed) g.arrow.push_back({z});
    }
  }
  return g;
}

// Gather per-item pointers for a batched launch.
template <class F>
std::vector<double*> ptrs(const std::vector<int>& idx, F f) {
  std::vector<double*> v;
  v.reserve(idx.size());
  for (int z : idx) v.push_back(f(z));
  return v;
}

inline const double* const* cp(const std::vector<double*>& v) {
  return reinterpret_cast<const double* const*>(v.data());
}

// A b x b product of the sweep over the items idx: batched FP64
// (precision 0), or one tensor-core product per matrix: split TF32
// (precision 1) or FP64 emulated on BF16 tensor cores (precision 2).
bta_status big_product(const Gemm& g, const SweepItem* it, const std::vector<int>& idx,
                       int precision, cudaStream_t s) {
  if (precision == 0 || (precision == 2 && g.K > 5120)) return gemm_f64(g, s);
  for (size_t z = 0; z < idx.size(); ++z) {
    const SweepWs& ws = it[idx[z]].ws;
    if (!ws.tc) return BTA_ERR_ARG;
    Gemm one = g;
    one.batch = 1;
    one.Ab = nullptr; one.Bb = nullptr; one.Cb = nullptr; one.Cinb = nullptr;
    one.A = g.Ab[z]; one.B = g.Bb[z]; one.C = g.Cb[z];
    one.Cin = g.Cinb ? g.Cinb[z] : g.Cb[z];
    if (precision == 2) {
      BTA_TRY(ozaki_gemm(one, ws.tc, ws.tcstat, s, nullptr, ws.tcgroup));
    } else {
      BTA_TRY(tc_gemm_mixed(one, ws.tc, ws.tcstat, s));
    }
  }
  return BTA_OK;
}

// Whether a product's output may overwrite one of its operands: the tensor-core
// products first copy their operands into planes; the FP64 tiles read them throughout.
bool in_place(int precision, int ld) {
  return precision == 1 || (precision == 2 && ld <= kOzakiMaxK);
}

bta_status check_set(const SweepItem* it, int m) {
  if (m < 1) return BTA_ERR_ARG;
  const bool low = it[0].q.B == nullptr;
  for (int z = 0; z < m; ++z) {
    if (it[z].q.n != it[0].q.n || it[z].q.ld != it[0].q.ld) return BTA_ERR_ARG;
    if (it[z].rev != it[0].rev || it[z].blocks() != it[0].blocks()) return BTA_ERR_ARG;
    if (it[z].q.a > kMaxTip) return BTA_ERR_ARG;
    if ((it[z].q.B == nullptr) != low) return BTA_ERR_ARG;
    if (low && it[z].q.n > 1 && (!it[z].md || !it[z].lay || !it[z].coef)) return BTA_ERR_ARG;
  }
  return BTA_OK;
}

// Where block i of a leg lives (SweepItem): its diagonal and arrow block, vector part and
// slots at block(i) of the matrix, the coupling to block i + 1 in B slot coupling(i),
// which holds Q[i+1, i] of a forward leg and the transpose of a reverse one's.
inline int block_of(const SweepItem& it, int i) { return it.rev ? it.q.n - 1 - i : i; }
inline int coupling_of(const SweepItem& it, int i) { return it.rev ? it.q.n - 2 - i : i; }
inline double* D_of(const SweepItem& it, int i) {
  return it.q.D + block_of(it, i) * (int64_t)it.q.ld * it.q.ld;
}
inline double* B_of(const SweepItem& it, int i) {
  return it.q.B + coupling_of(it, i) * (int64_t)it.q.ld * it.q.ld;
}
inline double* C_of(const SweepItem& it, int i) {
  return it.q.C + block_of(it, i) * (int64_t)it.q.a * it.q.ld;
}
inline double* vec_of(const SweepItem& it, int i) {
  return it.vec + block_of(it, i) * (int64_t)it.q.ld;
}
inline double* tip_vec(const SweepItem& it) { return it.vec + (int64_t)it.q.n * it.q.ld; }

// Low-memory sweeps: the coupling i of every item of idx into the item's W2.
bta_status assemble_b_items(const SweepItem* it, const std::vector<int>& idx, int i,
                            cudaStream_t s) {
  for (int z : idx)
    BTA_TRY(launch_assemble_b(*it[z].md, *it[z].lay, it[z].coef, coupling_of(it[z], i),
                              it[z].ws.W2, s));
  return BTA_OK;
}

}  // namespace

// ----------------------------------------------------------------------------
// Algorithm 1 on a set of matrices
// ----------------------------------------------------------------------------
bta_status factor_sweep_multi(const SweepItem* it, int m, cudaStream_t s, int precision, int i0,
                              int i1, cudaStream_t sv, cudaEvent_t ev) {
  BTA_TRY(check_set(it, m));
  if (!sv) sv = s;
  for (int z = 0; sv != s && z < m; ++z)
    if (!ev || !it[z].q.B) return BTA_ERR_ARG;
  const int n = it[0].blocks(), ld = it[0].q.ld;
  const bool rev = it[0].rev;
  if (i1 < 0) i1 = n;
  if (i0 < 0 || i0 > i1 || i1 > n) return BTA_ERR_ARG;
  const int64_t blk = (int64_t)ld * ld;
  const int p = potrf_inv_slots(ld);
  const Groups G = make_groups(it, m);
  const int M = (int)G.all.size();
  if (i0 == 0)
    for (int z = 0; z < m; ++z) {
      const int a = it[z].q.a;
      if (a > 0 && it[z].vec)
        BTA_CUDA_TRY(cudaMemsetAsync(it[z].ws.vT, 0, a * sizeof(double), s));
      if (a > 0 && it[z].tip)   // the reverse leg's share of the tip
        BTA_CUDA_TRY(cudaMemsetAsync(it[z].tip, 0, (size_t)a * a * sizeof(double), s));
      if (a == 0 && !rev)
        BTA_CUDA_TRY(cudaMemsetAsync(it[z].slots + (int64_t)it[z].q.n * p, 0, sizeof(double), s));
    }
  auto D = [&](int z, int i) { return D_of(it[z], i); };
  auto B = [&](int z, int i) { return B_of(it[z], i); };
  auto Cb = [&](int z, int i) { return C_of(it[z], i); };
  auto tip = [&](int z) { return it[z].tip ? it[z].tip : it[z].q.T; };
  const bool low = it[0].q.B == nullptr;
  // where the factor's coupling L_Bi lives: in place of B_i, or (low memory) in W1 until
  // block i + 1 has been updated with it
  auto LB = [&](int z, int i) { return low ? it[z].ws.W1 : B(z, i); };
  // Emulated FP64: one product per matrix; the arrow rides along (arrow_fused).
  const bool emu = precision == 2 && ld <= kOzakiMaxK;
  const bool over = in_place(precision, ld);
  auto fused = [&](int z) { return emu && arrow_fused(ld, it[z].q.a, precision); };
  auto emulate = [&](int z, const Gemm& g) -> bta_status {
    if (!it[z].ws.tc) return BTA_ERR_ARG;
    return ozaki_gemm(g, it[z].ws.tc, it[z].ws.tcstat, s, nullptr, it[z].ws.tcgroup);
  };
  // T -= L_Ci L_Ci^T and v_T += L_Ci z_i
  auto tip_update = [&](const std::vector<int>& grp, int i) -> bta_status {
    const int a = it[grp[0]].q.a;
    auto Ci = ptrs(grp, [&](int z) { return Cb(z, i); });
    auto T = ptrs(grp, tip);
    if (a <= kGramRows) {
      auto x = ptrs(grp, [&](int z) { return it[z].vec ? vec_of(it[z], i) : nullptr; });
      auto y = ptrs(grp, [&](int z) { return it[z].ws.vT; });
      Gram g; g.a = a; g.K = ld; g.batch = (int)grp.size();
      g.C = cp(Ci); g.T = T.data(); g.x = cp(x); g.y = y.data();
      return gram_f64(g, sv);
    }
    for (int z : grp) {
      if (!it[z].vec) continue;
      Gemv h; h.M = a; h.K = ld; h.A = Cb(z, i); h.lda = a;
      h.x = vec_of(it[z], i); h.y = it[z].ws.vT; h.beta = 1.0;
      BTA_TRY(gemv_f64(h, sv));
    }
    auto SK = ptrs(grp, [&](int z) { return it[z].ws.W3; });
    Gemm h; h.M = a; h.N = a; h.K = ld; h.batch = (int)grp.size();
    h.Ab = cp(Ci); h.lda = a; h.Bb = cp(Ci); h.ldb = a; h.transB = 1;
    h.Cb = T.data(); h.ldc = a; h.Cinb = cp(T); h.ldcin = a; h.alpha = -1.0; h.beta = 1.0;
    h.sk_wsb = SK.data(); h.sk_cap = blk;
    return gemm_f64(h, sv);
  };
  auto vector_step = [&](int i) -> bta_status {
    if (G.vec.empty()) return BTA_OK;
    // t = r_i - L_B,i-1 z_{i-1} into gv (r_0 itself for the first block; into r_i where
    // the legs join)
    const int c = (int)G.vec.size();
    auto ri = ptrs(G.vec, [&](int z) { return vec_of(it[z], i); });
    auto gv = ptrs(G.vec, [&](int z) { return i == i1 ? vec_of(it[z], i) : it[z].ws.gv; });
    if (i == 0) {
      BTA_TRY(copy_block_batch(c, cp(ri), ld, gv.data(), ld, ld, 1, 1.0, sv));
    } else {
      auto Bp = ptrs(G.vec, [&](int z) { return LB(z, i - 1); });
      auto rp = ptrs(G.vec, [&](int z) { return vec_of(it[z], i - 1); });
      Gemv g; g.M = ld; g.K = ld; g.lda = ld; g.alpha = -1.0; g.beta = 1.0; g.batch = c;
      g.Ab = cp(Bp); g.xb = cp(rp); g.yb = gv.data(); g.yinb = cp(ri);
      BTA_TRY(gemv_f64(g, sv));
    }
    return BTA_OK;
  };
  // The arrow in FP64 products, where none of b x b carries it: C_i -= L_C,i-1 L_B,i-1^T ...
  auto arrow_update = [&](int i) -> bta_status {
    for (const auto& grp : G.arrow) {
      if (fused(grp[0])) continue;      // carried by the product above
      const int a = it[grp[0]].q.a;
      auto Cp = ptrs(grp, [&](int z) { return Cb(z, i - 1); });
      auto Bp = ptrs(grp, [&](int z) { return LB(z, i - 1); });
      auto Ci = ptrs(grp, [&](int z) { return Cb(z, i); });
      auto SK = ptrs(grp, [&](int z) { return it[z].ws.W3; });   // W3 is free here
      Gemm g; g.M = a; g.N = ld; g.K = ld; g.batch = (int)grp.size();
      g.Ab = cp(Cp); g.lda = a; g.Bb = cp(Bp); g.ldb = ld; g.transB = 1;
      g.Cb = Ci.data(); g.ldc = a; g.Cinb = cp(Ci); g.ldcin = a; g.alpha = -1.0; g.beta = 1.0;
      g.sk_wsb = SK.data(); g.sk_cap = blk;
      BTA_TRY(gemm_f64(g, sv));
    }
    return BTA_OK;
  };
  // ... and L_Ci = C_i L_Di^{-T}
  auto arrow_factor = [&](int i) -> bta_status {
    const bool with_b = emu && i < n - 1;   // L_Ci as extra rows of L_Bi's product
    for (const auto& grp : G.arrow) {
      if (with_b && fused(grp[0])) continue;
      const int a = it[grp[0]].q.a, c = (int)grp.size();
      auto Ci = ptrs(grp, [&](int z) { return Cb(z, i); });
      auto Di = ptrs(grp, [&](int z) { return D(z, i); });
      auto W = ptrs(grp, [&](int z) { return it[z].ws.Wc1; });
      auto SK = ptrs(grp, [&](int z) { return it[z].ws.W3; });
      Gemm g; g.M = a; g.N = ld; g.K = ld; g.batch = c;
      g.Ab = cp(Ci); g.lda = a; g.Bb = cp(Di); g.ldb = ld; g.transB = 1; g.triB = TRI_UPPER;
      g.Cb = W.data(); g.ldc = a;
      g.sk_wsb = SK.data(); g.sk_cap = blk;
      BTA_TRY(gemm_f64(g, sv));
      BTA_TRY(copy_block_batch(c, cp(W), a, Ci.data(), a, a, ld, 1.0, sv));
    }
    return BTA_OK;
  };
  for (int i = i0; i <= i1 && i < n; ++i) {
    // the range's end: a reverse leg's last coupling updates the block the legs share
    const bool join = i == i1;
    if (join && !(rev && i1 == n - 1)) break;
    if (!join) BTA_SWEEP_MARK(s, 0, i);
    if (i > 0) {
      if (emu) {  // D_i -= L_B,i-1 L_B,i-1^T (lower); rows below: C_i -= L_C,i-1 L_B,i-1^T
        for (int z : G.all) {
          Gemm g; g.M = ld; g.N = ld; g.K = ld;
          g.A = LB(z, i - 1); g.lda = ld; g.B = g.A; g.ldb = ld; g.transB = 1;
          g.C = D(z, i); g.ldc = ld; g.Cin = g.C; g.ldcin = ld;
          g.alpha = -1.0; g.beta = 1.0; g.out_lower = 1;
          if (fused(z)) {
            const int a = it[z].q.a;
            g.M = ld + a; g.a_rows = ld; g.A21 = {Cb(z, i - 1), a, 0};
            g.c_rows = ld; g.C2 = Cb(z, i); g.ldc2 = a; g.Cin2 = g.C2; g.ldcin2 = a;
          }
          BTA_TRY(emulate(z, g));
        }
      } else {  // D_i -= S_{i-1} = L_B,i-1 L_B,i-1^T (lower)
        auto Bp = ptrs(G.all, [&](int z) { return LB(z, i - 1); });
        auto Di = ptrs(G.all, [&](int z) { return D(z, i); });
        Gemm g; g.M = ld; g.N = ld; g.K = ld; g.batch = M;
        g.Ab = cp(Bp); g.lda = ld; g.Bb = cp(Bp); g.ldb = ld; g.transB = 1;
        g.Cb = Di.data(); g.ldc = ld; g.Cinb = cp(Di); g.ldcin = ld;
        g.alpha = -1.0; g.beta = 1.0; g.out_lower = 1;
        BTA_TRY(big_product(g, it, G.all, precision, s));
      }
    }
    if (join || sv == s) {
      if (i > 0) BTA_TRY(arrow_update(i));
      BTA_TRY(vector_step(i));
    }
    if (join) return BTA_OK;
    {  // L_Di^{-1} in place, log-det slots
      auto Di = ptrs(G.all, [&](int z) { return D(z, i); });
      auto W = ptrs(G.all, [&](int z) { return it[z].ws.W2; });
      auto sl = ptrs(G.all, [&](int z) { return it[z].slots + (int64_t)block_of(it[z], i) * p; });
      std::vector<int32_t*> fl;
      std::vector<int32_t> code;
      for (int z : G.all) {
        fl.push_back(it[z].fail);
        code.push_back(block_of(it[z], i));
      }
      std::vector<void*> tw;
      std::vector<int32_t*> ts;
      for (int z : G.all) {
        tw.push_back(it[z].ws.tc);
        ts.push_back(it[z].ws.tcstat);
      }
      BTA_SWEEP_MARK(s, 1, i);
      BTA_TRY(potrf_inv_batch_prec(M, Di.data(), ld, ld, W.data(), sl.data(), fl.data(),
                                   code.data(), precision, tw.data(), ts.data(), s));
      BTA_SWEEP_MARK(s, 2, i);
    }
    if (sv == s) BTA_TRY(arrow_factor(i));
    if (i < n - 1) {  // L_Bi = Q[i+1, i] L_Di^{-T}
      if (low) BTA_TRY(assemble_b_items(it, G.all, i, s));
      auto Bi = ptrs(G.all, [&](int z) { return low ? it[z].ws.W2 : B(z, i); });
      auto Di = ptrs(G.all, [&](int z) { return D(z, i); });
      auto W = ptrs(G.all, [&](int z) { return low || !over ? it[z].ws.W1 : B(z, i); });
      if (emu) {  // rows below: L_Ci = C_i L_Di^{-T}
        for (size_t q = 0; q < G.all.size(); ++q) {
          const int z = G.all[q];
          Gemm g; g.M = ld; g.N = ld; g.K = ld;
          g.A = Bi[q]; g.lda = ld; g.transA = rev; g.B = Di[q]; g.ldb = ld; g.transB = 1;
          g.triB = TRI_UPPER; g.C = W[q]; g.ldc = ld;
          if (fused(z)) {
            const int a = it[z].q.a;
            g.M = ld + a; g.a_rows = ld; g.A21 = {Cb(z, i), a, 0};
            g.c_rows = ld; g.C2 = Cb(z, i); g.ldc2 = a;
          }
          BTA_TRY(emulate(z, g));
        }
      } else {
        Gemm g; g.M = ld; g.N = ld; g.K = ld; g.batch = M;
        g.Ab = cp(Bi); g.lda = ld; g.transA = rev; g.Bb = cp(Di); g.ldb = ld; g.transB = 1;
        g.triB = TRI_UPPER; g.Cb = W.data(); g.ldc = ld;
        BTA_TRY(big_product(g, it, G.all, precision, s));
      }
      if (!low && !over) BTA_TRY(copy_block_batch(M, cp(W), ld, Bi.data(), ld, ld, ld, 1.0, s));
    }
    if (sv != s) {
      BTA_CUDA_TRY(cudaEventRecord(ev, s));
      BTA_CUDA_TRY(cudaStreamWaitEvent(sv, ev, 0));
      if (i > 0) BTA_TRY(arrow_update(i));
      BTA_TRY(vector_step(i));
      BTA_TRY(arrow_factor(i));
    }
    if (!G.vec.empty()) {  // z_i = L_Di^{-1} t
      auto zi = ptrs(G.vec, [&](int z) { return vec_of(it[z], i); });
      auto gv = ptrs(G.vec, [&](int z) { return it[z].ws.gv; });
      auto Di = ptrs(G.vec, [&](int z) { return D(z, i); });
      Gemv g; g.M = ld; g.K = ld; g.lda = ld; g.triA = TRI_LOWER; g.batch = (int)G.vec.size();
      g.Ab = cp(Di); g.xb = cp(gv); g.yb = zi.data();
      BTA_TRY(gemv_f64(g, sv));
    }
    for (const auto& grp : G.arrow) BTA_TRY(tip_update(grp, i));
    BTA_SWEEP_MARK(s, 3, i);
  }
  if (i1 < n) return BTA_OK;
  if (sv != s) {
    BTA_CUDA_TRY(cudaEventRecord(ev, sv));
    BTA_CUDA_TRY(cudaStreamWaitEvent(s, ev, 0));
  }
  for (int z = 0; z < m; ++z) {
    const int a = it[z].q.a;
    if (a == 0) continue;
    tip_kernel<<<1, kTipThreads, 0, s>>>(0, a, it[z].q.T, it[z].vec ? tip_vec(it[z]) : nullptr,
                                         it[z].ws.vT, it[z].tip2, it[z].vT2,
                                         it[z].slots + (int64_t)it[z].q.n * p, it[z].fail,
                                         it[z].q.n);
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

bta_status factor_sweep(const bta_desc& q, double* rhs, double* slots, int32_t* fail,
                        const SweepWs& ws, cudaStream_t s, int precision) {
  SweepItem item;
  item.q = q; item.vec = rhs; item.slots = slots; item.fail = fail; item.ws = ws;
  return factor_sweep_multi(&item, 1, s, precision);
}

// ----------------------------------------------------------------------------
// Residual d - Q x of an assembled BTA matrix (the refinement step of
// bta_solve), as GEMVs on its blocks.  D_i is stored as its lower triangle:
// D_i x = L x + L^T x - diag(D_i) x with L the stored lower part.
// ----------------------------------------------------------------------------
namespace {
__global__ void diag_axpy_kernel(const double* __restrict__ D, int ld, const double* x,
                                 double* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < ld) y[i] = fma(D[i + (int64_t)i * ld], x[i], y[i]);
}
}  // namespace

bta_status bta_residual(const bta_desc& q, const double* x, double* d, cudaStream_t s) {
  const int n = q.n, ld = q.ld, a = q.a;
  const int64_t blk = (int64_t)ld * ld;
  const double* xT = x + (int64_t)n * ld;
  double* dT = d + (int64_t)n * ld;
  for (int i = 0; i < n; ++i) {
    const double* xi = x + (int64_t)i * ld;
    double* di = d + (int64_t)i * ld;
    const double* Di = q.D + i * blk;
    auto minus = [&](const double* A, int lda, int M, int K, int trans, int tri,
                     const double* v, double* y) {
      Gemv g; g.M = M; g.K = K; g.A = A; g.lda = lda; g.transA = trans; g.triA = tri;
      g.x = v; g.y = y; g.alpha = -1.0; g.beta = 1.0;
      return gemv_f64(g, s);
    };
    BTA_TRY(minus(Di, ld, ld, ld, 0, TRI_LOWER, xi, di));          // - L x
    BTA_TRY(minus(Di, ld, ld, ld, 1, TRI_UPPER, xi, di));          // - L^T x
    diag_axpy_kernel<<<cdiv(ld, 256), 256, 0, s>>>(Di, ld, xi, di);   // + diag x
    BTA_LAUNCHED();
    if (i > 0) BTA_TRY(minus(q.B + (i - 1) * blk, ld, ld, ld, 0, TRI_NONE, xi - ld, di));
    if (i < n - 1) BTA_TRY(minus(q.B + i * blk, ld, ld, ld, 1, TRI_NONE, xi + ld, di));
    if (a > 0) {
      const double* Ci = q.C + (int64_t)i * a * ld;
      BTA_TRY(minus(Ci, a, ld, a, 1, TRI_NONE, xT, di));           // - C_i^T x_T
      BTA_TRY(minus(Ci, a, a, ld, 0, TRI_NONE, xi, dT));           // tip row: - C_i x_i
    }
  }
  if (a > 0) {   // - T x_T (lower triangle referenced, as D)
    Gemv g; g.M = a; g.K = a; g.A = q.T; g.lda = a; g.triA = TRI_LOWER;
    g.x = xT; g.y = dT; g.alpha = -1.0; g.beta = 1.0;
    BTA_TRY(gemv_f64(g, s));
    g.transA = 1; g.triA = TRI_UPPER;
    BTA_TRY(gemv_f64(g, s));
    diag_axpy_kernel<<<1, 32, 0, s>>>(q.T, a, xT, dT);
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

// ----------------------------------------------------------------------------
// Lower solve alone (L z = r) with a factor
// ----------------------------------------------------------------------------
namespace {
// z_T = L_T^{-1} (r_T - v_T) with the factored tip: one warp, lane = row.
__global__ void tip_fwd_kernel(int a, const double* T, double* r, const double* vT) {
  const int lane = threadIdx.x;
  double s = lane < a ? r[lane] - vT[lane] : 0.0;
  for (int k = 0; k < a; ++k) {
    const double v = __shfl_sync(0xffffffffu, s, k) / T[k + k * a];
    if (lane == k) s = v;
    else if (lane > k && lane < a) s = fma(-T[lane + k * a], v, s);
  }
  if (lane < a) r[lane] = s;
}
}  // namespace

bta_status lower_solve(const SweepItem& it, cudaStream_t s) {
  const int n = it.q.n, ld = it.q.ld, a = it.q.a;
  if (it.rev || !it.vec || (n > 1 && !it.q.B)) return BTA_ERR_ARG;
  if (a > 0) BTA_CUDA_TRY(cudaMemsetAsync(it.ws.vT, 0, a * sizeof(double), s));
  for (int i = 0; i < n; ++i) {
    double* ri = vec_of(it, i);
    if (i == 0) {
      BTA_TRY(copy_block(ri, ld, it.ws.gv, ld, ld, 1, 1.0, s));
    } else {
      Gemv g; g.M = ld; g.K = ld; g.A = B_of(it, i - 1); g.lda = ld;
      g.x = vec_of(it, i - 1); g.y = it.ws.gv; g.yin = ri;
      g.alpha = -1.0; g.beta = 1.0;
      BTA_TRY(gemv_f64(g, s));
    }
    Gemv g; g.M = ld; g.K = ld; g.A = D_of(it, i); g.lda = ld; g.triA = TRI_LOWER;
    g.x = it.ws.gv; g.y = ri;
    BTA_TRY(gemv_f64(g, s));
    if (a > 0) {
      Gemv h; h.M = a; h.K = ld; h.A = C_of(it, i); h.lda = a; h.x = ri;
      h.y = it.ws.vT; h.beta = 1.0;
      BTA_TRY(gemv_f64(h, s));
    }
  }
  if (a > 0) {
    tip_fwd_kernel<<<1, 32, 0, s>>>(a, it.q.T, tip_vec(it), it.ws.vT);
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

// ----------------------------------------------------------------------------
// Eqs. 3-5 on a set of matrices (items with a vector)
// ----------------------------------------------------------------------------
bta_status upper_solve_multi(const SweepItem* it, int m, cudaStream_t s, int i_hi, int i_lo) {
  BTA_TRY(check_set(it, m));
  const int n = it[0].blocks(), ld = it[0].q.ld;
  if (i_hi < 0) i_hi = n - 1;
  if (i_lo < 0 || i_hi >= n || i_lo > i_hi + 1) return BTA_ERR_ARG;
  const Groups G = make_groups(it, m);
  if (G.vec.empty()) return BTA_OK;
  const int c = (int)G.vec.size();
  if (i_hi == n - 1)
    for (int z : G.vec) {
      const int a = it[z].q.a;
      if (a == 0) continue;
      tip_kernel<<<1, kTipThreads, 0, s>>>(1, a, it[z].q.T, tip_vec(it[z]), nullptr, nullptr,
                                           nullptr, nullptr, nullptr, 0);
      BTA_LAUNCHED();
    }
  bool same_a = true;   // one launch over the set: the arrow rides along
  for (int z : G.vec) same_a = same_a && it[z].q.a == it[G.vec[0]].q.a;
  if (!same_a) return BTA_ERR_ARG;
  const int a = it[G.vec[0]].q.a;
  const bool low = it[0].q.B == nullptr;
  auto gv = ptrs(G.vec, [&](int z) { return it[z].ws.gv; });
  auto xT = ptrs(G.vec, [&](int z) { return tip_vec(it[z]); });
  for (int i = i_hi; i >= i_lo; --i) {
    auto zi = ptrs(G.vec, [&](int z) { return vec_of(it[z], i); });
    auto Di = ptrs(G.vec, [&](int z) { return D_of(it[z], i); });
    std::vector<double*> Ci;
    if (a > 0) Ci = ptrs(G.vec, [&](int z) { return C_of(it[z], i); });
    const bool hasB = i < n - 1;
    std::vector<double*> xn;
    if (hasB) xn = ptrs(G.vec, [&](int z) { return vec_of(it[z], i + 1); });
    // gv = z_i - L_Bi^T x_{i+1} - L_Ci^T x_T
    Gemv g; g.M = ld; g.transA = 1; g.alpha = -1.0; g.beta = 1.0; g.batch = c;
    g.yb = gv.data(); g.yinb = cp(zi);
    if (hasB && !low) {
      auto Bi = ptrs(G.vec, [&](int z) { return B_of(it[z], i); });
      g.K = ld; g.lda = ld; g.Ab = cp(Bi); g.xb = cp(xn);
      if (a > 0) { g.K2 = a; g.lda2 = a; g.A2b = cp(Ci); g.x2b = cp(xT); }
      BTA_TRY(gemv_f64(g, s));
    } else if (a > 0) {
      g.K = a; g.lda = a; g.Ab = cp(Ci); g.xb = cp(xT);
      BTA_TRY(gemv_f64(g, s));
    } else {
      BTA_TRY(copy_block_batch(c, cp(zi), ld, gv.data(), ld, ld, 1, 1.0, s));
    }
    if (hasB && low) {
      // low memory: L_Bi^T x_{i+1} = L_Di^{-1} (Q[i+1, i]^T x_{i+1}), the coupling assembled
      // into W2, the product into W3's first ld entries
      BTA_TRY(assemble_b_items(it, G.vec, i, s));
      auto W2 = ptrs(G.vec, [&](int z) { return it[z].ws.W2; });
      auto t = ptrs(G.vec, [&](int z) { return it[z].ws.W3; });
      Gemv b; b.M = ld; b.K = ld; b.lda = ld; b.transA = !it[0].rev; b.batch = c;
      b.Ab = cp(W2); b.xb = cp(xn); b.yb = t.data();
      BTA_TRY(gemv_f64(b, s));
      Gemv h; h.M = ld; h.K = ld; h.lda = ld; h.triA = TRI_LOWER; h.alpha = -1.0; h.beta = 1.0;
      h.batch = c; h.Ab = cp(Di); h.xb = cp(t); h.yb = gv.data();
      BTA_TRY(gemv_f64(h, s));
    }
    {  // x_i = L_Di^{-T} gv
      Gemv h; h.M = ld; h.K = ld; h.lda = ld; h.transA = 1; h.triA = TRI_UPPER;
      h.batch = c; h.Ab = cp(Di); h.xb = cp(gv); h.yb = zi.data();
      BTA_TRY(gemv_f64(h, s));
    }
  }
  return BTA_OK;
}

// ----------------------------------------------------------------------------
// Selected inversion, in place, on a set of matrices.  With F_Bi = L_Bi
// L_Di^{-1}, F_Ci = L_Ci L_Di^{-1}:
//   Z_Ci = -Z_T F_Ci - Z_C,i+1 F_Bi
//   Z_Bi = -Z_D,i+1 F_Bi - Z_C,i+1^T F_Ci
//   Z_Di = L_Di^{-T} L_Di^{-1} - Z_Bi^T F_Bi - Z_Ci^T F_Ci
// ----------------------------------------------------------------------------
bta_status selinv_sweep_multi(const SweepItem* it, int m, cudaStream_t s, int precision,
                              int i_hi, int i_lo) {
  BTA_TRY(check_set(it, m));
  const int n = it[0].blocks(), ld = it[0].q.ld;
  const bool rev = it[0].rev;
  if (i_hi < 0) i_hi = n - 1;
  if (i_lo < 0 || i_hi >= n || i_lo > i_hi + 1) return BTA_ERR_ARG;
  const int64_t blk = (int64_t)ld * ld;
  const Groups G = make_groups(it, m);
  const int M = (int)G.all.size();
  auto D = [&](int z, int i) { return D_of(it[z], i); };
  auto B = [&](int z, int i) { return B_of(it[z], i); };
  auto Cb = [&](int z, int i) { return C_of(it[z], i); };
  if (i_hi == n - 1 && !rev)
    for (int z = 0; z < m; ++z) {
      if (it[z].q.a == 0) continue;
      tip_kernel<<<1, kTipThreads, 0, s>>>(2, it[z].q.a, it[z].q.T, nullptr, nullptr, nullptr,
                                           nullptr, nullptr, nullptr, 0);
      BTA_LAUNCHED();
    }
  auto W1 = ptrs(G.all, [&](int z) { return it[z].ws.W1; });
  const bool low = it[0].q.B == nullptr;
  // Emulated FP64: one product per matrix; the arrow rides along (arrow_fused).
  const bool emu = precision == 2 && ld <= kOzakiMaxK;
  const bool over = in_place(precision, ld);
  auto fused = [&](int z) { return emu && arrow_fused(ld, it[z].q.a, precision); };
  auto emulate = [&](int z, const Gemm& g) -> bta_status {
    if (!it[z].ws.tc) return BTA_ERR_ARG;
    return ozaki_gemm(g, it[z].ws.tc, it[z].ws.tcstat, s, nullptr, it[z].ws.tcgroup);
  };
  for (int i = i_hi; i >= i_lo; --i) {
    BTA_SWEEP_MARK(s, 4, i);
    const bool hasB = i < n - 1;
    auto Di = ptrs(G.all, [&](int z) { return D(z, i); });
    // Z_B in place of L_Bi, free once F_B is formed (low memory: in W2)
    std::vector<double*> ZB;
    if (hasB) ZB = ptrs(G.all, [&](int z) { return low ? it[z].ws.W2 : B(z, i); });
    // Z_D is built in place, or (FP64 products) in W3
    auto ZD = ptrs(G.all, [&](int z) { return over ? D(z, i) : it[z].ws.W3; });
    if (hasB && low) {  // low memory: W3 = L_Bi = Q[i+1, i] L_Di^{-T}, assembled into W2
      BTA_TRY(assemble_b_items(it, G.all, i, s));
      auto W2 = ptrs(G.all, [&](int z) { return it[z].ws.W2; });
      auto W3 = ptrs(G.all, [&](int z) { return it[z].ws.W3; });
      Gemm g; g.M = ld; g.N = ld; g.K = ld; g.batch = M;
      g.Ab = cp(W2); g.lda = ld; g.transA = rev; g.Bb = cp(Di); g.ldb = ld; g.transB = 1;
      g.triB = TRI_UPPER; g.Cb = W3.data(); g.ldc = ld;
      BTA_TRY(big_product(g, it, G.all, precision, s));
    }
    if (hasB) {  // W1 = F_B = L_Bi L_Di^{-1}
      auto Bi = ptrs(G.all, [&](int z) { return low ? it[z].ws.W3 : B(z, i); });
      if (emu) {  // rows below: Wc1 = F_C = L_Ci L_Di^{-1}
        for (size_t q = 0; q < G.all.size(); ++q) {
          const int z = G.all[q];
          Gemm g; g.M = ld; g.N = ld; g.K = ld;
          g.A = Bi[q]; g.lda = ld; g.B = Di[q]; g.ldb = ld; g.triB = TRI_LOWER;
          g.C = W1[q]; g.ldc = ld;
          if (fused(z)) {
            const int a = it[z].q.a;
            g.M = ld + a; g.a_rows = ld; g.A21 = {Cb(z, i), a, 0};
            g.c_rows = ld; g.C2 = it[z].ws.Wc1; g.ldc2 = a;
          }
          BTA_TRY(emulate(z, g));
        }
      } else {
        Gemm g; g.M = ld; g.N = ld; g.K = ld; g.batch = M;
        g.Ab = cp(Bi); g.lda = ld; g.Bb = cp(Di); g.ldb = ld; g.triB = TRI_LOWER;
        g.Cb = W1.data(); g.ldc = ld;
        BTA_TRY(big_product(g, it, G.all, precision, s));
      }
    }
    for (const auto& grp : G.arrow) {
      // with B_i, an arrow carried by the products (arrow_fused) gets F_C above
      // and Z_C with Z_B below
      if (hasB && fused(grp[0])) continue;
      const int a = it[grp[0]].q.a, c = (int)grp.size();
      auto Ci = ptrs(grp, [&](int z) { return Cb(z, i); });
      auto Dg = ptrs(grp, [&](int z) { return D(z, i); });
      auto Wc1 = ptrs(grp, [&](int z) { return it[z].ws.Wc1; });
      auto T = ptrs(grp, [&](int z) { return it[z].q.T; });
      auto SK = ptrs(grp, [&](int z) { return it[z].ws.W3; });   // W3 is free until LAUUM
      {  // Wc1 = F_C = L_Ci L_Di^{-1}
        Gemm g; g.M = a; g.N = ld; g.K = ld; g.batch = c;
        g.Ab = cp(Ci); g.lda = a; g.Bb = cp(Dg); g.ldb = ld; g.triB = TRI_LOWER;
        g.Cb = Wc1.data(); g.ldc = a;
        g.sk_wsb = SK.data(); g.sk_cap = blk;
        BTA_TRY(gemm_f64(g, s));
      }
      {  // Z_C = -Z_T F_C, in place of L_Ci
        Gemm g; g.M = a; g.N = ld; g.K = a; g.batch = c;
        g.Ab = cp(T); g.lda = a; g.Bb = cp(Wc1); g.ldb = a;
        g.Cb = Ci.data(); g.ldc = a; g.alpha = -1.0;
        BTA_TRY(gemm_f64(g, s));
      }
      if (hasB) {  // Z_C -= Z_C,i+1 F_B
        auto Cn = ptrs(grp, [&](int z) { return Cb(z, i + 1); });
        auto W1g = ptrs(grp, [&](int z) { return it[z].ws.W1; });
        Gemm g; g.M = a; g.N = ld; g.K = ld; g.batch = c;
        g.Ab = cp(Cn); g.lda = a; g.Bb = cp(W1g); g.ldb = ld;
        g.Cb = Ci.data(); g.ldc = a; g.Cinb = cp(Ci); g.ldcin = a; g.alpha = -1.0;
        g.beta = 1.0;
        g.sk_wsb = SK.data(); g.sk_cap = blk;
        BTA_TRY(gemm_f64(g, s));
      }
    }
    // Z_D = L_Di^{-T} L_Di^{-1} (lower part); emulated it follows F_B, whose planes of L_Di
    // serve it
    auto inverse_gram = [&]() -> bta_status {
      Gemm g; g.M = ld; g.N = ld; g.K = ld; g.batch = M;
      g.Ab = cp(Di); g.lda = ld; g.transA = 1; g.triA = TRI_UPPER;
      g.Bb = cp(Di); g.ldb = ld; g.triB = TRI_LOWER;
      g.Cb = ZD.data(); g.ldc = ld; g.out_lower = 1;
      if (!emu || !hasB) return big_product(g, it, G.all, precision, s);
      for (size_t q = 0; q < G.all.size(); ++q) {
        const int z = G.all[q];
        Gemm h = g;
        h.batch = 1;
        h.Ab = h.Bb = nullptr;
        h.Cb = nullptr;
        h.A = h.B = Di[q];
        h.C = ZD[q];
        h.b_kept = ld + (fused(z) ? it[z].q.a : 0);
        BTA_TRY(emulate(z, h));
      }
      return BTA_OK;
    };
    if (emu) BTA_TRY(inverse_gram());
    if (hasB) {
      auto Dn = ptrs(G.all, [&](int z) { return D(z, i + 1); });
      if (emu) {
        // Z_B = -Z_D,i+1 F_B; an arrow carried along as a 2 x 2 block product:
        // [Z_B; Z_C] = -[Z_D,i+1, Z_C,i+1^T; Z_C,i+1, Z_T] [F_B; F_C],
        // i.e. also Z_B -= Z_C,i+1^T F_C and Z_C = -Z_C,i+1 F_B - Z_T F_C
        for (size_t q = 0; q < G.all.size(); ++q) {
          const int z = G.all[q];
          Gemm g; g.M = ld; g.N = ld; g.K = ld;
          g.A = Dn[q]; g.lda = ld; g.B = W1[q]; g.ldb = ld;
          g.C = ZB[q]; g.ldc = ld; g.alpha = -1.0;
          if (fused(z)) {
            const int a = it[z].q.a;
            const double* Cn = Cb(z, i + 1);
            g.M = ld + a; g.K = ld + a; g.a_rows = ld; g.a_k = ld;
            g.A12 = {Cn, a, 1}; g.A21 = {Cn, a, 0}; g.A22 = {it[z].q.T, a, 0};
            g.b_k = ld; g.B21 = {it[z].ws.Wc1, a, 0};
            g.c_rows = ld; g.C2 = Cb(z, i); g.ldc2 = a;
          }
          BTA_TRY(emulate(z, g));
        }
      } else {  // Z_B = -Z_D,i+1 F_B
        Gemm g; g.M = ld; g.N = ld; g.K = ld; g.batch = M;
        g.Ab = cp(Dn); g.lda = ld; g.Bb = cp(W1); g.ldb = ld;
        g.Cb = ZB.data(); g.ldc = ld; g.alpha = -1.0;
        BTA_TRY(big_product(g, it, G.all, precision, s));
      }
      for (const auto& grp : G.arrow) {  // Z_B -= Z_C,i+1^T F_C
        if (fused(grp[0])) continue;
        const int a = it[grp[0]].q.a, c = (int)grp.size();
        auto Cn = ptrs(grp, [&](int z) { return Cb(z, i + 1); });
        auto Wc1 = ptrs(grp, [&](int z) { return it[z].ws.Wc1; });
        auto W2g = ptrs(grp, [&](int z) { return low ? it[z].ws.W2 : B(z, i); });
        Gemm g; g.M = ld; g.N = ld; g.K = a; g.batch = c;
        g.Ab = cp(Cn); g.lda = a; g.transA = 1; g.Bb = cp(Wc1); g.ldb = a;
        g.Cb = W2g.data(); g.ldc = ld; g.Cinb = cp(W2g); g.ldcin = ld; g.alpha = -1.0;
        g.beta = 1.0;
        BTA_TRY(gemm_f64(g, s));
      }
    }
    if (!emu) BTA_TRY(inverse_gram());
    if (hasB) {  // Z_D -= Z_B^T F_B
      if (emu) {  // an arrow carried along extends K: Z_D -= [Z_B; Z_C]^T [F_B; F_C]
        for (size_t q = 0; q < G.all.size(); ++q) {
          const int z = G.all[q];
          Gemm g; g.M = ld; g.N = ld; g.K = ld;
          g.A = ZB[q]; g.lda = ld; g.transA = 1; g.B = W1[q]; g.ldb = ld;
          g.C = ZD[q]; g.ldc = ld; g.Cin = ZD[q]; g.ldcin = ld; g.alpha = -1.0; g.beta = 1.0;
          g.out_lower = 1;
          g.b_kept = ld + (fused(z) ? it[z].q.a : 0);   // F_B's planes from Z_B's product
          if (fused(z)) {
            const int a = it[z].q.a;
            g.K = ld + a; g.a_k = ld; g.A12 = {Cb(z, i), a, 1};
            g.b_k = ld; g.B21 = {it[z].ws.Wc1, a, 0};
          }
          BTA_TRY(emulate(z, g));
        }
      } else {
        Gemm g; g.M = ld; g.N = ld; g.K = ld; g.batch = M;
        g.Ab = cp(ZB); g.lda = ld; g.transA = 1; g.Bb = cp(W1); g.ldb = ld;
        g.Cb = ZD.data(); g.ldc = ld; g.Cinb = cp(ZD); g.ldcin = ld; g.alpha = -1.0; g.beta = 1.0;
        g.out_lower = 1;
        BTA_TRY(big_product(g, it, G.all, precision, s));
      }
    }
    for (const auto& grp : G.arrow) {  // Z_D -= Z_C^T F_C
      if (hasB && fused(grp[0])) continue;
      const int a = it[grp[0]].q.a, c = (int)grp.size();
      auto Wc1 = ptrs(grp, [&](int z) { return it[z].ws.Wc1; });
      auto Ci = ptrs(grp, [&](int z) { return Cb(z, i); });
      auto ZDg = ptrs(grp, [&](int z) { return over ? D(z, i) : it[z].ws.W3; });
      Gemm g; g.M = ld; g.N = ld; g.K = a; g.batch = c;
      g.Ab = cp(Ci); g.lda = a; g.transA = 1; g.Bb = cp(Wc1); g.ldb = a;
      g.Cb = ZDg.data(); g.ldc = ld; g.Cinb = cp(ZDg); g.ldcin = ld; g.alpha = -1.0; g.beta = 1.0;
      g.out_lower = 1;
      BTA_TRY(gemm_f64(g, s));
    }
    BTA_TRY(mirror_batch(M, cp(ZD), ld, Di.data(), ld, ld, s));   // Z_D (full)
    if (hasB && low)   // Z_B is not kept: reduce it here
      for (int z = 0; z < m; ++z) {
        const SelinvFuse* fz = it[z].fuse;
        if (!fz) continue;
        const int b = coupling_of(it[z], i);
        BTA_TRY(launch_pattern_dot(*fz->md, it[z].ws.W2, 0, b, 1,
                                   fz->PB + (int64_t)b * pattern_doubles(*fz->md), s));
      }
    BTA_SWEEP_MARK(s, 5, i);
  }
  return BTA_OK;
}

bta_status selinv_sums(const SweepItem* it, int m, cudaStream_t s) {
  for (int z = 0; z < m; ++z) {
    const SelinvFuse* fz = it[z].fuse;
    if (!fz) continue;
    const ModelDev& md = *fz->md;
    const bta_desc& q = it[z].q;
    BTA_TRY(launch_pattern_dot(md, q.D, fz->counts, 0, q.n, fz->PD, s));
    if (q.B && q.n > 1) BTA_TRY(launch_pattern_dot(md, q.B, 0, 0, q.n - 1, fz->PB, s));
    if (q.a > 0 && fz->PC) BTA_TRY(launch_arrow_dot(md, q.C, q.n, fz->PC, s));
  }
  return BTA_OK;
}

bta_status selinv_sweep(const bta_desc& q, const SweepWs& ws, const SelinvFuse* fuse,
                        cudaStream_t s) {
  SweepItem item;
  item.q = q; item.ws = ws; item.fuse = fuse;
  BTA_TRY(selinv_sweep_multi(&item, 1, s));
  return selinv_sums(&item, 1, s);
}

}  // namespace bta
