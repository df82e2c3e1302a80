// Diagonal-block Cholesky factor and inverse as one persistent kernel over a
// tile task graph (FP64 results, 32 x 32 tiles, p = n / 32 tile rows).  Its
// tile products run as FP64 FMAs, or (the tensor-core modes, kernel
// instance TC) emulated in FP64 from BF16 slices on warp-level tensor-core
// MMAs (tile_mm_oz); pivots, reciprocals and log-dets stay in FP64.
//
// Same contract as the recursive potrf_inv: on return the lower triangle of
// A holds L^{-1} (A = L L^T), one log-det slot per diagonal tile, the failure
// code on a non-positive pivot.  The recursion issues ~5 p dependent
// launches per block, each using a sliver of the GPU; here the whole block
// is one launch whose CTAs pull tasks from a list in topological order and
// start each as soon as the tiles it reads are final.
//
// Tasks, for step k = 0..p-1 (A's lower tiles are reused in place: first the
// trailing matrix W, then the inverse's accumulator R, then the inverse X):
//   H         the chain, one task per block run by one CTA: for c = 0..p-1,
//             L_{c,c-1} = W_{c,c-1} X_{c-1,c-1}^T, W_cc -= L L^T, and the leaf
//             on W_cc (D / unit-L elimination with its inverse) -> X_cc =
//             L_cc^{-1} into A_cc, log-det slot c; X_cc stays in shared
//             memory for the next step
//   S(i,k)    L_ik = W_ik X_kk^T, i >= k+2           (into the scratch Lt)
//   G(k,j)    X_kj = X_kk R_kj            (j < k; R_kj = -sum_m L_km X_mj)
//   U(i,j,k)  W_ij -= L_ik L_jk^T         (k < j <= i, not (k+1,k+1); column k+1 first)
//   V(i,j,k)  R_ij -= L_ik X_kj           (k < i, j <= k; R_ij = -L_ij X_jj at k = j)
// A task waits only for tasks earlier in the list, which running CTAs hold,
// so the graph always drains.  Per-tile counters (W updates applied, R
// updates applied, F/S/G done) are published with release stores after the
// tile is written and read with acquire loads; tile data are read through
// L2 (cp.async.cg).
//
// A CTA is three parties.  Warp 8 fetches: it takes a ticket, waits for the tiles the
// task reads and loads them into one of two stages, so that the next task's ticket,
// waits (three L2 round trips) and loads run behind the current task's products.  Warps
// 0-7 compute, and store the result.  Warp 9 publishes: its release store waits for
// the stores to be visible (~900 clocks) while the others go on; the compute warps'
// barrier makes it cumulative.  On the chain the fetcher brings the next step's W tiles
// while the leaf runs (in the tensor-core modes split into slices) and the publisher
// sums the pivots' logs.  Stages change hands through mbarriers.
//
// Every wait is bounded by a globaltimer limit (2 s); on expiry the CTA raises a shared
// abort flag, writes BTA_ERR_TIMEOUT into the block's failure word (which otherwise
// holds -1 or the index of a block with a non-positive pivot) and returns, and every
// other CTA returns at its next wait.  A test switch (bta_set_wait_limit) lowers the
// limit and makes the chain wait on a counter nothing sets, so that this path runs
// without a fault.
#include <algorithm>
#include <cstdlib>
#include <vector>

#include <cuda_bf16.h>

#include "common.cuh"
#include "ozaki_digits.cuh"

// Timeline hooks of the chain (compile-time empty in the library): a
// measurement build that includes this file may define DAG_TRACE(event, step)
// before the include to stamp the chain's phases of each diagonal step:
// 0 the step's inputs are final (waits done), 1 the triangular product done,
// 2 the symmetric update done, 3 the leaf done, 4 the step published; and of the two bulk
// tasks that the chain's step k + 2 waits for, S(k+2,k) and U(k+2,k+1,k): 5 / 8 the task's
// tiles are final, 6 / 9 in place, 7 / 10 its result published, 11 the fetcher has seen
// step c's tiles final.
#ifndef DAG_TRACE
#define DAG_TRACE(event, step) ((void)0)
#endif

namespace bta {
namespace {

constexpr int T = kPad;                 // tile size
constexpr int kTP = T + 2;              // column pitch of a tile in shared memory (16-byte columns)
constexpr int kDagThreads = 256;        // compute threads (warps 0-7)
constexpr int kDagFetch = 8, kDagPublish = 9;   // service warps
constexpr int kDagAllThreads = kDagThreads + 64;
constexpr int kMaxP = 160;              // tile rows supported (ld <= 5120)

enum : int { TK_H = 0, TK_S = 1, TK_G = 2, TK_U = 3, TK_V = 4, TK_END = 5 };

struct DagInst {
  double* A;       // n x n block, ld
  double* Lt;      // scratch: L tiles (i > k), tile (i,k) at Lt + (i(i-1)/2 + k)*T*T
  int* st;         // counters: cntW[p*p], cntR[p*p], doneF[p], doneS[p*p], doneG[p*p]
  double* slots;   // log-det slots (p)
  int32_t* fail;
  int32_t code;
};

struct DagArgs {
  int p, ld, cnt;
  int total;                // tasks over all instances
  int* counter;             // global task ticket
  int* abort;               // shared abort flag
  int* smbusy;              // per SM: chain tasks running there (see TK_H)
  int yield;                // bulk tasks wait while a chain task holds their SM
  int vec;                  // the blocks are 16-byte aligned
  int stall;                // test switch: the chain waits on a counter nothing sets
  unsigned long long wait_ns;   // bound of every wait
  int off[kMaxP + 1];       // task offset of each step within one instance
  DagInst inst[kMaxBatch];
};

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int sm_id() {
  int v;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(v));
  return v;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Thread 0 waits until *p >= need (bounded by wait_ns); false on timeout / abort.
__device__ bool wait_ge(const int* p, int need, int* abort, unsigned long long wait_ns) {
  if (ld_acquire(p) >= need) return true;
  const unsigned long long t0 = now_ns();
  while (true) {
    __nanosleep(64);
    if (ld_acquire(p) >= need) return true;
    if (ld_acquire(abort)) return false;
    if (now_ns() - t0 > wait_ns) {
      atomicExch(abort, 1);
      return false;
    }
  }
}

// Tile (r, c) of the n x n block, column-major with leading dimension ld.
__device__ __forceinline__ double* tile(double* A, int ld, int r, int c) {
  return A + (int64_t)c * T * ld + (int64_t)r * T;
}

// A tile in shared memory: column-major, element (r, c) at S[c][r].
using Tile = double (*)[kTP];
__device__ __forceinline__ double& at(Tile S, int r, int c) { return S[c][r]; }

// One warp starts the load of a 32 x 32 tile (column-major, ld) through L2: 16
// asynchronous copies a lane, so that every tile of a task takes one round trip together
// (load_wait) and no registers.  A block that is not 16-byte aligned (a caller's; vec = 0)
// goes through registers.
__device__ __forceinline__ void load_tile(Tile S, const double* src, int ld, int vec) {
  const int lane = threadIdx.x & 31, r = 2 * (lane & 15);
  if (!vec) {
    for (int c = 0; c < T; ++c) S[c][lane] = __ldcg(src + (int64_t)c * ld + lane);
    return;
  }
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int c = 2 * q + (lane >> 4);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(&S[c][r])),
                 "l"(src + (int64_t)c * ld + r)
                 : "memory");
  }
}
__device__ __forceinline__ void load_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
}
// Zeros above the diagonal (one warp).
__device__ __forceinline__ void zero_upper(Tile S) {
  const int r = threadIdx.x & 31;
  for (int c = r + 1; c < T; ++c) S[c][r] = 0.0;
}

// Barrier of the compute warps.
__device__ __forceinline__ void compute_bar() {
  asm volatile("bar.sync 2, 256;" ::: "memory");
}
// ... which also tells them whether v holds in all of them: a decision that all share.
__device__ __forceinline__ bool compute_all(bool v) {
  int r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n"
      " barrier.cta.red.and.pred q, 2, 256, p;\n selp.s32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((int)v)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void store_tile(double* dst, int ld, Tile S, bool lower) {
  for (int e = threadIdx.x; e < T * T; e += kDagThreads) {
    const int r = e % T, c = e / T;
    if (!lower || r >= c) dst[(int64_t)c * ld + r] = at(S, r, c);
  }
}

// at(out, r, c) (+)= sign * sum_m at(X, r, m) * Y'[m][c], with Y' = Y^T when ytrans.
// 256 threads, each 2 x 2 outputs.
__device__ __forceinline__ void tile_mm(Tile X, Tile Y, bool ytrans,
                                        Tile out, double sign, bool accumulate) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double a00 = 0.0, a01 = 0.0, a10 = 0.0, a11 = 0.0;
#pragma unroll 8
  for (int m = 0; m < T; ++m) {
    const double x0 = at(X, tx, m), x1 = at(X, tx + 16, m);
    const double y0 = ytrans ? at(Y, ty, m) : at(Y, m, ty);
    const double y1 = ytrans ? at(Y, ty + 16, m) : at(Y, m, ty + 16);
    a00 = fma(x0, y0, a00); a01 = fma(x0, y1, a01);
    a10 = fma(x1, y0, a10); a11 = fma(x1, y1, a11);
  }
  if (accumulate) {
    at(out, tx, ty) += sign * a00; at(out, tx, ty + 16) += sign * a01;
    at(out, tx + 16, ty) += sign * a10; at(out, tx + 16, ty + 16) += sign * a11;
  } else {
    at(out, tx, ty) = sign * a00; at(out, tx, ty + 16) = sign * a01;
    at(out, tx + 16, ty) = sign * a10; at(out, tx + 16, ty + 16) = sign * a11;
  }
}

// at(out, r, c) = sum_{m <= c} at(W, r, m) at(Y, c, m) = (W Y^T)[r][c] for lower-triangular Y
// (its upper part is not read).  Same thread layout as tile_mm; the m range
// of a thread's columns (ty, ty + 16) is uniform within a warp, so the
// skipped half of the products issues no instructions.
__device__ __forceinline__ void tile_mm_lt(Tile W, Tile Y,
                                           Tile out) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double a00 = 0.0, a01 = 0.0, a10 = 0.0, a11 = 0.0;
  for (int m = 0; m <= ty; ++m) {
    const double x0 = at(W, tx, m), x1 = at(W, tx + 16, m);
    const double y0 = at(Y, ty, m), y1 = at(Y, ty + 16, m);
    a00 = fma(x0, y0, a00); a01 = fma(x0, y1, a01);
    a10 = fma(x1, y0, a10); a11 = fma(x1, y1, a11);
  }
  for (int m = ty + 1; m <= ty + 16; ++m) {
    const double y1 = at(Y, ty + 16, m);
    a01 = fma(at(W, tx, m), y1, a01);
    a11 = fma(at(W, tx + 16, m), y1, a11);
  }
  at(out, tx, ty) = a00; at(out, tx, ty + 16) = a01;
  at(out, tx + 16, ty) = a10; at(out, tx + 16, ty + 16) = a11;
}

// at(W, r, c) -= sum_m at(L, r, m) at(L, c, m) on the lower triangle (r >= c): threads
// 0..135 each own one 2 x 2 block of the 16 x 16 block triangle, so only 5
// of the 8 warps issue FMAs.  Upper entries of diagonal blocks get the same
// update (W is symmetric; only its lower part is read afterwards).
__device__ __forceinline__ void tile_syrk_lower(Tile L, Tile W) {
  const int b = threadIdx.x;
  if (b >= 136) return;
  int bi = 0;
  while ((bi + 1) * (bi + 2) / 2 <= b) ++bi;
  const int bj = b - bi * (bi + 1) / 2;
  const int r = 2 * bi, c = 2 * bj;
  double a00 = 0.0, a01 = 0.0, a10 = 0.0, a11 = 0.0;
#pragma unroll 8
  for (int m = 0; m < T; ++m) {
    const double x0 = at(L, r, m), x1 = at(L, r + 1, m), y0 = at(L, c, m), y1 = at(L, c + 1, m);
    a00 = fma(x0, y0, a00); a01 = fma(x0, y1, a01);
    a10 = fma(x1, y0, a10); a11 = fma(x1, y1, a11);
  }
  at(W, r, c) -= a00; at(W, r, c + 1) -= a01;
  at(W, r + 1, c) -= a10; at(W, r + 1, c + 1) -= a11;
}

// ---- emulated-FP64 tile products (tensor-core modes) -----------------------
// out (+)= sign * X op(Y) on 32 x 32 tiles, op(Y) = Y^T (ytrans) or Y, to FP64
// accuracy from 8 BF16 digit slices per operand on warp-level tensor-core
// MMAs (mma.sync m16n8k16): on GB300 these run ~1900 BF16 flop per clock per
// SM against ~1.6 FP64 FMAs, so the 36 slice-pair products of a tile cost
// ~1.2 k clocks where its 32^3 FP64 FMAs cost ~20 k.  A row is scaled to
// 56-bit integers by its exponent bound and written in signed base-128 digits
// (Ozaki's error-free splitting, fixed point); a level L = i + j of slice pairs
// sums to an integer |S_L| < 2^21 over K = 32, exact in FP32; levels 0..5 are
// added as 64-bit integers in units of level 5, levels 6 and 7 rounded to that
// unit, and the FP64 result assembled by integer operations.  Levels from 8 on
// are dropped.  Error: with u, w the powers of two above a row's and a column's largest
// entries, level L's unit is 2^(-14 - 7 L) u w.  The rounding to level 5's unit is off by
// 2^-50 u w, the dropped levels by at most 7 2^17 units of level 8 (and 1 % more)
// = 2^-50.2 u w, the 56-bit operands by 2^-51 u w: 2^-48.7 u w in all for 32 terms, where
// the bound of FP64 FMAs is 2^-43 times the largest entries' product.  Unlike theirs it is
// absolute in a row and column of a tile: small entries keep fewer bits.
constexpr int kOzPitch = 40;                      // bf16 a slice row: 80 bytes, conflict-free ldmatrix
constexpr int kOzPlane = T * kOzPitch;            // one 32 x 32 slice
constexpr int kOzTileSmem = 2 * 8 * kOzPlane * 2 + 2 * T * 4;   // both operands' slices, exponents

struct OzTile {
  __nv_bfloat16* xp;   // [8][32][kOzPitch]: slices of the rows of X
  __nv_bfloat16* yp;   // [8][32][kOzPitch]: slices of the rows of op(Y)^T
  int* ex;             // [32] row exponents of X
  int* ey;             // [32] row exponents of op(Y)^T
};

// Slices of a 32 x 32 matrix (element (r, k) = get(r, k)) into planes[8][r][.]
// and its row exponent bounds e[r].  A half-warp takes a row, a lane its elements
// k and k + 16, which sit side by side in the slice row (both operands of a
// product use this order of k); the two rows of a warp are four apart, so that
// their 4-byte stores fall on different banks.
// part 0..7: the eighth of the rows the calling warp takes.
template <class Get>
__device__ __forceinline__ void oz_split(Get get, __nv_bfloat16* planes, int* e, int part) {
  const int lane = threadIdx.x & 31;
  const int k = lane & 15;
  const int r0 = (part & 3) + 16 * (part >> 2) + 4 * (lane >> 4);
  double v[2][2];
  int er[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    v[q][0] = get(r0 + 8 * q, k);
    v[q][1] = get(r0 + 8 * q, k + 16);
    er[q] = max((int)((__double_as_longlong(v[q][0]) >> 52) & 0x7FF),
                (int)((__double_as_longlong(v[q][1]) >> 52) & 0x7FF));
  }
#pragma unroll
  for (int o = 8; o; o >>= 1)
#pragma unroll
    for (int q = 0; q < 2; ++q) er[q] = max(er[q], __shfl_xor_sync(0xffffffffu, er[q], o));
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int r = r0 + 8 * q;
    float d0[8], d1[8];
    oz::digits(v[q][0], er[q], d0);
    oz::digits(v[q][1], er[q], d1);
    uint32_t* y = reinterpret_cast<uint32_t*>(planes + r * kOzPitch) + k;
#pragma unroll
    for (int j = 0; j < 8; ++j)   // |digit| <= 128: its BF16 pattern is the upper half
      y[j * (kOzPlane / 2)] = __byte_perm(__float_as_uint(d0[j]), __float_as_uint(d1[j]), 0x7632);
    if (k == 0) e[r] = er[q];
  }
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The products of the slices and their combination: warp w computes the
// 16 x 8 output block (rows 16 (w / 4).., columns 8 (w % 4)..).
__device__ __forceinline__ void oz_combine(const __nv_bfloat16* xp, const __nv_bfloat16* yp,
                                           const int* ex, const int* ey, Tile out,
                                           double sign, bool accumulate) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int mt = warp >> 2, nt = warp & 3;
  // one accumulator per level, the pairs issued slice by slice of A so that
  // consecutive MMAs go to different accumulators (no dependent chain); one 16-wide
  // K step at a time, which keeps the kernel at two CTAs an SM
  float c[8][4];
#pragma unroll
  for (int L = 0; L < 8; ++L)
#pragma unroll
    for (int q = 0; q < 4; ++q) c[L][q] = 0.f;
  // ldmatrix rows: A's four 8 x 8 blocks (rows 0-7 / 8-15 by k 0-7 / 8-15); B's two
  // (columns 0-7 by k 0-7 / 8-15) of two slices
  const int ar = 16 * mt + (lane & 7) + ((lane >> 3) & 1) * 8, ac = (lane >> 4) * 8;
  const int br = 8 * nt + (lane & 7), bc = ((lane >> 3) & 1) * 8, bs = lane >> 4;
  const uint32_t xb = (uint32_t)__cvta_generic_to_shared(xp) + 2u * (ar * kOzPitch + ac);
  const uint32_t yb =
      (uint32_t)__cvta_generic_to_shared(yp) + 2u * (bs * kOzPlane + br * kOzPitch + bc);
#pragma unroll
  for (int ks = 0; ks < 2; ++ks) {
    uint32_t a[8][4], b[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) ldsm_x4(yb + 2u * (2 * j * kOzPlane + 16 * ks), b[j]);
#pragma unroll
    for (int j = 0; j < 8; ++j) ldsm_x4(xb + 2u * (j * kOzPlane + 16 * ks), a[j]);
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; i + j < 8; ++j)
        mma_bf16(c[i + j], a[i], b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]);
  }
  // |S_L| < 2^21: to integers by the exact FP32 rounding against 1.5 2^23 (no
  // 64-bit conversions, which GB300 runs at its FP64 rate); two levels 7 bits
  // apart share one 32-bit integer, then
  // tot = S_0 2^35 + S_1 2^28 + ... + S_5 + round(S_6 2^-7 + S_7 2^-14).
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int sl[6];
#pragma unroll
    for (int L = 0; L < 6; ++L) sl[L] = oz::f2i_small(c[L][q]);
    const int r67 = oz::f2i_small(fmaf(c[6][q], 0.0078125f, c[7][q] * 0.00006103515625f));
    const long long tot = ((long long)(sl[0] * 128 + sl[1]) << 28) +
                          ((long long)(sl[2] * 128 + sl[3]) << 14) + (sl[4] * 128 + sl[5] + r67);
    const int r = 16 * mt + g + (q >> 1) * 8, cc = 8 * nt + 2 * t + (q & 1);
    // a = sum_j d_j 2^(ex - 1029 - 7 j): the integer's unit is level 5's
    double v = oz::compose(tot, ex[r] + ey[cc] - 2093);
    if (sign < 0.0) v = -v;
    at(out, r, cc) = accumulate ? at(out, r, cc) + v : v;
  }
}

// All compute threads; out must not alias X or Y.
__device__ __forceinline__ void tile_mm_oz(Tile X, Tile Y, bool ytrans, Tile out, double sign,
                                           bool accumulate, const OzTile& z) {
  const int warp = threadIdx.x >> 5;
  oz_split([&](int r, int k) { return at(X, r, k); }, z.xp, z.ex, warp);
  oz_split([&](int n, int k) { return ytrans ? at(Y, n, k) : at(Y, k, n); }, z.yp, z.ey, warp);
  compute_bar();
  oz_combine(z.xp, z.yp, z.ex, z.ey, out, sign, accumulate);
}

struct Task {
  int type, i, j, k;
};

// Number of tasks of step k (see potrf_dag_batch for the list order).
__host__ __device__ inline int step_tasks(int p, int k) {
  const int nS = p - 2 - k > 0 ? p - 2 - k : 0;
  const int nU = (p - 1 - k) * (p - k) / 2 - (k + 1 < p ? 1 : 0);
  const int nV = (p - 1 - k) * (k + 1);
  return nS + k + nU + nV;
}

// Decode task index l of one instance.  Index 0 is the chain H; then for
// each step k: S(i,k) for i >= k+2, G(k,j), U(i,j,k) (column k+1 first,
// without (k+1,k+1), which the chain applies) and V(i,j,k).
__device__ Task decode(const DagArgs& g, int l) {
  const int p = g.p;
  Task t{TK_H, 0, 0, 0};
  if (l == 0) return t;
  l -= 1;
  int lo = 0, hi = p - 1;
  while (lo < hi) {   // largest k with off[k] <= l
    const int mid = (lo + hi + 1) >> 1;
    if (g.off[mid] <= l) lo = mid; else hi = mid - 1;
  }
  const int k = lo;
  int r = l - g.off[k];
  t.k = k;
  const int nS = p - 2 - k > 0 ? p - 2 - k : 0;
  if (r < nS) { t.type = TK_S; t.i = k + 2 + r; t.j = k; return t; }
  r -= nS;
  if (r < k) { t.type = TK_G; t.i = k; t.j = r; return t; }
  r -= k;
  const int nU = (p - 1 - k) * (p - k) / 2 - (k + 1 < p ? 1 : 0);
  if (r < nU) {   // columns j = k+1.. in order, rows i = j..p-1, skipping (k+1, k+1)
    int j = k + 1;
    int len = p - j - 1;            // column k+1 without its diagonal tile
    while (r >= len) { r -= len; ++j; len = p - j; }
    t.type = TK_U; t.j = j; t.i = (j == k + 1 ? j + 1 : j) + r; return t;
  }
  r -= nU;
  t.type = TK_V;   // rows i = k+1.. in order, columns j = 0..k
  t.i = k + 1 + r / (k + 1);
  t.j = r % (k + 1);
  return t;
}

// 1 / v to FP64 accuracy by one third-order step (Householder's iteration,
// r (1 + e + e^2) with e = 1 - v r) from the FP32 reciprocal of v's leading
// bits, all of it in integers: a GB300 FP64 instruction, conversions included,
// has ~72 clocks of latency, a dependent 32 x 32 -> 64 bit multiply ~10.  With
// the significand M = v 2^52 (53 bits) and the seed R = r 2^24 (24 bits),
// e 2^76 = 2^76 - M R fits 64 bits (|e| <= 2^-22), so its low word is exact;
// the result is rounded once from 56 bits (error within 0.53 of the last place).
// Values outside the seed's exponent range use the division.
__device__ __forceinline__ double recip(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const int ef = (int)((hi >> 20) & 0x7FF);
  if (ef < 1023 - 100 || ef > 1023 + 100) return 1.0 / v;
  const unsigned mh = (hi & 0xFFFFFu) | 0x100000u;   // M = mh 2^32 + lo
  // seed in [1/2, 1): of the significand's leading 24 bits
  float rf;
  asm("rcp.approx.ftz.f32 %0, %1;"
      : "=f"(rf)
      : "f"(__uint_as_float(0x3F800000u | ((hi & 0xFFFFFu) << 3) | (lo >> 29))));
  const unsigned R = (min(max(__float_as_uint(rf), 0x3F000000u), 0x3F7FFFFFu) & 0x7FFFFFu) |
                     0x800000u;
  const unsigned long long mr =
      (unsigned long long)lo * R + ((unsigned long long)(mh * R) << 32);   // M R mod 2^64
  long long e = (long long)(0ull - mr);                                    // e 2^76
  const int eh = (int)(e >> 24);                                           // |eh| <= 2^30
  e += ((long long)eh * eh) >> 28;                                         // e + e^2
  const int th = (int)(e >> 24);
  const unsigned tl = (unsigned)e & 0xFFFFFFu;
  // r (1 + e + e^2) 2^56, in [2^55, 2^56]
  const long long corr = (long long)th * (int)R + (long long)(((unsigned long long)tl * R) >> 24);
  const unsigned long long q = ((unsigned long long)R << 32) + (unsigned long long)(corr >> 20);
  const unsigned long long m = (q + 4) >> 3;   // 53 bits, or 2^53
  // v = M 2^(ef - 1075): 1 / v = m 2^-53 2^(1023 - ef)
  return __longlong_as_double((long long)((b & 0x8000000000000000ull) |
                                          ((((unsigned long long)(2045 - ef)) << 52) +
                                           (m - (1ull << 52)))));
}

// d^{-1/2} to FP64 accuracy: FP32 seed of the narrowed value widened by
// integer operations, then y (1 + e/2 + 3e^2/8) with e = 1 - d y^2 (relative
// error ~e^3): five dependent FP64 operations.  Outside the seed's range the
// library square root and division.
__device__ __forceinline__ double rsqrt_fp64(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int e = (int)((b >> 52) & 0x7FF);
  if (!(d > 0.0) || e < 1023 - 100 || e > 1023 + 100) return 1.0 / sqrt(d);
  const unsigned f = ((unsigned)(e - 1023 + 127) << 23) | (unsigned)((b >> 29) & 0x7FFFFFu);
  float yf;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__uint_as_float(f)));
  const unsigned rb = __float_as_uint(yf);
  const unsigned long long db = ((unsigned long long)(((rb >> 23) & 0xFF) - 127 + 1023) << 52) |
                                ((unsigned long long)(rb & 0x7FFFFFu) << 29);
  const double y = __longlong_as_double((long long)db);
  const double err = fma(-d, y * y, 1.0);
  return fma(y, fma(0.375, err, 0.5) * err, y);
}

// Leaf on smem tile S (lower, W_kk): D / unit-L elimination carrying the
// inverse of the unit-L factor in X, then X = D^{-1/2} (unit L)^{-1} =
// L_kk^{-1} (lower part; its upper part is not written); the pivots d_i stay in
// piv[] (leaf_logdet sums their logs, off the critical path).
//
// Pivot j eliminates column j with the multipliers l_ij = S_ij / d_j:
// S_ik -= l_ij S_kj (j < k <= i) and X_ik -= l_ij X_jk (k <= j < i).  Warp 0
// runs one pivot ahead: while warps 1-7 apply pivot j to columns
// k >= j+2 and to X, it applies pivot j to column j+1, takes d_{j+1}, its
// reciprocal and the next multipliers.  A position (i, k) belongs to one thread
// for the whole leaf, which holds S_ik and, from pivot k on, X_ik in a register;
// only what others read goes through shared memory, double buffered by the
// pivot's parity: the multipliers and the column of the pivot (from warp 0),
// column j+2 (for warp 0) and row j+1 of X.  So each pivot costs one barrier, and the
// serial chain is one FMA, the integer reciprocal and one multiply.  An SM sub-partition
// issues one FP64 warp instruction per 64 clocks, so of the 17 warps' worth of
// positions warp 4, which shares warp 0's, takes two and each other sub-partition five.
// Measured: 10.4 us of a chain step's 17.4 (512 rows, tensor-core modes).
struct LeafBuf {
  double l[2][T], v[2][T], x[2][T], s[2][T];
};

__device__ __forceinline__ void leaf(Tile S, Tile X, LeafBuf& B,
                                     double* piv, double* rs) {
  constexpr int kPos = T * (T + 1) / 2;   // lower-triangle positions, row by row
  constexpr int kBulk = kDagThreads - 32;   // warps 1-7
  constexpr int kPer = (kPos + kBulk - 1) / kBulk;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp == 0) {
    double v = at(S, lane, 0);
    double d = __shfl_sync(0xffffffffu, v, 0);
    double l = v * recip(d);
    B.l[0][lane] = l;
    B.v[0][lane] = v;
    B.s[0][lane] = at(S, lane, 1);
    if (lane == 0) {
      B.x[0][0] = 1.0;
      piv[0] = d;
    }
    compute_bar();
    for (int j = 0; j < T - 1; ++j) {
      // column c = j+1 with pivot j, then pivot c and its multipliers
      const int c = j + 1, p = c & 1;
      const double vc = __shfl_sync(0xffffffffu, v, c);
      v = fma(-l, vc, B.s[j & 1][lane]);
      d = __shfl_sync(0xffffffffu, v, c);
      l = v * recip(d);
      B.l[p][lane] = l;
      B.v[p][lane] = v;
      if (lane == 0) piv[c] = d;
      compute_bar();
    }
    rs[lane] = rsqrt_fp64(piv[lane]);   // rows scale by d_i^{-1/2}
    compute_bar();
  } else {
    // warps 1-3, 5-7 and then 4: the last positions go to the first three
    const int bt = (warp < 4 ? warp - 1 : warp == 4 ? 6 : warp - 2) * 32 + lane;
    int pi[kPer], pk[kPer];
    double val[kPer];
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int q = bt + kBulk * r;
      int i = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
      if (i * (i + 1) / 2 > q) --i;
      if ((i + 1) * (i + 2) / 2 <= q) ++i;
      pi[r] = q < kPos ? i : -1;
      pk[r] = q < kPos ? q - i * (i + 1) / 2 : 0;
      val[r] = q < kPos ? at(S, i, pk[r]) : 0.0;
    }
    compute_bar();
    for (int j = 0; j < T - 1; ++j) {
      const int p = j & 1;
      double src[kPer], lv[kPer];
#pragma unroll
      for (int r = 0; r < kPer; ++r) {
        if (pi[r] > j) {
          src[r] = pk[r] > j ? B.v[p][pk[r]] : B.x[p][pk[r]];
          lv[r] = B.l[p][pi[r]];
        }
      }
#pragma unroll
      for (int r = 0; r < kPer; ++r) {
        const int i = pi[r], k = pk[r];
        if (i > j) {
          // (k == j+1, warp 0's column, is computed here too but not used: at
          // pivot k the position turns into X_ik, which starts from 0)
          val[r] = fma(-lv[r], src[r], k == j ? 0.0 : val[r]);
          if (k == j + 2) B.s[p ^ 1][i] = val[r];
          if (i == j + 1) B.x[p ^ 1][k] = k == i ? 1.0 : val[r];
        }
      }
      compute_bar();
    }
    compute_bar();
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int i = pi[r], k = pk[r];
      if (i >= 0) at(X, i, k) = k == i ? rs[i] : val[r] * rs[i];
    }
  }
  compute_bar();
}

// Log-det slot of a leaf: sum of log d_i over its pivots, and the failure
// code on a non-positive or non-finite pivot (one warp, d its lane's pivot).
__device__ __forceinline__ void leaf_logdet(double d, double* slot, int32_t* fail,
                                            int32_t code) {
  const bool b = !(d > 0.0) || !isfinite(d);
  double l = b ? 0.0 : log(d);
#pragma unroll
  for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  const unsigned anyb = __ballot_sync(0xffffffffu, b);
  if ((threadIdx.x & 31) == 0) {
    *slot = l;
    if (anyb) atomicCAS(fail, -1, code);
  }
}

struct Slot {
  int type, i, j, k, z;
};

// Shared memory of a CTA: two stages of three tiles (first and second operand,
// accumulator and result), and in the tensor-core modes the slices of two tiles.
struct DagSmem {
  alignas(16) double t[2][3][T][kTP];
  LeafBuf lbuf;
  double piv[2][T], rs[T];
  Slot slot[2];
  // mbarriers: stage filled / result stored / stage free, chain step's tiles in place,
  // chain step's L / X stored (by parity of the step)
  unsigned long long full[2], done[2], free[2], ch[2], lst[2], xst[2];
  int abort;
};
template <bool TC>
constexpr int dag_smem() {
  return (int)((sizeof(DagSmem) + 15) / 16 * 16) + (TC ? kOzTileSmem : 0);
}

__device__ __forceinline__ void mb_init(unsigned long long* b) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(b))
               : "memory");
}
__device__ __forceinline__ void mb_arrive(unsigned long long* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(b))
               : "memory");
}
// Waits for the phase of the given parity; false after an abort in the CTA, or after
// four times the limit of a wait on another CTA (which ends first).
__device__ __forceinline__ bool mb_wait(unsigned long long* b, int parity, volatile int* abort,
                                        unsigned long long wait_ns) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(b);
  unsigned long long t0 = 0;
  for (unsigned it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    if (*abort) return false;
    if ((it & 63) == 63) {
      const unsigned long long t = now_ns();
      if (t0 == 0) t0 = t;
      else if (t - t0 > 4 * wait_ns) {
        *abort = 1;
        return false;
      }
    }
  }
}

// TC: the tile products emulated in FP64 on the tensor cores (tile_mm_oz,
// the tensor-core modes); otherwise FP64 FMAs.  Two CTAs fit an SM, or one beside a
// product of another leg.
template <bool TC>
__global__ void __launch_bounds__(kDagAllThreads, 2) potrf_dag_kernel(DagArgs g) {
  extern __shared__ __align__(16) unsigned char dsm[];
  DagSmem& sm = *reinterpret_cast<DagSmem*>(dsm);
  OzTile oz;
  oz.xp = reinterpret_cast<__nv_bfloat16*>(dsm + (sizeof(DagSmem) + 15) / 16 * 16);
  oz.yp = oz.xp + 8 * kOzPlane;
  oz.ex = reinterpret_cast<int*>(oz.yp + 8 * kOzPlane);
  oz.ey = oz.ex + T;
  const int p = g.p, ld = g.ld, pp = p * p;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int q = 0; q < 2; ++q) {
      mb_init(&sm.full[q]);
      mb_init(&sm.done[q]);
      mb_init(&sm.free[q]);
      mb_init(&sm.ch[q]);
      mb_init(&sm.lst[q]);
      mb_init(&sm.xst[q]);
    }
    sm.abort = 0;
  }
  __syncthreads();
  volatile int* const abort = &sm.abort;
  auto Lt = [&](const DagInst& I, int i, int k) {
    return I.Lt + ((int64_t)i * (i - 1) / 2 + k) * T * T;
  };
  auto cntW = [&](const DagInst& I) { return I.st; };
  auto cntR = [&](const DagInst& I) { return I.st + pp; };
  auto doneF = [&](const DagInst& I) { return I.st + 2 * pp; };
  auto doneS = [&](const DagInst& I) { return I.st + 2 * pp + p; };
  auto doneG = [&](const DagInst& I) { return I.st + 3 * pp + p; };
  // phase of a chain step's barriers (by parity of the step), hc chains before this one on
  // this CTA (blocks of one or two tiles have no tasks that tie a chain to its CTA)
  auto step_phase = [&](int c, int hc) { return hc * ((p + 1 - (c & 1)) / 2) + (c >> 1); };
  auto l_phase = [&](int c, int hc) {   // steps from 1 on
    return hc * (c & 1 ? p / 2 : (p - 1) / 2) + ((c - 1) >> 1);
  };
  int hc = 0;
  auto wait = [&](unsigned long long* b, int parity) {
    return mb_wait(b, parity & 1, abort, g.wait_ns);
  };

  if (warp == kDagFetch) {
    // ---- fetcher: task n into stage n & 1
    int* busy = &g.smbusy[sm_id() & 255];
    for (int n = 0;; ++n) {
      const int s = n & 1;
      if (n >= 2 && !wait(&sm.free[s], (n >> 1) - 1)) return;
      int tg = 0;
      if (lane == 0) {
        // On an SM that runs a chain, take no task while the chain is there: it
        // gets the SM's whole FP64 pipe.  Waiting before taking a ticket holds
        // nothing another task needs.
        if (g.yield && ld_acquire(busy) > 0) {
          const unsigned long long t0 = now_ns();
          while (ld_acquire(busy) > 0 && ld_acquire(g.counter) < g.total &&
                 !ld_acquire(g.abort)) {
            __nanosleep(256);
            if (now_ns() - t0 > g.wait_ns) {
              atomicExch(g.abort, 1);
              break;
            }
          }
        }
        tg = atomicAdd(g.counter, 1);
      }
      tg = __shfl_sync(0xffffffffu, tg, 0);
      if (tg >= g.total) {
        if (lane == 0) {
          sm.slot[s].type = TK_END;
          mb_arrive(&sm.full[s]);
        }
        return;
      }
      const int z = tg % g.cnt;
      const Task t = decode(g, tg / g.cnt);
      const DagInst& I = g.inst[z];
      // lanes 0..2 wait for one counter each
      auto wait_all = [&](const int* c0, int v0, const int* c1, int v1, const int* c2,
                          int v2) -> bool {
        const int* c = lane == 0 ? c0 : lane == 1 ? c1 : c2;
        const int v = lane == 0 ? v0 : lane == 1 ? v1 : v2;
        const bool ok = lane > 2 || !c || wait_ge(c, v, g.abort, g.wait_ns);
        const bool all = __all_sync(0xffffffffu, ok);
        __syncwarp();   // the acquires of lanes 0..2 hold for all lanes
        if (!all && lane == 0) {
          atomicExch(I.fail, (int32_t)BTA_ERR_TIMEOUT);
          *abort = 1;
        }
        return all;
      };
      if (t.type == TK_H) {
        // the chain takes both stages: the task before it has left the other one
        if (n >= 1 && !wait(&sm.free[s ^ 1], (n - 1) >> 1)) return;
        if (lane == 0) {
          if (g.yield) atomicAdd(busy, 1);
          sm.slot[s] = {TK_H, 0, 0, 0, z};
          mb_arrive(&sm.full[s]);
        }
        bool ok = true;
        for (int c = 0; c < p && ok; ++c) {
          // W_{c,c-1} and W_cc updated through step c-2 by the U tasks (the test
          // switch instead waits for a count no task reaches).  They imply that step
          // c-2, and the product of step c-1, are done with this stage and the slices.
          Tile W = sm.t[c & 1][0];
          if (c > 0 || g.stall)
            ok = wait_all(c > 0 ? cntW(I) + c * p + c - 1 : nullptr, c - 1, cntW(I) + c * p + c,
                          g.stall ? 0x7fffffff : c - 1, nullptr, 0);
          if (!ok) break;
          if (lane == 0 && z == 0) DAG_TRACE(11, c);
          if (c > 0) load_tile(W, tile(I.A, ld, c, c - 1), ld, g.vec);
          load_tile(sm.t[c & 1][2], tile(I.A, ld, c, c), ld, g.vec);
          load_wait();
          if constexpr (TC) {
            if (c > 0)
#pragma unroll 1
              for (int part = 0; part < 8; ++part)
                oz_split([&](int r, int k) { return at(W, r, k); }, oz.xp, oz.ex, part);
          }
          __syncwarp();
          if (lane == 0) mb_arrive(&sm.ch[c & 1]);
        }
        ok = ok && wait(&sm.free[s], n >> 1);
        if (lane == 0 && g.yield) atomicSub(busy, 1);
        if (!ok) return;
        continue;
      }
      bool ok;
      switch (t.type) {
        case TK_S:
          ok = wait_all(doneF(I) + t.k, 1, cntW(I) + t.i * p + t.k, t.k, nullptr, 0);
          break;
        case TK_G:
          ok = wait_all(doneF(I) + t.i, 1, cntR(I) + t.i * p + t.j, t.i - t.j, nullptr, 0);
          break;
        case TK_U:
          ok = wait_all(doneS(I) + t.i * p + t.k, 1, doneS(I) + t.j * p + t.k, 1,
                        cntW(I) + t.i * p + t.j, t.k);
          break;
        default:   // TK_V
          ok = wait_all(doneS(I) + t.i * p + t.k, 1,
                        t.j == t.k ? doneF(I) + t.k : doneG(I) + t.k * p + t.j, 1,
                        cntR(I) + t.i * p + t.j, t.k - t.j);
      }
      if (!ok) return;
      // (measurement builds) the tasks on the way to the chain's step k + 2
      const bool crit = z == 0 && t.i == t.k + 2 &&
                        (t.type == TK_S || (t.type == TK_U && t.j == t.k + 1));
      if (crit && lane == 0) DAG_TRACE(t.type == TK_S ? 5 : 8, t.k);
      auto st = sm.t[s];
      switch (t.type) {
        case TK_S:   // L_ik = W_ik X_kk^T
          load_tile(st[0], tile(I.A, ld, t.i, t.k), ld, g.vec);
          load_tile(st[1], tile(I.A, ld, t.k, t.k), ld, g.vec);
          break;
        case TK_G:   // X_kj = X_kk R_kj  (t.i = k)
          load_tile(st[0], tile(I.A, ld, t.i, t.i), ld, g.vec);
          load_tile(st[1], tile(I.A, ld, t.i, t.j), ld, g.vec);
          break;
        case TK_U:   // W_ij -= L_ik L_jk^T
          load_tile(st[0], Lt(I, t.i, t.k), T, 1);
          load_tile(st[1], Lt(I, t.j, t.k), T, 1);
          load_tile(st[2], tile(I.A, ld, t.i, t.j), ld, g.vec);
          break;
        default:     // TK_V: R_ij -= L_ik X_kj (R_ij starts at 0 with k = j, X_jj lower)
          load_tile(st[0], Lt(I, t.i, t.k), T, 1);
          load_tile(st[1], tile(I.A, ld, t.k, t.j), ld, g.vec);
          if (t.k != t.j) load_tile(st[2], tile(I.A, ld, t.i, t.j), ld, g.vec);
      }
      load_wait();
      // a diagonal tile of the inverse is lower
      if (t.type == TK_S || (t.type == TK_V && t.k == t.j)) zero_upper(st[1]);
      if (t.type == TK_G) zero_upper(st[0]);
      __syncwarp();
      if (lane == 0) {
        sm.slot[s] = {t.type, t.i, t.j, t.k, z};
        mb_arrive(&sm.full[s]);
        if (crit) DAG_TRACE(t.type == TK_S ? 6 : 9, t.k);
      }
    }
  }

  if (warp == kDagPublish) {
    // ---- publisher
    for (int n = 0;; ++n) {
      const int s = n & 1;
      if (!wait(&sm.full[s], n >> 1)) return;
      const Slot t = sm.slot[s];
      if (t.type == TK_END) return;
      const DagInst& I = g.inst[t.z];
      if (t.type == TK_H) {
        for (int c = 0; c < p; ++c) {
          if (c > 0) {
            if (!wait(&sm.lst[c & 1], l_phase(c, hc))) return;
            if (lane == 0) st_release(doneS(I) + c * p + c - 1, 1);
          }
          if (!wait(&sm.xst[c & 1], step_phase(c, hc))) return;
          const double d = sm.piv[c & 1][lane];   // before the release lets step c+2 go on
          if (lane == 0) {
            st_release(cntW(I) + c * p + c, c);
            st_release(doneF(I) + c, 1);
            if (t.z == 0) DAG_TRACE(4, c);
          }
          __syncwarp();
          leaf_logdet(d, &I.slots[c], I.fail, I.code);
        }
        ++hc;
      }
      if (!wait(&sm.done[s], n >> 1)) return;
      if (lane == 0) {
        switch (t.type) {
          case TK_H: break;
          case TK_S: st_release(doneS(I) + t.i * p + t.k, 1); break;
          case TK_G: st_release(doneG(I) + t.i * p + t.j, 1); break;
          case TK_U: st_release(cntW(I) + t.i * p + t.j, t.k + 1); break;
          default: st_release(cntR(I) + t.i * p + t.j, t.k - t.j + 1);
        }
        if (t.z == 0 && t.i == t.k + 2 && t.type == TK_S) DAG_TRACE(7, t.k);
        if (t.z == 0 && t.i == t.k + 2 && t.type == TK_U && t.j == t.k + 1) DAG_TRACE(10, t.k);
        mb_arrive(&sm.free[s]);
      }
      __syncwarp();
    }
  }

  // ---- compute warps
  auto mm = [&](Tile X, Tile Y, bool ytrans, Tile o,
                double sign, bool acc) {
    if constexpr (TC) tile_mm_oz(X, Y, ytrans, o, sign, acc, oz);
    else tile_mm(X, Y, ytrans, o, sign, acc);
  };
  for (int n = 0;; ++n) {
    const int s = n & 1;
    if (!compute_all(wait(&sm.full[s], n >> 1))) return;
    const Slot t = sm.slot[s];
    if (t.type == TK_END) return;
    const DagInst& I = g.inst[t.z];
    auto st = sm.t[s];
    if (t.type == TK_H) {
      // ---- the chain: every diagonal step of this block on this CTA
      for (int c = 0; c < p; ++c) {
        Tile W = sm.t[c & 1][0];      // W_{c,c-1}, then X_cc
        Tile L = sm.t[c & 1][1];      // L_{c,c-1}
        Tile Wc = sm.t[c & 1][2];     // W_cc
        Tile X = sm.t[(c & 1) ^ 1][0];   // X_{c-1,c-1}
        if (c > 0) {
          if constexpr (TC)                      // while the fetcher may still be at W
            oz_split([&](int r, int k) { return k > r ? 0.0 : at(X, r, k); }, oz.yp, oz.ey, warp);
        }
        if (!compute_all(wait(&sm.ch[c & 1], step_phase(c, hc)))) return;
        if (threadIdx.x == 0 && t.z == 0) DAG_TRACE(0, c);
        if (c > 0) {
          if constexpr (TC) oz_combine(oz.xp, oz.yp, oz.ex, oz.ey, L, 1.0, false);
          else tile_mm_lt(W, X, L);              // L_{c,c-1} = W X_{c-1,c-1}^T
          compute_bar();
          if (threadIdx.x == 0 && t.z == 0) DAG_TRACE(1, c);
          store_tile(Lt(I, c, c - 1), T, L, false);
          // W_cc -= L L^T (lower)
          if constexpr (TC) {
            oz_split([&](int r, int k) { return at(L, r, k); }, oz.yp, oz.ey, warp);
            compute_bar();
            if (threadIdx.x == 0) mb_arrive(&sm.lst[c & 1]);
            if (warp != 2 && warp != 3)           // output rows 0-15 by columns 16-31
              oz_combine(oz.yp, oz.yp, oz.ey, oz.ey, Wc, -1.0, true);
          } else {
            compute_bar();
            if (threadIdx.x == 0) mb_arrive(&sm.lst[c & 1]);
            tile_syrk_lower(L, Wc);
          }
          compute_bar();
          if (threadIdx.x == 0 && t.z == 0) DAG_TRACE(2, c);
        }
        leaf(Wc, W, sm.lbuf, sm.piv[c & 1], sm.rs);   // X_cc = L_cc^{-1}
        if (threadIdx.x == 0 && t.z == 0) DAG_TRACE(3, c);
        store_tile(tile(I.A, ld, c, c), ld, W, true);
        compute_bar();
        if (threadIdx.x == 0) mb_arrive(&sm.xst[c & 1]);
      }
      ++hc;
    } else {
      switch (t.type) {
        case TK_S:
          if constexpr (TC) tile_mm_oz(st[0], st[1], true, st[2], 1.0, false, oz);
          else tile_mm_lt(st[0], st[1], st[2]);
          compute_bar();
          store_tile(Lt(I, t.i, t.k), T, st[2], false);
          break;
        case TK_G:
          mm(st[0], st[1], false, st[2], 1.0, false);
          compute_bar();
          store_tile(tile(I.A, ld, t.i, t.j), ld, st[2], false);
          break;
        case TK_U:
          mm(st[0], st[1], true, st[2], -1.0, true);
          compute_bar();
          store_tile(tile(I.A, ld, t.i, t.j), ld, st[2], t.i == t.j);
          break;
        default:
          mm(st[0], st[1], false, st[2], -1.0, t.k != t.j);
          compute_bar();
          store_tile(tile(I.A, ld, t.i, t.j), ld, st[2], false);
      }
    }
    compute_bar();
    if (threadIdx.x == 0) mb_arrive(&sm.done[s]);
  }
}

// Resident CTAs per SM of the persistent grid.  The kernel is bound by its
// chain, and one CTA per SM (as fast as two, measured) leaves room on every
// SM for a tensor-core GEMM CTA of the other sweep.  BTA_DAG_CTAS_PER_SM
// overrides the default.
int dag_ctas_per_sm() {
  static int v = [] {
    const char* e = getenv("BTA_DAG_CTAS_PER_SM");
    int x = e ? atoi(e) : 1;
    return x < 1 ? 1 : (x > 8 ? 8 : x);
  }();
  return v;
}

// Most CTAs of the persistent grid (BTA_DAG_MAX_CTAS, overriding the caller's
// cap; 0: the caller's cap for each matrix, or one per SM).  A leaf's critical path is its
// chain on one CTA; CTAs beyond what keeps its bulk tasks off that path only
// hold SMs that a concurrent sweep's products could use.
int dag_max_ctas() {
  static int v = [] {
    const char* e = getenv("BTA_DAG_MAX_CTAS");
    return e ? atoi(e) : 0;
  }();
  return v;
}

// Whether bulk tasks may yield the SM to chain tasks (BTA_DAG_YIELD=0 disables).
int dag_yield() {
  static int v = [] {
    const char* e = getenv("BTA_DAG_YIELD");
    return e ? (atoi(e) != 0) : 1;
  }();
  return v;
}

__global__ void pivot_reciprocals_kernel(const double* __restrict__ v, int64_t n,
                                         double* __restrict__ r, double* __restrict__ q) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    if (r) r[i] = recip(v[i]);
    if (q) q[i] = rsqrt_fp64(v[i]);
  }
}

}  // namespace

unsigned long long g_dag_wait_ns = 2000000000ull;
int g_dag_stall = 0;

int potrf_dag_tasks(int p) {
  int tot = 1;
  for (int k = 0; k < p; ++k) tot += step_tasks(p, k);
  return tot;
}

size_t potrf_dag_state_ints(int p) { return (size_t)4 * p * p + p + 64 + 256; }

// scratch[z] holds the packed L tiles (p(p-1)/2 tiles) followed by the
// counters; n*n doubles are enough.
bta_status potrf_dag_batch(int count, double* const* A, int n, int ld, double* const* scratch,
                           double* const* logdet_parts, int32_t* const* fail,
                           const int32_t* fail_code, cudaStream_t s, int max_ctas, int tc) {
  const int p = n / T;
  if (n <= 0 || n % T || p > kMaxP || count < 1) return BTA_ERR_ARG;
  const size_t lt_doubles = (size_t)p * (p - 1) / 2 * T * T;
  for (int z0 = 0; z0 < count; z0 += kMaxBatch) {
    const int cnt = std::min(kMaxBatch, count - z0);
    DagArgs g;
    g.p = p; g.ld = ld; g.cnt = cnt;
    int acc = 0;
    for (int k = 0; k < p; ++k) {
      g.off[k] = acc;
      acc += step_tasks(p, k);
    }
    g.off[p] = acc;
    g.total = (acc + 1) * cnt;
    g.vec = 1;
    for (int z = 0; z < cnt; ++z) {
      DagInst& I = g.inst[z];
      I.A = A[z0 + z];
      I.Lt = scratch[z0 + z];
      I.st = reinterpret_cast<int*>(scratch[z0 + z] + lt_doubles);
      I.slots = logdet_parts[z0 + z];
      I.fail = fail[z0 + z];
      I.code = fail_code[z0 + z];
      if (reinterpret_cast<uintptr_t>(I.A) % 16) g.vec = 0;
      if (reinterpret_cast<uintptr_t>(I.Lt) % 16) return BTA_ERR_ARG;   // library workspace
      BTA_CUDA_TRY(cudaMemsetAsync(I.st, 0, potrf_dag_state_ints(p) * sizeof(int), s));
    }
    // ticket counter and abort flag live after instance 0's counters
    g.counter = g.inst[0].st + 4 * p * p + p + 8;
    g.abort = g.counter + 16;
    g.smbusy = g.inst[0].st + 4 * p * p + p + 64;
    g.stall = g_dag_stall;
    g.wait_ns = g_dag_wait_ns;
    int grid = std::min(g.total, sm_count() * dag_ctas_per_sm());
    const int cap = dag_max_ctas() > 0 ? dag_max_ctas() : max_ctas * cnt;
    if (cap > 0) grid = std::min(grid, std::max(2, cap));   // the chain and a bulk CTA
    grid = std::max(grid, std::min(g.total, cnt + 1));   // every chain, and a bulk CTA
    // Two CTAs fit an SM, so the chains' SMs hold at most 2 cnt of them: only with more do
    // the bulk tasks have a CTA that does not wait for a chain to leave its SM.
    g.yield = cnt <= 2 && grid > 2 * cnt ? dag_yield() : 0;
    auto* const kernel = tc ? &potrf_dag_kernel<true> : &potrf_dag_kernel<false>;
    const int smem = tc ? dag_smem<true>() : dag_smem<false>();
    static std::atomic<uint64_t> allowed[2];   // above 48 KB of dynamic shared memory
    BTA_TRY(allow_smem(allowed[tc ? 1 : 0], reinterpret_cast<const void*>(kernel), smem));
    BTA_CUDA_TRY(launch_prio_smem(kernel, dim3(grid), dim3(kDagAllThreads), smem, s, g));
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

}  // namespace bta

extern "C" bta_status bta_pivot_reciprocals(const double* v, int64_t n, double* recip_out,
                                            double* rsqrt_out, cudaStream_t stream) {
  if (n < 0 || (n > 0 && !v) || (!recip_out && !rsqrt_out)) return BTA_ERR_ARG;
  if (n == 0) return BTA_OK;
  const int64_t blocks = (n + 255) / 256;
  if (blocks > 0x7fffffff) return BTA_ERR_ARG;
  bta::pivot_reciprocals_kernel<<<(unsigned)blocks, 256, 0, stream>>>(v, n, recip_out, rsqrt_out);
  BTA_LAUNCHED();
  return BTA_OK;
}
