// FP64 GEMM emulated on BF16 tensor cores by residues (the modular form of the
// Ozaki scheme: Ozaki, Uchino and Imamura, "Ozaki Scheme II: a GEMM-oriented
// emulation of floating-point matrix multiplication using an integer modular
// technique", arXiv 2504.08009, 2025):
//
//   C = alpha op(A) op(B) + beta C,   FP64 in and out.
//
// Operands.  Row i of op(A) is scaled by a power of two to integers
// F_ik = round(a_ik 2^(1022 + p - e_i)), |F| < 2^p, where e_i is the biased
// exponent of the row's largest entry; column n of op(B) likewise.  p = 56
// bits: three more than an FP64 significand, so that entries within a factor
// 8 of the row's largest are exact.
//
// Products.  The integer product X_mn = sum_k F_mk G_kn, |X| <= K 2^(2p), is
// computed exactly modulo 14 pairwise coprime moduli p_i <= 511 whose product
// P = 2^125.2 exceeds 2 |X| (K <= 4847 with p = 56; p = 55 above), and
// recovered by the Chinese remainder theorem.  A residue |r| <= 255 is exact
// in BF16, and a sum of 256 products of residues stays below 2^24, exact in
// the tensor core's FP32 accumulator; each 256 of K the accumulator is
// reduced modulo p_i in FP32 (exactly).  So one FP64 product costs 14 BF16
// products.  Splitting into 8 base-128 digits, with 36 digit products, cost
// 2.6 times that: 4800^3 whole call 5.38 ms before, 2.61 ms now, at no larger
// error (no digit products are dropped: 8e-16 of the norm at K = 4847 and 5120, now 4e-17
// and, with p = 55, 9e-17).
//
// Kernels: exponents of the rows (ozaki_exp_kernel), residue planes (residue_kernel),
// the 14 products (crt_gemm_kernel, crt_gemm_small_kernel), and the recovery with alpha,
// beta (crt_compose_kernel).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>

#include "common.cuh"
#include "ozaki_digits.cuh"
#include "tma.cuh"

namespace bta {
namespace {

using namespace tc;

// ---- moduli ------------------------------------------------------------------
// The 14 pairwise coprime numbers up to 511 with the largest product.
constexpr int kNumMod = kOzakiModuli;
constexpr int kMod[kNumMod] = {511, 509, 508, 505, 503, 501, 499,
                               493, 491, 487, 481, 479, 473, 467};
constexpr int kMaxK56 = 4847;   // 2 K 2^112 <= P

constexpr int sym_mod(long long a, int p) {   // residue of smallest magnitude
  const int r = (int)(((a % p) + p) % p);
  return r > p / 2 ? r - p : r;
}
constexpr int cofactor_inverse(int i) {   // (P / p_i)^{-1} mod p_i
  int c = 1;
  for (int j = 0; j < kNumMod; ++j)
    if (j != i) c = c * (kMod[j] % kMod[i]) % kMod[i];
  int w = 1;
  while (c * w % kMod[i] != 1) ++w;
  return w;
}
constexpr unsigned __int128 mod_product() {
  unsigned __int128 p = 1;
  for (int j = 0; j < kNumMod; ++j) p *= (unsigned)kMod[j];
  return p;
}
// Recovery from pairs of residues: X / P = sum_i r_i w_i / p_i modulo 1, w_i = the inverse
// of P / p_i modulo p_i of smallest magnitude.  Moduli p = p_2q and p' = p_2q+1 together
// give (r a + r' b) / (p p') with a = w p', b = w' p below 2^17, so a 32-bit integer y and
// one product of it by round(2^113 / (p p')) < 2^96 stand for two residues (half the wide
// multiplications of one 96-bit fraction per residue).
constexpr int kFracBits = 113;
// the residues are stored + 256 (non-negative 16-bit integers below kStored)
constexpr int kBias = 256, kStored = 513;
constexpr int pair_coef(int i, int j) { return sym_mod(cofactor_inverse(i), kMod[i]) * kMod[j]; }
constexpr int pair_shift(int i, int j) {   // makes y non-negative
  const int a = pair_coef(i, j), b = pair_coef(j, i);
  return (a < 0 ? -a * (kStored - 1) : 0) + (b < 0 ? -b * (kStored - 1) : 0);
}
constexpr unsigned __int128 pair_fraction(int i, int j) {
  const unsigned pp = (unsigned)(kMod[i] * kMod[j]);
  return (((unsigned __int128)1 << kFracBits) + pp / 2) / pp;
}
// minus the sum when every residue is 0, modulo 2^128
constexpr unsigned __int128 crt_offset() {
  unsigned __int128 s = 0;
  for (int j = 0; j < kNumMod; j += 2)
    s -= (unsigned __int128)(kBias * (pair_coef(j, j + 1) + pair_coef(j + 1, j)) +
                             pair_shift(j, j + 1)) * pair_fraction(j, j + 1);
  return s;
}
constexpr unsigned long long kPTop = (unsigned long long)(mod_product() >> 62);   // P 2^-62
static_assert(kPTop >> 63, "P lies in [2^125, 2^126)");

template <int I>
struct Modulus {
  static constexpr float p = (float)kMod[I];
  static constexpr float inv = 1.0f / (float)kMod[I];
  // residues of 2^14, 2^28, 2^42
  static constexpr float c1 = (float)sym_mod(1ll << 14, kMod[I]);
  static constexpr float c2 = (float)sym_mod(1ll << 28, kMod[I]);
  static constexpr float c3 = (float)sym_mod(1ll << 42, kMod[I]);
};
template <int I>   // moduli I and I + 1
struct ModPair {
  static constexpr int a = pair_coef(I, I + 1), b = pair_coef(I + 1, I);
  static constexpr int c = pair_shift(I, I + 1);
  static constexpr uint32_t f0 = (uint32_t)pair_fraction(I, I + 1);
  static constexpr uint32_t f1 = (uint32_t)(pair_fraction(I, I + 1) >> 32);
  static constexpr uint32_t f2 = (uint32_t)(pair_fraction(I, I + 1) >> 64);
};
struct CrtOffset {
  static constexpr uint32_t l0 = (uint32_t)crt_offset(), l1 = (uint32_t)(crt_offset() >> 32);
  static constexpr unsigned long long l2 =   // modulo 2^113 like the sum: 49 bits
      (unsigned long long)(crt_offset() >> 64) & ((1ull << (kFracBits - 64)) - 1);
};

struct ModTable {
  float p[kNumMod], inv[kNumMod];
};
constexpr ModTable make_mod_table() {
  ModTable t{};
  for (int i = 0; i < kNumMod; ++i) {
    t.p[i] = (float)kMod[i];
    t.inv[i] = 1.0f / (float)kMod[i];
  }
  return t;
}
__constant__ ModTable c_mod = make_mod_table();

constexpr float kMagic = 12582912.0f;   // 1.5 2^23: x + kMagic rounds x to an integer

// Two FP32 operations per instruction.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// The launches of a product follow one another with programmatic serialization: a kernel may
// start once every block of the one before has called launch_next (or ended), and waits in
// await_prior for its completion before it touches what that one writes.
// So a kernel's launch, set-up and first operand loads run behind the tail of the one
// before (call of 1024^3 94.9 -> 90.3 us, 1216 x 1184 x 1184 127.8 -> 119.9).  The products
// themselves leave it at their end: a recovery that waits beside them takes SMs from the
// other legs' kernels (b = 2400 gradient 54.2 ms, 55.2 with it).
__device__ __forceinline__ void await_prior() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void launch_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... KArgs, class... Args>
cudaError_t launch_after(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                         cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// ---- the 14 products ---------------------------------------------------------
//
// A unit is one 256 x 256 output tile modulo one p_i, taken by a pair of CTAs on
// two SMs (a thread-block cluster of 2, tcgen05 cta_group::2: M = 256, N = 256):
// CTA r holds A rows r*128.. and B rows (columns of op(B)) r*128.. of the tile,
// and its tensor memory accumulates output rows r*128.. .  Every operand byte
// is used once per unit, so the tile is as large as tensor memory allows with
// two accumulators (2 x 256 of its 512 columns): an SM reads 8 KB of shared
// memory per 256 x 256 x 16 MMA (128 clocks) and loads 64 bytes a clock from L2,
// half of what 128 x 128 tiles would.
//
// A pair works through up to `per` units; accumulator e & 1 takes the e-th chunk
// of 256 of K, and the drain of one chunk (and the store of a finished unit)
// overlaps the MMAs of the next.  320 threads: warps 0-7 drain (two per TMEM lane
// quarter, 128 columns each; the tile's residues stay in their registers across the
// chunks), warp 8 loads (TMA, 128-byte swizzle, 64-wide K slabs, a ring of three stages
// of two slabs: with a barrier round per slab 6 % slower),
// warp 9 of the leader CTA issues the MMAs.
//
// Across the pair: both CTAs' loads of a slab complete on the leader's `loaded`
// barrier (a peer that waited for its own half and relayed it held the pair to one
// slab per 1250 clocks).  The leader's commits arrive on both CTAs' `empty` and
// `accfull` barriers (multicast); each drain warp, when its loads of a chunk are
// done, arrives on the leader's `accempty`.  Before releasing tensor memory the two
// CTAs exchange `done` arrivals, so neither deallocates or exits while the other
// may still touch its shared or tensor memory.  Every wait is bounded: on expiry a
// CTA records BTA_ERR_TIMEOUT in the status word, stops issuing work and still takes
// part in the exchange, in which the leader waits (bounded) for the loads in flight.
constexpr int CT = 256;                   // tile rows and columns of a pair
constexpr int CH = 128;                   // rows of A, and of B, per CTA
constexpr int CK = 64;                    // bf16 per K slab: 128-byte rows
constexpr int kHalfTile = CH * CK * 2;    // 16 KB
constexpr int kSlab = 2 * kHalfTile;
constexpr int kStageSlabs = 2;            // K slabs a stage: one barrier round for 128 of K
constexpr int kStage = kStageSlabs * kSlab;
constexpr int kStages = 3;
constexpr int kChunkSlabs = 4;            // 256 of K: the exactness limit of a sum
constexpr int kDrainWarps = 8;
constexpr int kCrtThreads = (kDrainWarps + 2) * 32;
constexpr int kCrtSmem = kStages * kStage + 1024 + 512;
constexpr long long kCrtWaitLimit = 1ll << 21;   // bounded mbarrier polls
// kind::f16: FP32 accumulator, A and B BF16, both K-major, N = 256, M = 256
constexpr uint32_t kCrtIdesc = (1u << 4) | (1u << 7) | (1u << 10) |
                               ((uint32_t)(CT >> 3) << 17) | ((uint32_t)(CT >> 4) << 24);

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row
// groups 1024 bytes apart.
__device__ __forceinline__ uint64_t sdesc128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);   // start address
  d |= (uint64_t)1 << 16;                     // leading-dimension offset (unused)
  d |= (uint64_t)(1024 >> 4) << 32;           // stride between 8-row groups
  d |= (uint64_t)1 << 46;                     // descriptor version
  d |= (uint64_t)2 << 61;                     // 128-byte swizzle
  return d;
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// The shared::cluster address of the same shared-memory offset in CTA `rank`.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}

__device__ __forceinline__ void mbar_arrive_remote(uint32_t caddr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(caddr)
               : "memory");
}


// Bounded wait with cluster-scope acquire (the barrier receives arrivals from
// the peer CTA or the leader's tensor-core commits).
__device__ __forceinline__ bool mbar_wait_cl(uint32_t addr, uint32_t parity, long long limit) {
  for (long long it = 0; it < limit; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// Commit of the leader's pair MMAs: arrive on the barrier at this offset in
// both CTAs once they complete.
__device__ __forceinline__ void pair_commit_both(uint32_t mbar, uint32_t leader) {
  const uint16_t mask = 3;
  asm volatile(
      "{\n .reg .pred e;\n setp.ne.b32 e, %1, 0;\n"
      " @e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %2;\n}\n" ::"r"(mbar),
      "r"(leader), "h"(mask)
      : "memory");
}

// ... on the leader's barrier only.
__device__ __forceinline__ void pair_commit_own(uint32_t mbar, uint32_t leader) {
  asm volatile(
      "{\n .reg .pred e;\n setp.ne.b32 e, %1, 0;\n"
      " @e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(
          mbar),
      "r"(leader)
      : "memory");
}


// A load into this CTA's shared memory that completes on a barrier of either CTA of
// the pair (mbar: its shared::cluster address).
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t mbar,
                                              int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(mbar), "r"(x), "r"(y)
      : "memory");
}

// Arrive on a barrier of either CTA; the tcgen05 fences around it order the tensor
// memory accesses.
__device__ __forceinline__ void mbar_arrive_pair(uint32_t caddr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(caddr) : "memory");
}

__device__ __forceinline__ void pair_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(kCrtIdesc), "r"(acc)
      : "memory");
}

// Start the load of 8 consecutive fp32 columns of this thread's TMEM lane; tmem_wait
// completes every load started.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[8]) {   // r: not read before
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                 "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
}

// A chunk's sums into the running residues: per column t = S + acc (|t| < 2^24, exact),
// acc = t mod p, two columns per instruction.
struct CrtMod {
  uint64_t np, inv, magic, nmagic;
  __device__ __forceinline__ explicit CrtMod(int m) {
    const float pf = -c_mod.p[m], invf = c_mod.inv[m];
    np = pack2(pf, pf);
    inv = pack2(invf, invf);
    magic = pack2(kMagic, kMagic);
    nmagic = pack2(-kMagic, -kMagic);
  }
  __device__ __forceinline__ void add(const uint32_t (&v)[8], uint64_t* acc) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint64_t s = add2(
          pack2(__uint_as_float(v[2 * q]), __uint_as_float(v[2 * q + 1])), acc[q]);
      const uint64_t k = add2(fma2(s, inv, magic), nmagic);
      acc[q] = fma2(k, np, s);
    }
  }
};
// Drain of 2 N columns from taddr on; loaded() once all are in registers.  Ahead: the loads
// of the next 8 columns run behind the arithmetic of the last 8 (with one CTA per SM the
// drain's latency is on the product's critical path: an accumulator is refilled two chunks
// later).  With two CTAs per SM the other one fills the wait, and loads of 16 columns
// without overlap are 3 to 8 % faster.
template <bool Ahead, int N, class Loaded>
__device__ __forceinline__ void crt_drain(uint32_t taddr, const CrtMod& mod, uint64_t (&acc)[N],
                                          Loaded loaded) {
  uint32_t v[2][8];
  if constexpr (Ahead) tmem_ld8(taddr, v[0]);
#pragma unroll
  for (int h = 0; h < N / 4; ++h) {
    if constexpr (Ahead) {
      tmem_wait(v[h & 1]);
      if (h + 1 < N / 4) tmem_ld8(taddr + 8 * (h + 1), v[(h + 1) & 1]);
      else loaded();
    } else if ((h & 1) == 0) {
      tmem_ld8(taddr + 8 * h, v[0]);
      tmem_ld8(taddr + 8 * (h + 1), v[1]);
      tmem_wait(v[0]);
      tmem_wait(v[1]);
      if (h + 2 == N / 4) loaded();
    }
    mod.add(v[h & 1], acc + 4 * h);
  }
}
// Residues of 2 n consecutive columns of a row (columns `ld` apart) as 16-bit integers: the
// low half of x + kMagic is x.
template <int N>
__device__ __forceinline__ void crt_store(uint16_t* out, int ld, const uint64_t (&acc)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) {
    float a0, a1;
    unpack2(acc[q], a0, a1);
    out[(int64_t)(2 * q) * ld] = (uint16_t)__float_as_uint(a0 + (kMagic + kBias));
    out[(int64_t)(2 * q + 1) * ld] = (uint16_t)__float_as_uint(a1 + (kMagic + kBias));
  }
}

struct CrtArgs {
  int Mp, Np, Ap, Bp;   // output rows / columns (padded); rows per A / B plane
  int nk;               // 64-wide K slabs
  int mt, nt, tiles;    // tile rows, tile columns, tiles taken
  int group;            // tile rows per group of the launch order
  int lower;            // only tiles that reach the lower triangle
  int tri_a, tri_b;     // triangle of op(A) / op(B) (Tri): their zero K ranges are skipped
  int slots, per;       // pairs resident together; units per pair
  int mod0, nmod;       // the moduli whose planes these are (ozaki_gemm: group)
  uint16_t* R;          // [kNumMod][Np][Mp] residues + kBias
  int32_t* status;
};

struct CrtUnit {
  int mod, m0, n0, ks0, ks1;   // mod: among the launch's moduli
};

// Unit u of CT x CT tiles: modulus-major, so that the resident pairs work on the planes of one
// modulus (they fit in L2).  Within it groups of `group` tile rows, column by
// column; or, for the lower triangle, rows of tiles up to the diagonal.
template <int CT>
__device__ __forceinline__ CrtUnit crt_unit(const CrtArgs& g, int u) {
  CrtUnit t;
  t.mod = u / g.tiles;
  int q = u - t.mod * g.tiles, i, j;
  if (g.lower) {
    const int full = g.nt * (g.nt + 1) / 2;   // rows i < nt hold i + 1 tiles, then nt each
    if (q < full) {
      i = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
      while (i * (i + 1) / 2 > q) --i;
      while ((i + 1) * (i + 2) / 2 <= q) ++i;
      j = q - i * (i + 1) / 2;
    } else {
      i = g.nt + (q - full) / g.nt;
      j = (q - full) % g.nt;
    }
  } else {
    const int grp = q / (g.group * g.nt);
    const int gm = min(g.group, g.mt - grp * g.group);
    q -= grp * g.group * g.nt;
    i = grp * g.group + q % gm;
    j = q / gm;
  }
  t.m0 = i * CT;
  t.n0 = j * CT;
  // the K slabs on which op(A) and op(B) can be nonzero: a lower op(A) has
  // a_mk = 0 for k > m, an upper one for k < m; a lower op(B) has b_kn = 0 for
  // k < n, an upper one for k > n (the planes hold zeros there)
  int kb = 0, ke = g.nk;
  if (g.tri_a == TRI_LOWER) ke = min(ke, (t.m0 + CT) / CK);
  if (g.tri_a == TRI_UPPER) kb = max(kb, t.m0 / CK);
  if (g.tri_b == TRI_LOWER) kb = max(kb, t.n0 / CK);
  if (g.tri_b == TRI_UPPER) ke = min(ke, (t.n0 + CT) / CK);
  t.ks0 = kb;
  t.ks1 = max(kb, ke);
  return t;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kCrtThreads, 1)
    crt_gemm_kernel(const __grid_constant__ CUtensorMap mA,
                    const __grid_constant__ CUtensorMap mB, CrtArgs g) {
  const uint32_t rank = cluster_rank();
  // unit j of this pair: pairs launched together take consecutive units
  const int pair = (int)blockIdx.x >> 1, total = g.tiles * g.nmod;
  const int u0 = (pair / g.slots) * g.per * g.slots + pair % g.slots;
  if (u0 >= total) return;   // the same decision in both CTAs, before any set-up
  const int units = min(g.per, (total - u0 + g.slots - 1) / g.slots);
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStage);
  const int kLoaded = 0, kEmpty = kStages, kAccFull = 2 * kStages, kAccEmpty = 2 * kStages + 2,
            kFinal = 2 * kStages + 4, kDone = 2 * kStages + 5;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 6);
  __shared__ int s_abort, s_issued, s_waited, s_peer;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&bars[kLoaded + s]), 1);
      mbar_init(smem_u32(&bars[kEmpty + s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bars[kAccFull + b]), 1);
      mbar_init(smem_u32(&bars[kAccEmpty + b]), 2 * kDrainWarps);   // both CTAs' drain warps
    }
    mbar_init(smem_u32(&bars[kFinal]), 1);
    mbar_init(smem_u32(&bars[kDone]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
    s_issued = 0;
    s_waited = 0;
    s_peer = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  // both CTAs' barriers and tensor memory are set up before either touches the other's
  asm volatile("barrier.cluster.arrive.release.aligned;\n"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == kDrainWarps) {
    // ---- TMA producer (both CTAs): this CTA's halves of every slab
    if (lane == 0) {
      const uint32_t loaded0 = cluster_addr(smem_u32(&bars[kLoaded]), 0);
      await_prior();
      int r = 0;
      bool stop = false;
      for (int j = 0; j < units && !stop; ++j) {
        const CrtUnit t = crt_unit<CT>(g, u0 + j * g.slots);
        const int ya = t.mod * g.nk * g.Ap + t.m0 + (int)rank * CH;
        const int yb = t.mod * g.nk * g.Bp + t.n0 + (int)rank * CH;
        for (int kt = t.ks0; kt < t.ks1; kt += kStageSlabs, ++r) {
          const int s = r % kStages;
          if (r >= kStages && !mbar_wait(smem_u32(&bars[kEmpty + s]),
                                         (uint32_t)((r / kStages - 1) & 1), kCrtWaitLimit)) {
            atomicExch(&s_abort, 1);
            stop = true;
            break;
          }
          if (*(volatile int*)&s_abort) {
            stop = true;
            break;
          }
          const int ns = min(kStageSlabs, t.ks1 - kt);
          if (rank == 0) mbar_expect_tx(smem_u32(&bars[kLoaded + s]), 2u * kSlab * ns);
          const uint32_t full = loaded0 + 8u * (uint32_t)s;
          for (int u = 0; u < ns; ++u) {
            uint8_t* st = smem + s * kStage + u * kSlab;
            tma_load_pair(smem_u32(st), &mA, full, 0, ya + (kt + u) * g.Ap);
            tma_load_pair(smem_u32(st + kHalfTile), &mB, full, 0, yb + (kt + u) * g.Bp);
          }
          *(volatile int*)&s_issued = r + 1;
        }
      }
    }
    __syncwarp();
  } else if (warp == kDrainWarps + 1) {
    // ---- MMA issuer (leader CTA): lane 0 alone runs the loop and issues
    if (lane == 0 && rank == 0) {
      const uint64_t dbase = sdesc128(smem_u32(smem));
      bool stop = false;
      int r = 0, e = 0;   // slabs consumed, chunks begun
      for (int j = 0; j < units && !stop; ++j) {
        const CrtUnit t = crt_unit<CT>(g, u0 + j * g.slots);
        for (int kc = t.ks0; kc < t.ks1 && !stop; kc += kChunkSlabs, ++e) {
          const int b = e & 1;
          // both CTAs have drained this accumulator's last chunk
          if (e >= 2 && !mbar_wait(smem_u32(&bars[kAccEmpty + b]), (uint32_t)((e / 2 - 1) & 1),
                                   kCrtWaitLimit)) {
            stop = true;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int ke = min(t.ks1, kc + kChunkSlabs);
          for (int kt = kc; kt < ke; kt += kStageSlabs, ++r) {
            const int s = r % kStages;
            const uint32_t par = (uint32_t)((r / kStages) & 1);
            if (!mbar_wait(smem_u32(&bars[kLoaded + s]), par, kCrtWaitLimit)) {
              stop = true;
              break;
            }
            *(volatile int*)&s_waited = r + 1;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int u = 0; u < min(kStageSlabs, ke - kt); ++u) {
              const uint64_t da = dbase + (uint64_t)((s * kStage + u * kSlab) >> 4);
#pragma unroll
              for (int kk = 0; kk < CK / 16; ++kk)   // 16 bf16 = 32 bytes along K
                pair_mma(tmem + (uint32_t)(b * CT), da + 2 * kk, da + (kHalfTile >> 4) + 2 * kk,
                         kt + u > kc || kk > 0);
            }
            pair_commit_both(smem_u32(&bars[kEmpty + s]), 1u);   // both halves free
          }
          if (!stop) pair_commit_both(smem_u32(&bars[kAccFull + b]), 1u);   // sums ready
        }
      }
      if (stop) {
        atomicExch(&s_abort, 1);
        // wait (bounded) for the MMAs this thread issued before leaving
        pair_commit_own(smem_u32(&bars[kFinal]), 1u);
        mbar_wait(smem_u32(&bars[kFinal]), 0, kCrtWaitLimit);
      }
    }
    __syncwarp();
  } else {
    // ---- warps 0-7 (both CTAs): thread = output row (TMEM lane) x 128 columns
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const int row = (int)rank * CH + (warp & 3) * 32 + lane, col0 = (warp >> 2) * 128;
    const uint32_t acc_empty = cluster_addr(smem_u32(&bars[kAccEmpty]), 0);
    bool failed = false;
    int e = 0;
    for (int j = 0; j < units && !failed; ++j) {
      const CrtUnit t = crt_unit<CT>(g, u0 + j * g.slots);
      const CrtMod mod(g.mod0 + t.mod);
      uint64_t acc[64];
#pragma unroll
      for (int q = 0; q < 64; ++q) acc[q] = 0ull;
      for (int kc = t.ks0; kc < t.ks1; kc += kChunkSlabs, ++e) {
        const int b = e & 1;
        bool ok = mbar_wait(smem_u32(&bars[kAccFull + b]), (uint32_t)((e / 2) & 1),
                            kCrtWaitLimit);
        ok = ok && !*(volatile int*)&s_abort;
        if (!__all_sync(0xffffffffu, ok)) {
          failed = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        crt_drain<true>(tmem + lane_off + (uint32_t)(b * CT + col0), mod, acc, [&]() {
          // this warp's loads are done: the accumulator may be refilled
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive_pair(acc_empty + 8u * (uint32_t)b);
        });
      }
      if (failed) break;
      // a warp's lanes are 32 consecutive rows
      crt_store(g.R + ((int64_t)(g.mod0 + t.mod) * g.Np + t.n0 + col0) * g.Mp + t.m0 + row, g.Mp,
                acc);
    }
    if (failed && lane == 0) atomicExch(&s_abort, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    // the exchange: the peer arrives, then waits; the leader waits, then arrives.  After
    // an abort the peer first leaves -(slabs it has issued) - 1 with the leader, which
    // waits (bounded) for the slabs either of them has in flight: the ones that only the
    // peer issued it expects here, the peer's bytes alone.
    bool ok;
    if (rank != 0) {
      if (s_abort)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(smem_u32(&s_peer), 0)),
                     "r"(-s_issued - 1)
                     : "memory");
      mbar_arrive_remote(cluster_addr(smem_u32(&bars[kDone]), 0));
      ok = mbar_wait_cl(smem_u32(&bars[kDone]), 0, kCrtWaitLimit);
    } else {
      ok = mbar_wait_cl(smem_u32(&bars[kDone]), 0, kCrtWaitLimit);
      const int peer = *(volatile int*)&s_peer;
      if (s_abort || peer < 0) {
        const int issued = s_issued, all = max(issued, peer < 0 ? -peer - 1 : 0);
        for (int r = s_waited; r < all; ++r) {
          const uint32_t full = smem_u32(&bars[kLoaded + r % kStages]);
          if (r >= issued) mbar_expect_tx(full, (uint32_t)kStage);
          mbar_wait(full, (uint32_t)((r / kStages) & 1), kCrtWaitLimit);
        }
      }
      mbar_arrive_remote(cluster_addr(smem_u32(&bars[kDone]), 1));
    }
    if ((s_abort || !ok) && g.status) atomicExch(g.status, (int)BTA_ERR_TIMEOUT);
  }
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
  }
}

// ---- the 14 products, small shapes -------------------------------------------
//
// The same with one 128 x 128 tile modulo one p_i per CTA (twice the loads of a pair's
// tile per product): 98 KB of shared memory, half of tensor memory and at most 102 registers a thread, so that two CTAs share an SM,
// or one runs beside a task-graph leaf of another leg, where a pair finds no place
// until the leaves end.
constexpr int ST = 128;
constexpr int kSmallStages = 3;
constexpr int kSmallStage = 2 * kHalfTile;
constexpr int kSmallSmem = kSmallStages * kSmallStage + 1024 + 256;
constexpr uint32_t kSmallIdesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                 ((uint32_t)(ST >> 3) << 17) | ((uint32_t)(ST >> 4) << 24);

__device__ __forceinline__ void small_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(kSmallIdesc), "r"(acc)
      : "memory");
}

__global__ void __launch_bounds__(kCrtThreads, 2)
    crt_gemm_small_kernel(const __grid_constant__ CUtensorMap mA,
                          const __grid_constant__ CUtensorMap mB, CrtArgs g) {
  const CrtUnit t = crt_unit<ST>(g, blockIdx.x);
  const int slabs = t.ks1 - t.ks0, chunks = (slabs + kChunkSlabs - 1) / kChunkSlabs;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kSmallStages * kSmallStage);
  const int kLoaded = 0, kEmpty = kSmallStages, kAccFull = 2 * kSmallStages,
            kAccEmpty = kAccFull + 2, kFinal = kAccFull + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kAccFull + 5);
  __shared__ int s_abort, s_issued, s_waited;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSmallStages; ++s) {
      mbar_init(smem_u32(&bars[kLoaded + s]), 1);
      mbar_init(smem_u32(&bars[kEmpty + s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bars[kAccFull + b]), 1);
      mbar_init(smem_u32(&bars[kAccEmpty + b]), kDrainWarps);
    }
    mbar_init(smem_u32(&bars[kFinal]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
    s_issued = 0;
    s_waited = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(2 * ST)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == kDrainWarps) {
    if (lane == 0) {   // ---- TMA producer
      await_prior();
      for (int r = 0; r < slabs; ++r) {
        const int s = r % kSmallStages;
        if (r >= kSmallStages && !mbar_wait(smem_u32(&bars[kEmpty + s]),
                                            (uint32_t)((r / kSmallStages - 1) & 1),
                                            kCrtWaitLimit)) {
          atomicExch(&s_abort, 1);
          break;
        }
        if (*(volatile int*)&s_abort) break;
        const uint32_t full = smem_u32(&bars[kLoaded + s]);
        mbar_expect_tx(full, (uint32_t)kSmallStage);
        uint8_t* st = smem + s * kSmallStage;
        const int ks = t.mod * g.nk + t.ks0 + r;
        tma_load_2d(smem_u32(st), &mA, full, 0, ks * g.Ap + t.m0);
        tma_load_2d(smem_u32(st + kHalfTile), &mB, full, 0, ks * g.Bp + t.n0);
        *(volatile int*)&s_issued = r + 1;
      }
    }
    __syncwarp();
  } else if (warp == kDrainWarps + 1) {
    if (lane == 0) {   // ---- MMA issuer
      const uint64_t dbase = sdesc128(smem_u32(smem));
      bool stop = false;
      int r = 0;
      for (int e = 0; e < chunks && !stop; ++e) {
        const int b = e & 1;
        if (e >= 2 && !mbar_wait(smem_u32(&bars[kAccEmpty + b]), (uint32_t)((e / 2 - 1) & 1),
                                 kCrtWaitLimit)) {
          stop = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int re = min(slabs, (e + 1) * kChunkSlabs);
        for (; r < re; ++r) {
          const int s = r % kSmallStages;
          if (!mbar_wait(smem_u32(&bars[kLoaded + s]), (uint32_t)((r / kSmallStages) & 1),
                         kCrtWaitLimit)) {
            stop = true;
            break;
          }
          *(volatile int*)&s_waited = r + 1;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = dbase + (uint64_t)((s * kSmallStage) >> 4);
#pragma unroll
          for (int kk = 0; kk < CK / 16; ++kk)
            small_mma(tmem + (uint32_t)(b * ST), da + 2 * kk, da + (kHalfTile >> 4) + 2 * kk,
                      r > e * kChunkSlabs || kk > 0);
          mma_commit(smem_u32(&bars[kEmpty + s]));
        }
        if (!stop) mma_commit(smem_u32(&bars[kAccFull + b]));
      }
      if (stop) {
        atomicExch(&s_abort, 1);
        // wait (bounded) for the MMAs this thread issued before leaving
        mma_commit(smem_u32(&bars[kFinal]));
        mbar_wait(smem_u32(&bars[kFinal]), 0, kCrtWaitLimit);
      }
    }
    __syncwarp();
  } else {
    // ---- warps 0-7: thread = output row (TMEM lane) x 64 columns
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const int row = (warp & 3) * 32 + lane, col0 = (warp >> 2) * 64;
    const CrtMod mod(g.mod0 + t.mod);
    bool failed = false;
    uint64_t acc[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) acc[q] = 0ull;
    for (int e = 0; e < chunks; ++e) {
      const int b = e & 1;
      bool ok = mbar_wait(smem_u32(&bars[kAccFull + b]), (uint32_t)((e / 2) & 1), kCrtWaitLimit);
      ok = ok && !*(volatile int*)&s_abort;
      if (!__all_sync(0xffffffffu, ok)) {
        failed = true;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      crt_drain<false>(tmem + lane_off + (uint32_t)(b * ST + col0), mod, acc, [&]() {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(
                           smem_u32(&bars[kAccEmpty + b]))
                       : "memory");
      });
    }
    if (!failed)
      crt_store(g.R + ((int64_t)(g.mod0 + t.mod) * g.Np + t.n0 + col0) * g.Mp + t.m0 + row, g.Mp,
                acc);
    else if (lane == 0)
      atomicExch(&s_abort, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && s_abort) {
    // loads issued but not seen complete: wait (bounded) for them to land
    for (int r = s_waited; r < s_issued; ++r)
      mbar_wait(smem_u32(&bars[kLoaded + r % kSmallStages]), (uint32_t)((r / kSmallStages) & 1),
                kCrtWaitLimit);
    if (g.status) atomicExch(g.status, (int)BTA_ERR_TIMEOUT);
  }
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * ST)
                 : "memory");
  }
}

// The kernels on operands and results run in blocks of 128 threads at no more than 48
// registers, one of which fits an SM's registers beside a CTA of crt_gemm_kernel (and 9 KB
// its shared memory), so that one leg's conversions proceed behind another's products; the
// smaller blocks also fill an SM more evenly (4800^3: residues 272 us with 256 threads, 252
// with 128; b = 4800, 8 blocks gradient 176.0 / 174.7 ms).
constexpr int kElemThreads = 128;
constexpr int kElemRows = 16;   // an operand's block: 16 rows x 64 columns

// ---- recovery ----------------------------------------------------------------

// alpha and beta as integer modes (decided on the host: comparisons of
// doubles would run on the FP64 pipe once per element): alpha 0 -> +1,
// 1 -> -1, 2 -> general; beta 0 -> 0, 1 -> +1, 2 -> general.
inline int alpha_mode(double a) { return a == 1.0 ? 0 : a == -1.0 ? 1 : 2; }
inline int beta_mode(double b) { return b == 0.0 ? 0 : b == 1.0 ? 1 : 2; }

__device__ __forceinline__ double scale_add(double out, int am, double alpha, int bm, double beta,
                                            double cin) {
  if (am == 1) out = -out;
  else if (am == 2) out *= alpha;
  if (bm == 1) out += cin;
  else if (bm == 2) out = fma(beta, cin, out);
  return out;
}

// C = alpha X 2^(exA + exB + scale) + beta Cin with X recovered from its residues:
// T = X / P 2^113 modulo 2^113 (signed; the fractions' rounding errors, 2^27 / 2 for each
// pair's y about its centre at most, are 2^40 of X, where the operands' last bit is worth
// 2^56), then |X| = |T| P 2^-113 by one 64-bit product of leading parts and one rounding.
// All residues zero give exactly zero.
struct ComposeArgs {
  int M, N, Mp, Np, out_lower, scale;
  double alpha, beta;
  int amode, bmode;
  double* C;
  int ldc;
  const double* Cin;
  int ldcin;
  // rows m >= c_rows (INT_MAX: none) go to C2 / Cin2, without the lower mask
  int c_rows;
  double* C2;
  int ldc2;
  const double* Cin2;
  int ldcin2;
  const int* exA;
  const int* exB;
  const uint16_t* R;
};

template <int I>
__device__ __forceinline__ void crt_add(const uint32_t (&r)[kNumMod], int half,
                                        unsigned long long (&l)[3]) {
  if constexpr (I < kNumMod) {
    using Q = ModPair<I>;
    const int x0 = half ? r[I] >> 16 : r[I] & 0xFFFFu;
    const int x1 = half ? r[I + 1] >> 16 : r[I + 1] & 0xFFFFu;
    const unsigned long long y = (uint32_t)(x1 * Q::b + (x0 * Q::a + Q::c));   // < 2^27
    l[0] += y * Q::f0;
    l[1] += y * Q::f1;
    l[2] += y * Q::f2;
    crt_add<I + 2>(r, half, l);
  }
}

__device__ __forceinline__ double crt_value(const uint32_t (&r)[kNumMod], int half, int E) {
  unsigned long long l[3] = {CrtOffset::l0, CrtOffset::l1, CrtOffset::l2};
  crt_add<0>(r, half, l);
  // words of T modulo 2^113 (signed), then of |T|
  uint32_t w[4];
  unsigned long long c = (l[0] >> 32) + (uint32_t)l[1];
  w[0] = (uint32_t)l[0];
  w[1] = (uint32_t)c;
  c = (c >> 32) + (l[1] >> 32) + l[2];
  w[2] = (uint32_t)c;
  w[3] = (uint32_t)((int)((uint32_t)(c >> 32) << (128 - kFracBits)) >> (128 - kFracBits));
  const bool neg = (int)w[3] < 0;
  if (neg)
    asm("sub.cc.u32 %0, 0, %0;\n subc.cc.u32 %1, 0, %1;\n subc.cc.u32 %2, 0, %2;\n"
        " subc.u32 %3, 0, %3;"
        : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]));
  // leading 64 bits u of the 128: |T| = u 2^(64 - lz)
  int lz = 0;
  while (w[3] == 0) {
    if (lz == 96) return 0.0;
    w[3] = w[2];
    w[2] = w[1];
    w[1] = w[0];
    w[0] = 0;
    lz += 32;
  }
  const int z = __clz((int)w[3]);
  lz += z - (128 - kFracBits);
  const unsigned long long u = (unsigned long long)__funnelshift_l(w[2], w[3], z) << 32 |
                               __funnelshift_l(w[1], w[2], z);
  // v 2^(E + 62 - lz) rounded to nearest even; v >= 2^62 as u and kPTop are >= 2^63
  unsigned long long v = __umul64hi(u, kPTop);
  int be = 1023 + 63 + 62 + E - lz;
  if (!(v >> 63)) {
    v <<= 1;
    --be;
  }
  if (be <= 0 || be >= 2046) return oz::compose_mag(neg, v, be - (1023 + 63));
  // may carry to 2^53, which the sum turns into the next exponent
  const unsigned long long m = (v >> 11) + ((v & 0x7FFull) + ((v >> 11) & 1ull) > 0x400ull);
  return __longlong_as_double(
      (long long)((neg ? 1ull << 63 : 0ull) + ((unsigned long long)(be - 1) << 52) + m));
}

// Thread: rows m, m + 1 of column n, whose residues (and the entries of Cin) are loaded
// before the first is used; the padding of R makes the load beyond row M harmless.
// Column bases are the same for a block, so a load's address is one 32-bit offset.
// Bound by instruction issue (4800^3: 200 us with 96-bit fractions per residue, 179 now).
__global__ void __launch_bounds__(kElemThreads) crt_compose_kernel(ComposeArgs g) {
  const unsigned m = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  await_prior();
  if (m >= (unsigned)g.M) return;
  const int64_t plane = (int64_t)g.Mp * g.Np;
  for (int n = blockIdx.y; n < g.N; n += gridDim.y) {
    if (g.out_lower && (int)m + 1 < n && (int)m + 1 < g.c_rows) break;
    uint32_t r[kNumMod];
    const uint16_t* col = g.R + (int64_t)n * g.Mp;
#pragma unroll
    for (int i = 0; i < kNumMod; ++i)
      r[i] = __ldg(reinterpret_cast<const unsigned int*>(col + i * plane + m));
    double ci[2];
    bool out[2], top[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int mm = (int)m + h;
      top[h] = mm < g.c_rows;
      out[h] = mm < g.M && !(g.out_lower && top[h] && mm < n);
      ci[h] = 0.0;
      if (out[h] && g.bmode)
        ci[h] = top[h] ? (g.Cin + (int64_t)n * g.ldcin)[mm]
                       : (g.Cin2 + (int64_t)n * g.ldcin2)[mm - g.c_rows];
    }
    const int eb = g.exB[n] + g.scale;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int mm = (int)m + h;
      if (!out[h]) continue;
      const double v = scale_add(crt_value(r, h, g.exA[mm] + eb), g.amode, g.alpha, g.bmode,
                                 g.beta, ci[h]);
      if (top[h]) (g.C + (int64_t)n * g.ldc)[mm] = v;
      else (g.C2 + (int64_t)n * g.ldc2)[mm - g.c_rows] = v;
    }
  }
}

// ---- residues of the operands ------------------------------------------------

// Element (r, k) of op(X) masked to its triangle (0 outside).
__device__ __forceinline__ double op_elem(const double* X, int ldx, int trans, int tri, int r,
                                          int k) {
  if ((tri == TRI_LOWER && k > r) || (tri == TRI_UPPER && k < r)) return 0.0;
  return trans ? X[k + (int64_t)r * ldx] : X[r + (int64_t)k * ldx];
}

// One operand to split: rows of op(X) (op(B)^T for the B side), their
// exponent bounds ex[rowsP] and planes Y (residue_kernel).  op(X) may be a 2 x 2
// block matrix cut after row rc and column kc: the leading block is (X, ldx,
// trans, tri), the others P[0] (rows < rc, k >= kc), P[1] (rows >= rc,
// k < kc) and P[2] (rows >= rc, k >= kc), each untriangular, zero when its
// pointer is null.  An operand without cuts has rc = kc = INT_MAX.  The
// leading block's trans also fixes the order in which the kernels read.
struct SplitPart {
  const double* X;
  int ld, trans;
};
struct SplitOp {
  const double* X;
  int ldx, trans, tri, rows, rowsP;
  int* ex;
  int* pm;   // [eblocks][rowsP] partial maxima of the exponents
  __nv_bfloat16* Y;
  int rc, kc;
  SplitPart P[3];
};

// Element (r, k) of a block part (r, k within op(X) as a whole).
__device__ __forceinline__ double op_part(const SplitOp& o, int r, int k) {
  const bool rb = r >= o.rc, kb = k >= o.kc;
  const SplitPart& q = !rb ? o.P[0] : !kb ? o.P[1] : o.P[2];
  if (!q.X) return 0.0;
  if (rb) r -= o.rc;
  if (kb) k -= o.kc;
  return q.trans ? q.X[k + (int64_t)r * q.ld] : q.X[r + (int64_t)k * q.ld];
}

// Element (r, k) of op(X): the leading block inline with its memory order
// TR known at compile time, then the other parts.
template <int TR>
__device__ __forceinline__ double op_get(const SplitOp& o, int r, int k) {
  if (r < o.rc && k < o.kc) return op_elem(o.X, o.ldx, TR, o.tri, r, k);
  return op_part(o, r, k);
}
struct SplitArgs {
  SplitOp op[2];   // blockIdx.z selects the operand
  int K, Kp;
  int bits;   // of the integers F (see the file's head)
  int eblocks;   // partial maxima per row (0: ex holds the exponents)
  int tile;      // of the products
  int mod0, nmod;   // the moduli whose planes are written
};

// The block of op(X) at (r0, k0), 8 elements a thread: thread t holds (r, k) = (t & 15,
// (t >> 4) + 8 i) with rows contiguous in memory, else ((t >> 6) + 2 i, t & 63).  A block
// outside the triangle is not read, and one that lies wholly inside it and the leading block
// takes 8 loads without tests between them: with the tests of the general form in between,
// each load waited for the one before it (4800^3: exponents 127 us, 61 without; residues
// 350, 272).
template <int TR>
__device__ __forceinline__ void load_block(const SplitOp& o, int K, int r0, int k0,
                                           double (&v)[8]) {
  const int t = threadIdx.x;
  const int rr = TR ? t >> 6 : t & 15, kk = TR ? t & 63 : t >> 4;
  const int r1 = r0 + kElemRows - 1, k1 = k0 + CK - 1;   // last row and column
  const bool zero = (o.tri == TRI_LOWER && k0 > r1) || (o.tri == TRI_UPPER && k1 < r0);
  const bool full = r1 < min(o.rows, o.rc) && k1 < min(K, o.kc) &&
                    !(o.tri == TRI_LOWER && k1 > r0) && !(o.tri == TRI_UPPER && k0 < r1);
  if (zero) {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = 0.0;
  } else if (full) {
    const double* x = TR ? o.X + (k0 + kk) + (int64_t)(r0 + rr) * o.ldx
                         : o.X + (r0 + rr) + (int64_t)(k0 + kk) * o.ldx;
    const int64_t step = (int64_t)(TR ? 2 : 8) * o.ldx;
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = x[i * step];
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = r0 + rr + (TR ? 2 * i : 0), k = k0 + kk + (TR ? 0 : 8 * i);
      v[i] = r < o.rows && k < K ? op_get<TR>(o, r, k) : 0.0;
    }
  }
}

// The row exponents: the biased exponent field's maximum over the 64 columns of block kb
// of op(X)[r][k].  Up to kPartialK columns it goes to pm[kb][r], of which residue_kernel
// takes the maximum (nothing to clear: two launches less on a short product's path);
// above, to ex[r] by an atomic maximum (ex zeroed beforehand).
constexpr int kPartialK = 1024;
__global__ void __launch_bounds__(kElemThreads) ozaki_exp_kernel(SplitArgs a) {
  const SplitOp o = blockIdx.z == 0 ? a.op[0] : a.op[1];
  const int r0 = blockIdx.x * kElemRows, k0 = blockIdx.y * CK;
  launch_next();
  if (r0 >= o.rows) return;
  __shared__ int smax[kElemRows];
  const int t = threadIdx.x;
  if (t < kElemRows) smax[t] = 0;
  __syncthreads();
  double v[8];
  auto field = [](double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); };
  if (!o.trans) {
    load_block<0>(o, a.K, r0, k0, v);
    int e = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) e = max(e, field(v[i]));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
    if ((t & 16) == 0) atomicMax(&smax[t & 15], e);
  } else {
    load_block<1>(o, a.K, r0, k0, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) {   // a warp shares its row
      const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)field(v[i]));
      if ((t & 31) == 0) atomicMax(&smax[(t >> 6) + 2 * i], e);
    }
  }
  __syncthreads();
  if (t >= kElemRows) return;
  if (a.eblocks) o.pm[(int64_t)blockIdx.y * o.rowsP + r0 + t] = smax[t];
  else if (r0 + t < o.rows && smax[t] > 0) atomicMax(&o.ex[r0 + t], smax[t]);
}

// F = v 2^(1022 + bits - er) rounded to an integer (see the file's head), as
// four signed 14-bit digits F = d3 2^42 + d2 2^28 + d1 2^14 + d0.
__device__ __forceinline__ void fixed_digits(double v, int er, int bits, float (&d)[4]) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int E = (int)((b >> 52) & 0x7FF);
  long long F = 0;
  if (E != 0) {
    const unsigned long long mant = (b & ((1ull << 52) - 1)) | (1ull << 52);
    const int sh = E - er + (bits - 53);
    if (sh >= 0) F = (long long)(mant << sh);
    else if (sh > -54) F = (long long)((mant + (1ull << (-sh - 1))) >> (-sh));
    if (b >> 63) F = -F;
  }
  const int hi = (int)((F + (1ll << 27)) >> 28);            // |hi| <= 2^28
  const int lo = (int)(F - (long long)hi * (1ll << 28));    // in [-2^27, 2^27)
  const int d0 = (lo << 18) >> 18, d2 = (hi << 18) >> 18;
  d[0] = oz::i2f_small(d0);
  d[1] = oz::i2f_small((lo - d0) >> 14);
  d[2] = oz::i2f_small(d2);
  d[3] = oz::i2f_small((hi - d2) >> 14);
}

// The plane of modulus I and the following ones: t = d0 + d1 c1 + d2 c2 + d3 c3 is
// congruent to F and |t| < 2^23 (|d3| <= 2^14, the others 2^13, |c| <= 255), so every
// FP32 step is exact and the rounded quotient the nearest one (the error of t / p is
// below 2^-24 |t| / p < 1 / (2 p)): |r| <= (p - 1) / 2, or p / 2 for the even modulus.
// All: of every modulus; else of nmod moduli from mod0 on (y: the plane of mod0).
template <bool All, int I>
__device__ __forceinline__ void residue_planes(const uint64_t (&d)[4][4], __nv_bfloat16* y,
                                               size_t plane, int mod0, int nmod) {
  if constexpr (I < kNumMod) {
    if (All || (unsigned)(I - mod0) < (unsigned)nmod) {
      using Q = Modulus<I>;
      const uint64_t c1 = pack2(Q::c1, Q::c1), c2 = pack2(Q::c2, Q::c2), c3 = pack2(Q::c3, Q::c3);
      const uint64_t inv = pack2(Q::inv, Q::inv), np = pack2(-Q::p, -Q::p);
      const uint64_t magic = pack2(kMagic, kMagic), nmagic = pack2(-kMagic, -kMagic);
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint64_t t = fma2(d[3][e], c3, fma2(d[2][e], c2, fma2(d[1][e], c1, d[0][e])));
        const uint64_t k = add2(fma2(t, inv, magic), nmagic);
        float r0, r1;
        unpack2(fma2(k, np, t), r0, r1);
        // at most 8 significant bits: the BF16 pattern is the upper half
        w[e] = __byte_perm(__float_as_uint(r0), __float_as_uint(r1), 0x7632);
      }
      *reinterpret_cast<uint4*>(y + (All ? I : I - mod0) * plane) =
          make_uint4(w[0], w[1], w[2], w[3]);
    }
    residue_planes<All, I + 1>(d, y, plane, mod0, nmod);
  }
}

// Y[i][k / 64][r][k % 64] (i < kNumMod, r < rowsP, k < Kp) = residue of op(X)[r][k] modulo
// p_i in BF16; zero in the padding, unwritten where no product reads it.  A 64-wide K slab
// of a plane is contiguous, so that a block writes 2 KB in a row to each plane, and a TMA
// load of the products reads 16 KB (not 128-byte pieces a row apart: 4800^3 call 2.95 ms,
// 3.05 so).  The block is staged through a swizzled shared tile: column c of row q sits at
// c ^ ((q ^ (c >> 3)) & 15), which keeps both the transposing writes (16 rows, one column)
// and the digit reads (2 rows x 8 column groups) of every half-warp on 16 distinct 8-byte
// banks.
__device__ __forceinline__ int split_swz(int q, int c) { return c ^ ((q ^ (c >> 3)) & 15); }

template <bool All>
__global__ void __launch_bounds__(kElemThreads) residue_kernel(SplitArgs a) {
  const SplitOp o = blockIdx.z == 0 ? a.op[0] : a.op[1];
  const int r0 = blockIdx.x * kElemRows, k0 = blockIdx.y * CK;
  if (r0 >= o.rowsP) return;
  // slabs outside the triangle of the products' tile are never read (crt_unit); the first
  // block of a row also writes the exponents
  const int t0 = r0 / a.tile * a.tile;
  if (blockIdx.y > 0 && ((o.tri == TRI_LOWER && k0 >= t0 + a.tile) ||
                         (o.tri == TRI_UPPER && k0 + CK <= t0)))
    return;
  __shared__ double tile[kElemRows][CK];   // tile[r - r0][split_swz(r - r0, k - k0)]
  __shared__ int s_er[8][kElemRows];
  const int t = threadIdx.x;
  double v[8];
  if (!o.trans) {
    load_block<0>(o, a.K, r0, k0, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) tile[t & 15][split_swz(t & 15, (t >> 4) + 8 * i)] = v[i];
  } else {
    load_block<1>(o, a.K, r0, k0, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int rr = (t >> 6) + 2 * i;
      tile[rr][split_swz(rr, t & 63)] = v[i];
    }
  }
  await_prior();
  launch_next();
  if (a.eblocks) {   // the rows' exponents: each eighth of the threads takes every eighth one
    const int r = r0 + (t & 15);
    int e = 0;
    if (r < o.rows)
      for (int b = t >> 4; b < a.eblocks; b += 8) e = max(e, o.pm[(int64_t)b * o.rowsP + r]);
    s_er[t >> 4][t & 15] = e;
  }
  __syncthreads();
  const size_t plane = (size_t)o.rowsP * a.Kp;   // of one modulus
  // thread: row q = t >> 3 and columns 8 g .. 8 g + 7, g = t & 7, so that a
  // warp writes 4 rows x 128 contiguous bytes of each plane, one 16-byte
  // store per thread and plane
  const int q = t >> 3, g = t & 7, r = r0 + q;
  int er = 0;
  if (a.eblocks) {
#pragma unroll
    for (int w = 0; w < 8; ++w) er = max(er, s_er[w][q]);
    if (blockIdx.y == 0 && g == 0 && r < o.rows) o.ex[r] = er;
  } else if (r < o.rows) {
    er = o.ex[r];
  }
  uint64_t d[4][4];   // [digit][pair of columns]
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    float x[4], y[4];
    fixed_digits(tile[q][split_swz(q, 8 * g + e)], er, a.bits, x);
    fixed_digits(tile[q][split_swz(q, 8 * g + e + 1)], er, a.bits, y);
#pragma unroll
    for (int j = 0; j < 4; ++j) d[j][e / 2] = pack2(x[j], y[j]);
  }
  residue_planes<All, 0>(d, o.Y + ((size_t)blockIdx.y * o.rowsP + r) * 64 + 8 * g, plane, a.mod0,
                         a.nmod);
}

// 2D map over Y viewed as rowsAll = moduli * slabs * rowsP rows of 64 BF16, box 128 rows.
bta_status make_map_bf16(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap* map,
                         const __nv_bfloat16* base, int rowsAll) {
  cuuint64_t dims[2] = {(cuuint64_t)CK, (cuuint64_t)rowsAll};
  cuuint64_t strides[1] = {(cuuint64_t)CK * 2};
  cuuint32_t box[2] = {(cuuint32_t)CK, (cuuint32_t)CH};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(base),
                   dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? BTA_OK : BTA_ERR_ARG;
}

// CTA pairs that fit on the GPU at once (1 CTA per SM; a pair needs two SMs of
// one cluster-capable group), queried once per device.
int pair_slots() {
  static int cache[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    dev = 0;
  }
  int* slot = dev >= 0 && dev < 64 ? &cache[dev] : nullptr;
  if (slot && *slot > 0) return *slot;
  int n = 0;
  if (cudaFuncSetAttribute(crt_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kCrtSmem) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * 512);
    cfg.blockDim = dim3(kCrtThreads);
    cfg.dynamicSmemBytes = kCrtSmem;
    if (cudaOccupancyMaxActiveClusters(&n, crt_gemm_kernel, &cfg) != cudaSuccess) n = 0;
  }
  cudaGetLastError();
  if (n < 1) n = std::max(1, sm_count() / 2);
  if (slot) *slot = n;
  return n;
}

// Tile size of a product: pairs of CTAs on 256 x 256 tiles, or, while all units of 128 x
// 128 tiles fit the GPU about four times over, single CTAs on those.  There a product is
// bound by latency and by finding free SMs beside the leaves of other legs, above by
// operand loads, which the larger tile halves.  Product kernel alone, pairs / single CTAs:
// 192^3 12.8 / 8.8 us, 512^3 15.1 / 11.9, 1024^3 35.9 / 35.4.
int crt_tile(int M, int N) {
  const int64_t units = (int64_t)cdiv(M, ST) * cdiv(N, ST) * kNumMod;
  return units <= 8 * sm_count() ? ST : CT;
}

struct OzLayout {
  int Mp, Np, Kp, eblocks;
  size_t a_off, b_off, ea_off, eb_off, pa_off, pb_off, r_off, total;
  OzLayout(int M, int N, int K, int tile, int group) {
    Mp = cdiv(M, tile) * tile;
    Np = cdiv(N, tile) * tile;
    Kp = cdiv(K, CK) * CK;
    eblocks = K <= kPartialK ? cdiv(K, CK) : 0;
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    b_off = 0;   // B's part first: where it lies does not depend on M (Gemm::b_kept)
    pb_off = up((size_t)group * Np * Kp * 2);
    eb_off = pb_off + up((size_t)eblocks * Np * 4);
    ea_off = eb_off + up((size_t)Np * 4);   // (one memset clears both ex)
    pa_off = ea_off + up((size_t)Mp * 4);
    a_off = pa_off + up((size_t)eblocks * Mp * 4);
    r_off = a_off + up((size_t)group * Mp * Kp * 2);
    total = r_off + up((size_t)kNumMod * Mp * Np * 2) + 256;
  }
};

// marks (optional): two events recorded on s around the tensor-core product
// kernel's launch alone (the measurement entry point bta_gemm_emulated_timed).
bta_status launch_ozaki(const Gemm& g, uint8_t* ws, int32_t* status, cudaStream_t s,
                        const cudaEvent_t* marks, int group) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = nullptr;
  BTA_TRY(tensor_map_encoder(&enc));
  const int M = g.M, N = g.N, K = g.K;
  const int tile = crt_tile(M, N);
  const OzLayout L(M, N, K, tile, group);
  __nv_bfloat16* YA = reinterpret_cast<__nv_bfloat16*>(ws + L.a_off);
  __nv_bfloat16* YB = reinterpret_cast<__nv_bfloat16*>(ws + L.b_off);
  int* exA = reinterpret_cast<int*>(ws + L.ea_off);
  int* exB = reinterpret_cast<int*>(ws + L.eb_off);
  uint16_t* R = reinterpret_cast<uint16_t*>(ws + L.r_off);
  // rows of op(B)^T: Y[n][k] = op(B)[k][n]; the triangle flips with the transpose
  const int trib = g.triB == TRI_LOWER ? TRI_UPPER : g.triB == TRI_UPPER ? TRI_LOWER : TRI_NONE;
  // op(B)^T == the first N rows of op(A) (the symmetric update L L^T, with
  // or without extra rows of A below): one set of planes serves both
  const bool b_parts = g.B12.X || g.B21.X || g.B22.X || g.b_k || g.b_cols;
  const bool a_kparts = g.A12.X || g.A22.X || g.a_k;
  const bool same = g.A == g.B && g.lda == g.ldb && g.transA == !g.transB && g.triA == trib &&
                    !b_parts && !a_kparts && N <= (g.a_rows ? g.a_rows : M);
  SplitArgs sa;
  sa.K = K;
  sa.Kp = L.Kp;
  sa.bits = K <= kMaxK56 ? 56 : 55;
  sa.eblocks = L.eblocks;
  sa.tile = tile;
  auto cut = [](int c) { return c > 0 ? c : INT_MAX; };
  sa.op[0] = {g.A, g.lda, g.transA, g.triA, M, L.Mp, exA,
              reinterpret_cast<int*>(ws + L.pa_off), YA, cut(g.a_rows), cut(g.a_k),
              {{g.A12.X, g.A12.ld, g.A12.trans},
               {g.A21.X, g.A21.ld, g.A21.trans},
               {g.A22.X, g.A22.ld, g.A22.trans}}};
  // the B side holds op(B)^T: its row cut is op(B)'s column cut and each
  // part is the transpose of the matching block of op(B)
  sa.op[1] = {g.B, g.ldb, !g.transB, trib, N, L.Np, exB,
              reinterpret_cast<int*>(ws + L.pb_off), YB, cut(g.b_cols), cut(g.b_k),
              {{g.B21.X, g.B21.ld, !g.B21.trans},
               {g.B12.X, g.B12.ld, !g.B12.trans},
               {g.B22.X, g.B22.ld, !g.B22.trans}}};
  // op(B)'s planes from the product before (laid out alike), in a symmetric product op(A)'s
  // too (b = 4800, 8 blocks gradient 174.5 ms without, 171.1 with)
  const bool kept = g.b_kept > 0 && group == kNumMod && crt_tile(g.b_kept, N) == tile &&
                    (!same || (L.Mp <= L.Np && !g.a_rows));
  const int nops = (same ? 1 : 2) - (kept ? 1 : 0);
  if (same && kept) {
    YA = YB;
    exA = exB;
  }
  if (nops > 0) {
    const int rows = nops > 1 ? std::max(M, N) : M;
    if (!L.eblocks) {
      if (kept) BTA_CUDA_TRY(cudaMemsetAsync(exA, 0, L.pa_off - L.ea_off, s));
      else BTA_CUDA_TRY(cudaMemsetAsync(exB, 0, L.pa_off - L.eb_off, s));
    }
    ozaki_exp_kernel<<<dim3(cdiv(rows, kElemRows), cdiv(K, CK), nops), kElemThreads, 0, s>>>(sa);
    BTA_LAUNCHED();
  }
  CrtArgs q{};
  q.Mp = L.Mp; q.Np = L.Np; q.Ap = same && kept ? L.Np : L.Mp; q.Bp = same ? q.Ap : L.Np;
  q.nk = L.Kp / CK;
  q.mt = L.Mp / tile;
  q.nt = L.Np / tile;
  // tile row i holds columns up to i; a C2 row (row >= c_rows) needs every column, so
  // it must lie in a row of tiles that holds them all
  q.lower = g.out_lower && !(g.C2 && g.c_rows / tile < q.nt - 1);
  const int h = std::min(q.mt, q.nt);
  q.tiles = q.lower ? h * (h + 1) / 2 + (q.mt - h) * q.nt : q.mt * q.nt;
  q.tri_a = g.triA;
  q.tri_b = g.triB;
  q.R = R;
  q.status = status;
  static std::atomic<uint64_t> allowed[2];
  if (tile == ST)
    BTA_TRY(allow_smem(allowed[0], reinterpret_cast<const void*>(&crt_gemm_small_kernel),
                       kSmallSmem));
  else
    BTA_TRY(allow_smem(allowed[1], reinterpret_cast<const void*>(&crt_gemm_kernel), kCrtSmem));
  // group by group: planes of its moduli, then their products (a group's residues wait for
  // the products of the one before, whose planes they overwrite)
  for (int m0 = 0; m0 < kNumMod; m0 += group) {
    sa.mod0 = q.mod0 = m0;
    sa.nmod = q.nmod = std::min(group, kNumMod - m0);
    if (nops > 0) {
      const int rowsP = nops > 1 ? std::max(L.Mp, L.Np) : L.Mp;
      BTA_CUDA_TRY(launch_after(group == kNumMod ? residue_kernel<true> : residue_kernel<false>,
                                dim3(rowsP / kElemRows, L.Kp / CK, nops), dim3(kElemThreads), 0,
                                s, sa));
      BTA_LAUNCHED();
    }
    CUtensorMap mA, mB;
    BTA_TRY(make_map_bf16(enc, &mA, YA, q.nmod * q.nk * q.Ap));
    BTA_TRY(make_map_bf16(enc, &mB, same ? YA : YB, q.nmod * q.nk * q.Bp));
    const int units = q.tiles * q.nmod;
    if (marks && m0 == 0) BTA_CUDA_TRY(cudaEventRecord(marks[0], s));
    if (tile == ST) {
      q.group = q.mt;
      BTA_CUDA_TRY(launch_after(crt_gemm_small_kernel, dim3(units), dim3(kCrtThreads), kSmallSmem,
                                s, mA, mB, q));
    } else {
      // A wave of pairs spans a near-square patch of tiles.  A pair takes several units
      // (the store of one overlaps the next) but at most ~300 slabs, ~75 us, so that the
      // launches of a concurrent sweep find free SMs.
      q.slots = pair_slots();
      q.group = std::min(q.mt, std::max(1, (int)std::lround(std::sqrt((double)q.slots))));
      q.slots = std::min(q.slots, units);
      q.per = std::max(1, std::min(cdiv(units, q.slots), 300 / q.nk));
      BTA_CUDA_TRY(launch_after(crt_gemm_kernel, dim3(2 * q.slots * cdiv(units, q.slots * q.per)),
                                dim3(kCrtThreads), kCrtSmem, s, mA, mB, q));
    }
    BTA_LAUNCHED();
  }
  if (marks) BTA_CUDA_TRY(cudaEventRecord(marks[1], s));
  ComposeArgs c;
  c.M = M; c.N = N; c.Mp = L.Mp; c.Np = L.Np;
  c.out_lower = g.out_lower;
  c.scale = -2044 - 2 * sa.bits;
  c.alpha = g.alpha; c.beta = g.beta; c.C = g.C; c.ldc = g.ldc;
  c.amode = alpha_mode(g.alpha); c.bmode = beta_mode(g.beta);
  c.Cin = g.Cin ? g.Cin : g.C; c.ldcin = g.Cin ? g.ldcin : g.ldc;
  c.c_rows = g.C2 ? g.c_rows : INT_MAX;
  c.C2 = g.C2; c.ldc2 = g.ldc2;
  c.Cin2 = g.Cin2 ? g.Cin2 : g.C2; c.ldcin2 = g.Cin2 ? g.ldcin2 : g.ldc2;
  c.exA = exA; c.exB = same ? exA : exB; c.R = R;
  BTA_CUDA_TRY(launch_after(crt_compose_kernel, dim3(cdiv(M, 2 * kElemThreads), std::min(N, 65535)),
                            dim3(kElemThreads), 0, s, c));
  BTA_LAUNCHED();
  return BTA_OK;
}

}  // namespace

// An upper bound over every product of at most M x N x K: a sweep sizes one
// workspace for all of its products (the larger tile's layout, and the partial maxima of a
// smaller K).
size_t ozaki_ws_bytes(int M, int N, int K, int group) {
  const size_t full = OzLayout(M, N, K, CT, group).total;
  return K > kPartialK ? std::max(full, OzLayout(M, N, kPartialK, CT, group).total) : full;
}

bool ozaki_supported(const Gemm& g) {
  if (!(g.batch == 1 && !g.Ab && g.A && g.B && g.C && g.K >= 1 && g.K <= kOzakiMaxK && g.M >= 1 &&
        g.N >= 1))
    return false;
  if (!g.blocked()) return true;
  // block operands: cuts inside the matrix, parts only where a cut makes
  // room for them, no triangle in an operand with parts, C2 with its cut
  auto in = [](int c, int n) { return c == 0 || (c > 0 && c < n); };
  auto ok = [](const Gemm::Part& q) { return !q.X || q.ld >= 1; };
  if (!in(g.a_rows, g.M) || !in(g.a_k, g.K) || !in(g.b_k, g.K) || !in(g.b_cols, g.N) ||
      !in(g.c_rows, g.M))
    return false;
  if (!ok(g.A12) || !ok(g.A21) || !ok(g.A22) || !ok(g.B12) || !ok(g.B21) || !ok(g.B22))
    return false;
  if ((g.A21.X || g.A22.X) && !g.a_rows) return false;
  if ((g.A12.X || g.A22.X) && !g.a_k) return false;
  if ((g.B21.X || g.B22.X) && !g.b_k) return false;
  if ((g.B12.X || g.B22.X) && !g.b_cols) return false;
  if ((g.a_rows || g.a_k) && g.triA != TRI_NONE) return false;
  if ((g.b_k || g.b_cols) && g.triB != TRI_NONE) return false;
  if ((g.C2 != nullptr) != (g.c_rows > 0) || (g.C2 && g.ldc2 < 1)) return false;
  if (g.Cin2 && g.ldcin2 < 1) return false;
  return true;
}

bta_status ozaki_gemm(const Gemm& g, void* ws, int32_t* status, cudaStream_t s,
                      const cudaEvent_t* marks, int group) {
  if (g.M <= 0 || g.N <= 0) return BTA_OK;
  if (!ozaki_supported(g) || !ws || group < 1 || group > kNumMod) return BTA_ERR_ARG;
  uint8_t* w = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ws) + 255) &
                                          ~(uintptr_t)255);
  return launch_ozaki(g, w, status, s, marks, group);
}

}  // namespace bta
