// Block sweeps over a BTA descriptor (sweep.cu).
#pragma once

#include "model.cuh"

namespace bta {

// Scratch for one sweep: three ld x ld blocks, an a x ld arrow block, a solve vector and
// the arrow accumulator v_T.  W2 holds low-memory sweeps' assembled couplings, and before
// a block's coupling is assembled (in the others throughout) its diagonal factor's scratch.
struct SweepWs {
  double *W1 = nullptr, *W2 = nullptr, *W3 = nullptr;
  double *Wc1 = nullptr, *gv = nullptr, *vT = nullptr;   // gv: ld
  // tensor-core modes only: operand copies of the products (sweep_tc_ws_bytes), the moduli
  // whose planes they hold at once (ozaki_gemm) and the products' status word (set by the
  // owner, not by carve)
  void* tc = nullptr;
  int tcgroup = kOzakiModuli;
  int32_t* tcstat = nullptr;
  static size_t bytes(int ld, int a);
  void carve(double* base, int ld, int a);
};

// The Eq. 7 reductions of a selected inversion (selinv_sums).
struct SelinvFuse {
  const ModelDev* md = nullptr;
  int counts = 0;          // add the observation-count diagonal (Q_c)
  double* PD = nullptr;    // [nt][kk][pchunks][kNP]
  double* PB = nullptr;    // [nt-1][kk][pchunks][kNP]
  double* PC = nullptr;    // [nt][k][achunks] or null
};

int logdet_slots(int n, int ld);   // n * (ld / 32) + 1 (tip)

// Emulated FP64 (precision 2) carries the arrow through the b x b products
// of both sweeps: its a rows ride along the rows of the product that shares
// their right-hand operand (in the row padding when b is not a multiple of
// 128), and its rank-a terms extend K, so that no FP64 product of the a x b
// arrow blocks with a b x b block is left per block step.
bool arrow_fused(int ld, int a, int precision);
// Bytes of the tensor-core workspace (SweepWs::tc) of a sweep of block size ld and arrow a
// in the given precision, the arrow-extended products and the diagonal factor's included.
size_t sweep_tc_ws_bytes(int ld, int a, int precision, int group = kOzakiModuli);

// One matrix of a set swept together, or one leg of it.  All matrices of a set share n and
// ld; the arrow width may differ (Q_c with a > 0 next to the block-tridiagonal
// Q_p).  Every block step of the sweep is then one launch over the set.
//
// A matrix may be eliminated from both ends towards a shared block: a forward leg
// takes blocks 0, 1, .. and a reverse leg (rev) the blocks n-1, n-2, ..; each counts
// its blocks from its own end, len of them with the shared block last, which
// belongs to the forward leg.  The order of elimination changes no result beyond rounding
// (log|Q|, x* and the selected inverse are the matrix's), takes the same products, and
// halves the serial chain of diagonal factors.  The reverse leg's couplings stay in their
// slots, as the factor's block Q[i-1, i] L_Di^{-T} of its own order.
struct SweepItem {
  bta_desc q{};
  double* vec = nullptr;           // factor: rhs -> z (or null); solves: z -> x
  double* slots = nullptr;         // factor: log-det slots
  int32_t* fail = nullptr;         // factor: failure flag (first failing block)
  SweepWs ws;
  const SelinvFuse* fuse = nullptr;   // Eq. 7 sums (or null)
  int rev = 0;                     // reverse leg
  int len = 0;                     // blocks of the leg, the shared one included (0: all)
  double* tip = nullptr;           // reverse leg: its share of the tip (a x a), else null
  const double* tip2 = nullptr;    // forward leg: the reverse leg's share of the tip and
  const double* vT2 = nullptr;     // of v_T (null: none)
  // Low-memory sweeps (q.B == nullptr): the off-diagonal factors L_Bi are not
  // kept; B_i is assembled from the model when a step needs it and L_Bi =
  // B_i L_Di^{-T} recomputed.
  const ModelDev* md = nullptr;
  const CoefLayout* lay = nullptr;
  const double* coef = nullptr;
  int blocks() const { return len > 0 ? len : q.n; }
};
// precision 0: every product in FP64; 1: the b x b off-diagonal Schur
// products (and the selected-inversion products) in split precision on the
// tensor cores, the diagonal-block factorisation to FP64 accuracy (in FP64 up to 512
// rows, above with emulated products: potrf_inv_batch_prec), arrow and log-det in
// FP64; 2: the b x b products emulated in FP64, the diagonal factor as in 1.
// Block range (optional): blocks i0 <= i < i1 of the factor sweep (i1 < 0:
// to the end) and i_hi >= i >= i_lo of the solves and the selected inversion
// (i_hi < 0: from the last block), the set-up with the first block and the tip with
// the last, so that consecutive ranges issue exactly the whole sweep.  A
// caller interleaves several sweeps' ranges to create their operations (and the
// nodes of a captured graph) in alternation.  A reverse leg's factor ends before
// the shared block, which it updates (D, C and the vector) at the end of its last
// range: the forward leg's step of that block, the tip and the shared block's x and Z must
// be ordered after it, and the reverse leg's solve and selected inversion (from
// block len - 2) after theirs.
//
// sv (optional, not for low-memory sweeps; ev an event of its own): a block's vector part,
// the arrow where no b x b product carries it, and the tip's share go to this stream, after
// the block's factor on s; they read finished parts of the factor only.  s waits for it
// before the tip; a reverse leg's last share, which updates the shared block's, stays on sv.
bta_status factor_sweep_multi(const SweepItem* items, int m, cudaStream_t s, int precision = 0,
                              int i0 = 0, int i1 = -1, cudaStream_t sv = nullptr,
                              cudaEvent_t ev = nullptr);
bta_status upper_solve_multi(const SweepItem* items, int m, cudaStream_t s, int i_hi = -1,
                             int i_lo = 0);
bta_status selinv_sweep_multi(const SweepItem* items, int m, cudaStream_t s, int precision = 0,
                              int i_hi = -1, int i_lo = 0);

bta_status factor_sweep(const bta_desc& q, double* rhs, double* slots, int32_t* fail,
                        const SweepWs& ws, cudaStream_t s, int precision = 0);
// The Eq. 7 sums of inverted matrices (items with fuse), all blocks in one launch per
// array; after every leg.
bta_status selinv_sums(const SweepItem* items, int m, cudaStream_t s);
// d <- d - Q x for an assembled BTA matrix Q (D lower triangle referenced, B,
// C, T as in bta_desc); x, d: n*ld + a.
bta_status bta_residual(const bta_desc& q, const double* x, double* d, cudaStream_t s);
// L z = r in place of item.vec with a forward factor (B kept).
bta_status lower_solve(const SweepItem& item, cudaStream_t s);
bta_status selinv_sweep(const bta_desc& q, const SweepWs& ws, const SelinvFuse* fuse,
                        cudaStream_t s);

}  // namespace bta
