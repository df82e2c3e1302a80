// C ABI: model set-up, the bta_* descriptor calls and inla_value_and_grad.
//
// inla_value_and_grad runs, for one theta (Eq. 1 and Eq. 6):
//   stream 0 : theta -> coefficients (closed-form Kronecker coefficients and
//              their theta-derivatives)
//   stream 1 : assemble Q_c, r -> Algorithm 1 with fused lower solve ->
//              Eqs. 3-5 -> x*, residuals ->  [grad] selected inversion of Q_c, Phase A sums
//   stream 2 : assemble Q_p -> block Cholesky -> (after x*) stencil quadratic
//              forms (Phase B, x*^T Q_p x*) -> [grad] selected inversion of Q_p,
//              Phase C sums
//   streams 3, 4 : the reverse legs of Q_c and Q_p (three time blocks or more)
//   streams 5, 6 : the vector's part of Q_c's legs, the sums over x
//   stream 0 : join, final combination into f and grad.
// Both matrices are eliminated from both ends towards the middle block (see SweepItem), so
// four chains of dependent block steps run concurrently and fill each other's idle SMs.
// The whole evaluation is captured once into a CUDA graph per (value / value+grad)
// and replayed.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <new>
#include <vector>

#include "sweep.cuh"

using namespace bta;

// One evaluation context: everything a single theta's evaluation writes.
struct EvalCtx {
  double* coefbuf = nullptr;
  bta_desc qc{}, qp{};
  double* x = nullptr;          // r -> z -> x*  (n*ld + a)
  double* slots_c = nullptr;
  double* slots_p = nullptr;
  int32_t* fail = nullptr;      // [2]
  double *PDc = nullptr, *PBc = nullptr, *PCc = nullptr, *PDp = nullptr, *PBp = nullptr;
  double *QD = nullptr, *QB = nullptr, *RS = nullptr;
  double* out = nullptr;
  // forward legs of Q_c and Q_p, then the reverse ones (null until a call takes them)
  SweepWs legs[4];
  void* tc[3][4] = {};            // [precision][leg]: operand copies (null until used)
  int group[3] = {};              // SweepWs::tcgroup of tc[precision]
  double* tip2 = nullptr;         // the reverse leg's share of Q_c's tip
  SelinvFuse fc, fp;
  double* dr = nullptr;         // mixed mode: refinement residual / correction
  double* red = nullptr;        // sums of the final combination
  int have_factors = 0;         // last evaluation was value-only: factors still held ...
  int reverse = 0;              // ... of so many blocks in the reverse legs
};

struct GraphKey {
  int mode, count, precision, reverse;
  cudaGraphExec_t exec;
  int64_t kernels;
};

struct inla_model {
  ModelDev md;
  CoefLayout L;
  int n = 0, b = 0, ld = 0, a = 0, d = 0;
  int nslots = 0;
  int lowmem = 0;               // keep only the diagonal factors (see inla_model_spec)
  std::vector<EvalCtx> ctx;     // grown on demand (batched evaluations)
  std::vector<void*> allocs;
  // host
  double* hout = nullptr;       // pinned, kMaxBatch outputs
  double* htheta = nullptr;     // pinned, kMaxBatch thetas
  std::vector<double> last;     // output of the last single evaluation
  std::vector<GraphKey> graphs;
  int64_t launched = 0;         // kernels this model ran (graph replays included)
  // the legs of the Q_c set (s1, s3) and of the Q_p set (s2, s4) are swept on four streams,
  // the vector's part of Q_c's legs on two more (s5, s6; fork/join by events)
  cudaStream_t s1 = nullptr, s2 = nullptr, s3 = nullptr, s4 = nullptr, s5 = nullptr, s6 = nullptr;
  cudaStream_t s0 = nullptr;    // the model's own root stream inside a multi-model graph
  cudaEvent_t ev0 = nullptr, evx = nullptr, ev1 = nullptr, ev2 = nullptr;
  // reverse legs: assembled, ready for the shared block, shared block done, finished
  cudaEvent_t evac = nullptr, evap = nullptr, evjc = nullptr, evjp = nullptr, evmc = nullptr,
              evmp = nullptr, ev3 = nullptr, ev4 = nullptr;
  // vector streams: a block's factor ready (either leg), the shared block's part, its x, the
  // solve of a block (either leg), finished
  cudaEvent_t evv5 = nullptr, evv6 = nullptr, evjv = nullptr, evmv = nullptr, evs5 = nullptr,
              evs6 = nullptr, ev5 = nullptr;
  cudaEvent_t evj = nullptr;    // join event of a multi-model graph
  int small[3] = {};            // [precision]: form of the workspaces (kFormGroup)
  // blocks of the reverse legs: both ends meet in the middle
  // (mixed precision keeps the forward order: see group_program)
  int reverse_blocks(int prec) const {
    return n >= 3 && prec != 1 && !small[prec] ? (n - 1) / 2 : 0;
  }
};

// Several models evaluated by one CUDA graph (see inla_batch_value_and_grad).
struct inla_batch {
  std::vector<inla_model*> models;
  cudaGraphExec_t exec[2][3] = {};   // [grad][precision]
  int64_t kernels[2][3] = {};
  std::vector<int> reverse[2][3];   // of each model, in exec
  cudaEvent_t fork = nullptr;
};

namespace {

template <class T>
bta_status dmalloc(inla_model* m, T** p, size_t count) {
  void* q = nullptr;
  if (count == 0) { *p = nullptr; return BTA_OK; }
  cudaError_t e = cudaMalloc(&q, count * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return BTA_ERR_NOMEM;
  }
  m->allocs.push_back(q);
  *p = static_cast<T*>(q);
  return BTA_OK;
}

template <class T>
bta_status upload(inla_model* m, T** p, const T* host, size_t count) {
  BTA_TRY(dmalloc(m, p, count));
  if (count) BTA_CUDA_TRY(cudaMemcpy(*p, host, count * sizeof(T), cudaMemcpyHostToDevice));
  return BTA_OK;
}

bool finite_theta(const double* th, int d) {
  for (int i = 0; i < d; ++i)
    if (!std::isfinite(th[i])) return false;
  return true;
}

// Free what was allocated since the model held `mark` buffers.
void roll_back(inla_model* m, size_t mark) {
  for (; m->allocs.size() > mark; m->allocs.pop_back()) cudaFree(m->allocs.back());
}

// Work blocks of a context's legs first and first + 1 (Q_c's and Q_p's).
void leg_carve(const inla_model* m, EvalCtx& c, int first, double* buf) {
  const size_t wsb = SweepWs::bytes(m->ld, m->a) / sizeof(double);
  for (int q = 0; q < 2; ++q) {
    c.legs[first + q].carve(buf + q * wsb, m->ld, m->a);
    c.legs[first + q].tcstat = c.fail + 2;
  }
}

// Allocate evaluation context c (buffers for Q_c, Q_p, x*, reductions).
bta_status ctx_alloc(inla_model* m, EvalCtx& c) {
  const ModelDev& md = m->md;
  const int nt = md.nt, ld = md.ld, a = md.a, k = md.k;
  const size_t blk = (size_t)ld * ld;
  BTA_TRY(dmalloc(m, &c.coefbuf, m->L.total));
  c.qc.n = nt; c.qc.b = md.b; c.qc.a = a; c.qc.ld = ld;
  BTA_TRY(dmalloc(m, &c.qc.D, nt * blk));
  if (!m->lowmem) BTA_TRY(dmalloc(m, &c.qc.B, std::max(nt - 1, 1) * blk));
  BTA_TRY(dmalloc(m, &c.qc.C, std::max<size_t>((size_t)nt * a * ld, 1)));
  BTA_TRY(dmalloc(m, &c.qc.T, std::max(a * a, 1)));
  c.qp = c.qc;
  c.qp.a = 0; c.qp.C = nullptr; c.qp.T = nullptr;
  BTA_TRY(dmalloc(m, &c.qp.D, nt * blk));
  if (!m->lowmem) {
    BTA_TRY(dmalloc(m, &c.qp.B, std::max(nt - 1, 1) * blk));
  } else {
    c.qp.B = nullptr;
  }
  BTA_TRY(dmalloc(m, &c.x, (size_t)nt * ld + a));
  BTA_TRY(dmalloc(m, &c.slots_c, m->nslots));
  BTA_TRY(dmalloc(m, &c.slots_p, m->nslots));
  BTA_TRY(dmalloc(m, &c.fail, 4));   // [0] Q_c pivot, [1] Q_p pivot, [2] tensor-core status
  const size_t pblk = (size_t)k * k * pattern_chunks(md) * kNP;
  BTA_TRY(dmalloc(m, &c.PDc, nt * pblk));
  BTA_TRY(dmalloc(m, &c.PBc, std::max(nt - 1, 1) * pblk));
  BTA_TRY(dmalloc(m, &c.PCc, std::max<size_t>((size_t)nt * k * arrow_chunks(md), 1)));
  BTA_TRY(dmalloc(m, &c.PDp, nt * pblk));
  BTA_TRY(dmalloc(m, &c.PBp, std::max(nt - 1, 1) * pblk));
  BTA_TRY(dmalloc(m, &c.QD, nt * pblk));
  BTA_TRY(dmalloc(m, &c.QB, std::max(nt - 1, 1) * pblk));
  // residual_kernel writes kMaxK rows
  BTA_TRY(dmalloc(m, &c.RS, (size_t)kMaxK * resid_chunks(md)));
  BTA_TRY(dmalloc(m, &c.out, out_size(md.d)));
  BTA_TRY(dmalloc(m, &c.red, kRedDoubles));
  double* wsbuf = nullptr;   // every evaluation takes the forward legs
  BTA_TRY(dmalloc(m, &wsbuf, 2 * SweepWs::bytes(ld, a) / sizeof(double)));
  leg_carve(m, c, 0, wsbuf);
  BTA_TRY(dmalloc(m, &c.tip2, std::max(a * a, 1)));
  BTA_TRY(dmalloc(m, &c.dr, (size_t)nt * ld + a));
  c.fc.md = &m->md; c.fc.counts = 1; c.fc.PD = c.PDc; c.fc.PB = c.PBc; c.fc.PC = c.PCc;
  c.fp.md = &m->md; c.fp.counts = 0; c.fp.PD = c.PDp; c.fp.PB = c.PBp; c.fp.PC = nullptr;
  return BTA_OK;
}

bta_status ensure_ctx(inla_model* m, int count) {
  if ((int)m->ctx.size() >= count) return BTA_OK;
  cudaDeviceSynchronize();
  m->ctx.reserve(count);
  while ((int)m->ctx.size() < count) {
    m->ctx.emplace_back();
    const size_t mark = m->allocs.size();
    bta_status st = ctx_alloc(m, m->ctx.back());
    if (st != BTA_OK) {
      m->ctx.pop_back();
      roll_back(m, mark);
      return st;
    }
  }
  // contexts hold pointers to the model: the fuse blocks refer to m->md (stable)
  return BTA_OK;
}

// The workspaces of an evaluation in a precision: a context's legs take three work blocks
// each, and in the tensor-core modes their products' operand copies (emulated: 84 bytes an
// entry of a block, as much as ten blocks).  They are allocated when a call first needs
// them, outside capture.  The smaller forms have one leg per matrix and hold the planes of seven moduli at
// once (56 bytes an entry), or of four (44).  They are taken in turn where the one before does
// not fit the device, so that a model whose matrices leave little room is evaluated all the
// same; low-memory models whose full form would exceed kLowMemoryWork begin with the first of
// them (b = 4800 emulated, 5 blocks: 3.5 GiB instead of 9.5, gradient 126 ms instead of 113).
// BTA_SMALL_WORKSPACES = 1 or 2 asks for one.
constexpr size_t kLowMemoryWork = (size_t)1 << 30;
constexpr int kWorkForms = 3;
constexpr int kFormGroup[kWorkForms] = {kOzakiModuli, 7, kOzakiSmallGroup};

size_t work_bytes(const inla_model* m, int prec) {
  const size_t legs = m->reverse_blocks(prec) > 0 ? 4 : 2;
  return legs * (SweepWs::bytes(m->ld, m->a) +
                 (prec ? sweep_tc_ws_bytes(m->ld, m->a, prec) : 0));
}

// Allocates what contexts 0..count-1 lack, or nothing.
bta_status try_workspaces(inla_model* m, int count, int prec) {
  const int legs = m->reverse_blocks(prec) > 0 ? 4 : 2;
  const int group = kFormGroup[m->small[prec]];
  const size_t tcb = prec ? sweep_tc_ws_bytes(m->ld, m->a, prec, group) : 0;
  const size_t wsb = 2 * SweepWs::bytes(m->ld, m->a) / sizeof(double);
  const size_t mark = m->allocs.size();
  struct Got {   // one buffer each for the reverse legs and the areas
    double* legs = nullptr;
    uint8_t* tc = nullptr;
  };
  std::vector<Got> got(count);
  // (where the emulated mode has its areas, the mixed mode's products fit into them)
  auto shared = [&](const EvalCtx& c) {
    return prec == 1 && c.tc[2][0] && tcb <= sweep_tc_ws_bytes(m->ld, m->a, 2, c.group[2]);
  };
  bta_status st = BTA_OK;
  for (int e = 0; e < count && st == BTA_OK; ++e) {
    const EvalCtx& c = m->ctx[e];
    if (legs == 4 && !c.legs[2].W1) st = dmalloc(m, &got[e].legs, wsb);
    if (st == BTA_OK && !c.tc[prec][0] && !shared(c)) st = dmalloc(m, &got[e].tc, legs * tcb);
  }
  if (st != BTA_OK) {
    roll_back(m, mark);
    return st;
  }
  for (int e = 0; e < count; ++e) {
    EvalCtx& c = m->ctx[e];
    if (got[e].legs) leg_carve(m, c, 2, got[e].legs);
    if (c.tc[prec][0]) continue;
    for (int q = 0; q < legs; ++q)
      c.tc[prec][q] = got[e].tc ? got[e].tc + q * tcb : prec ? c.tc[2][q] : nullptr;
    c.group[prec] = group;
  }
  return BTA_OK;
}

bta_status ensure_workspaces(inla_model* m, int count, int prec) {
  const int form = m->small[prec];
  bta_status st = try_workspaces(m, count, prec);
  while (st == BTA_ERR_NOMEM && prec != 1 && m->small[prec] + 1 < kWorkForms) {
    ++m->small[prec];
    st = try_workspaces(m, count, prec);
  }
  if (st != BTA_OK) m->small[prec] = form;   // (fewer thetas go on in the larger form)
  return st;
}

// The workspace of a context's leg in a precision.
SweepWs leg_ws(const EvalCtx& c, int q, int prec) {
  SweepWs ws = c.legs[q];
  if (prec) {
    ws.tc = c.tc[prec][q];
    ws.tcgroup = c.group[prec];
  }
  return ws;
}

// The evaluation of contexts 0..cnt-1 as a list of issue steps.
//   mode 0: f only; 1: f and gradient; 2: reverse pass of a preceding mode-0
//   evaluation (the factors are still in place).
//   nb: blocks of the reverse legs (reverse_blocks; mode 2: those of the factors held).
// The conditional matrices Q_c of all contexts form one set and the priors
// Q_p another; each set is swept with one batched launch per block step.  Each set
// is eliminated from both ends towards the middle block (SweepItem: a forward and a
// reverse leg with workspaces of their own), so that a value takes half as many dependent
// diagonal factors, and the four legs run on four streams: a chain of small kernels
// leaves most of the GPU idle, and the serial diagonal steps of one leg overlap the wide
// products of the others.  Per call, one leg per matrix / two: b = 1024, 50 blocks emulated
// gradient 75.8 / 58.6 ms, value 55.2 / 38.7 ms; b = 4800, 8 blocks 215 / 205 ms; b = 64,
// 4 blocks FP64 0.92 / 0.72 ms; the FP64-bound b = 1024 gradient 68.6 / 67.4 ms.  Mixed
// precision keeps one forward leg per matrix: its products round to ~22 bits, so another
// order would move a gradient by its own error (3e-9 where the results agree to 1e-12).
// Each step issues one block of every leg, so the streams' operations, and the nodes of
// a captured graph, are created in alternation: the driver submits a graph's kernels in
// creation order into a bounded queue, and a whole sweep created first (~1600 launches a
// block) held the others back until the GPU had drained most of it.
using IssueStep = std::function<bta_status()>;

struct GroupSets {
  std::vector<SweepItem> ic, ip;   // forward legs
  std::vector<SweepItem> jc, jp;   // reverse legs (empty below three blocks)
};

bta_status group_program(inla_model* m, int mode, int cnt, int prec, int nb, cudaStream_t s0,
                         std::vector<IssueStep>& steps) {
  const ModelDev& md = m->md;
  const int grad = mode >= 1, nt = md.nt, mid = nt - 1 - nb;
  auto sets = std::make_shared<GroupSets>();
  for (int e = 0; e < cnt; ++e) {
    EvalCtx& c = m->ctx[e];
    SweepItem ic, ip;
    ic.q = c.qc; ic.vec = c.x; ic.slots = c.slots_c; ic.fail = c.fail;
    ic.ws = leg_ws(c, 0, prec); ic.fuse = &c.fc;
    ip.q = c.qp; ip.vec = nullptr; ip.slots = c.slots_p; ip.fail = c.fail + 1;
    ip.ws = leg_ws(c, 1, prec); ip.fuse = &c.fp;
    ic.md = ip.md = &md;
    ic.lay = ip.lay = &m->L;
    ic.coef = ip.coef = c.coefbuf;
    if (nb > 0) {
      SweepItem jc = ic, jp = ip;
      ic.len = ip.len = mid + 1;
      jc.rev = jp.rev = 1;
      jc.len = jp.len = nb + 1;
      jc.ws = leg_ws(c, 2, prec);
      jp.ws = leg_ws(c, 3, prec);
      if (md.a > 0) {
        jc.tip = c.tip2;
        ic.tip2 = c.tip2;
        ic.vT2 = jc.ws.vT;
      }
      sets->jc.push_back(jc);
      sets->jp.push_back(jp);
    }
    sets->ic.push_back(ic);
    sets->ip.push_back(ip);
  }
  // set-up on s0, the fork, and (mode < 2) the assembly of both sets
  steps.push_back([=]() -> bta_status {
    if (mode < 2) {
      for (int e = 0; e < cnt; ++e) {
        EvalCtx& c = m->ctx[e];
        BTA_TRY(launch_coef(md, m->L, c.coefbuf, s0));
        BTA_CUDA_TRY(cudaMemsetAsync(c.fail, 0xff, 2 * sizeof(int32_t), s0));
        BTA_CUDA_TRY(cudaMemsetAsync(c.fail + 2, 0, sizeof(int32_t), s0));
      }
    }
    BTA_CUDA_TRY(cudaEventRecord(m->ev0, s0));
    BTA_CUDA_TRY(cudaStreamWaitEvent(m->s1, m->ev0, 0));
    BTA_CUDA_TRY(cudaStreamWaitEvent(m->s2, m->ev0, 0));
    if (mode < 2)
      for (int e = 0; e < cnt; ++e) {
        BTA_TRY(launch_assemble(md, m->L, m->ctx[e].coefbuf, 1, m->ctx[e].qc, m->ctx[e].x,
                                m->s1));
        BTA_TRY(launch_assemble(md, m->L, m->ctx[e].coefbuf, 0, m->ctx[e].qp, nullptr, m->s2));
      }
    if (nb > 0) {
      BTA_CUDA_TRY(cudaEventRecord(m->evac, m->s1));
      BTA_CUDA_TRY(cudaEventRecord(m->evap, m->s2));
      BTA_CUDA_TRY(cudaStreamWaitEvent(m->s3, m->evac, 0));
      BTA_CUDA_TRY(cudaStreamWaitEvent(m->s4, m->evap, 0));
    }
    return BTA_OK;
  });
  // Q_c's vector parts, and its arrow where no b x b product carries it, on streams of their
  // own: they only read finished blocks of the factor, and on s1 and s3 they lay between the
  // dependent diagonal factors and before the selected inversion, which now follows the solve
  // block by block.  Low-memory sweeps recompute L_B in workspaces that the next block needs.
  // In line / on their own streams: b = 1024, 50 blocks emulated gradient 46.4 / 44.9 ms, value
  // 29.0 / 28.3; b = 64, 4 blocks 0.52 / 0.48 ms, with the arrow 0.45; mixed 75.2 / 73.5 ms by
  // the arrow.
  const bool side = !m->lowmem;
  const cudaStream_t v1 = side ? m->s5 : m->s1, v3 = side ? m->s6 : m->s3;
  if (mode < 2)
    for (int i = 0; i <= mid; ++i)
      steps.push_back([=]() -> bta_status {
        if (nb > 0 && i == mid) {   // the reverse legs have updated the shared block
          BTA_CUDA_TRY(cudaStreamWaitEvent(m->s1, m->evjc, 0));
          BTA_CUDA_TRY(cudaStreamWaitEvent(m->s2, m->evjp, 0));
          if (side) BTA_CUDA_TRY(cudaStreamWaitEvent(v1, m->evjv, 0));
        }
        BTA_TRY(factor_sweep_multi(sets->ic.data(), cnt, m->s1, prec, i, i + 1, v1, m->evv5));
        BTA_TRY(factor_sweep_multi(sets->ip.data(), cnt, m->s2, prec, i, i + 1));
        if (i >= nb) return BTA_OK;
        BTA_TRY(factor_sweep_multi(sets->jc.data(), cnt, m->s3, prec, i, i + 1, v3, m->evv6));
        BTA_TRY(factor_sweep_multi(sets->jp.data(), cnt, m->s4, prec, i, i + 1));
        if (i == nb - 1) {
          BTA_CUDA_TRY(cudaEventRecord(m->evjc, m->s3));
          BTA_CUDA_TRY(cudaEventRecord(m->evjp, m->s4));
          if (side) BTA_CUDA_TRY(cudaEventRecord(m->evjv, v3));
        }
        return BTA_OK;
      });
  // step t of the upper solve, from the shared block outwards, both legs at once
  auto upper_step = [=](const SweepItem* it, const SweepItem* jt, int count, int t,
                        cudaStream_t a, cudaStream_t b) -> bta_status {
    BTA_TRY(upper_solve_multi(it, count, a, mid - t, mid - t));
    if (nb == 0) return BTA_OK;
    if (t == 0) {
      BTA_CUDA_TRY(cudaEventRecord(m->evmv, a));
      BTA_CUDA_TRY(cudaStreamWaitEvent(b, m->evmv, 0));
    } else if (t <= nb) {
      BTA_TRY(upper_solve_multi(jt, count, b, nb - t, nb - t));
    }
    if (t == mid) {   // a has x
      BTA_CUDA_TRY(cudaEventRecord(m->evs6, b));
      BTA_CUDA_TRY(cudaStreamWaitEvent(a, m->evs6, 0));
    }
    return BTA_OK;
  };
  auto upper = [=](const SweepItem* it, const SweepItem* jt, int count) -> bta_status {
    for (int t = 0; t <= mid; ++t)
      BTA_TRY(upper_step(it, jt, count, t, m->s1, m->s3));
    return BTA_OK;
  };
  // the sums over x, on s5 behind the stream that has it
  auto x_sums = [=](cudaStream_t a) -> bta_status {
    BTA_CUDA_TRY(cudaEventRecord(m->evx, a));
    BTA_CUDA_TRY(cudaStreamWaitEvent(m->s5, m->evx, 0));
    for (int e = 0; e < cnt; ++e) {
      EvalCtx& c = m->ctx[e];
      BTA_TRY(launch_residual(md, c.x, c.RS, m->s5));
      BTA_TRY(launch_pattern_quad_all(md, c.x, c.QD, c.QB, m->s5));
    }
    BTA_CUDA_TRY(cudaEventRecord(m->ev5, m->s5));
    return BTA_OK;
  };
  // the solve rides along with the selected inversion, unless that would overwrite a factor
  // which the refinement of x reads again
  const bool along = side && prec != 1 && mode == 1;
  if (mode < 2)
    steps.push_back([=]() -> bta_status {
      if (side && prec != 1) {   // behind the tip
        BTA_CUDA_TRY(cudaEventRecord(m->evv5, m->s1));
        BTA_CUDA_TRY(cudaStreamWaitEvent(v1, m->evv5, 0));
        if (along) return BTA_OK;
        for (int t = 0; t <= mid; ++t)
          BTA_TRY(upper_step(sets->ic.data(), sets->jc.data(), cnt, t, v1, v3));
        return x_sums(v1);
      }
      BTA_TRY(upper(sets->ic.data(), sets->jc.data(), cnt));
      if (prec == 1) {
        // one step of iterative refinement in FP64: x += Q_c^{-1} (r - Q_c x)
        for (int e = 0; e < cnt; ++e) {
          EvalCtx& c = m->ctx[e];
          BTA_TRY(launch_rhs(md, m->L, c.coefbuf, c.dr, m->s1));
          BTA_TRY(launch_qc_residual(md, m->L, c.coefbuf, c.x, c.dr, m->s1));
          SweepItem dx = sets->ic[e];   // (the mixed mode has no reverse legs)
          dx.vec = c.dr;
          BTA_TRY(lower_solve(dx, m->s1));
          BTA_TRY(upper_solve_multi(&dx, 1, m->s1));
          BTA_TRY(launch_axpy((int64_t)md.nt * md.ld + md.a, 1.0, c.dr, c.x, m->s1));
        }
      }
      return x_sums(m->s1);
    });
  if (grad)
    for (int t = 0; t <= mid; ++t)
      steps.push_back([=]() -> bta_status {
        const int i = mid - t, r = nb - t;   // the reverse legs follow the shared block
        if (along) {
          BTA_TRY(upper_step(sets->ic.data(), sets->jc.data(), cnt, t, v1, v3));
          BTA_CUDA_TRY(cudaEventRecord(m->evs5, v1));
          BTA_CUDA_TRY(cudaStreamWaitEvent(m->s1, m->evs5, 0));
          if (t == mid) BTA_TRY(x_sums(v1));
        }
        BTA_TRY(selinv_sweep_multi(sets->ic.data(), cnt, m->s1, prec, i, i));
        BTA_TRY(selinv_sweep_multi(sets->ip.data(), cnt, m->s2, prec, i, i));
        if (nb == 0) return BTA_OK;
        if (t == 0) {
          BTA_CUDA_TRY(cudaEventRecord(m->evmc, m->s1));
          BTA_CUDA_TRY(cudaEventRecord(m->evmp, m->s2));
          BTA_CUDA_TRY(cudaStreamWaitEvent(m->s3, m->evmc, 0));
          BTA_CUDA_TRY(cudaStreamWaitEvent(m->s4, m->evmp, 0));
        } else if (r >= 0) {
          if (along) {
            BTA_CUDA_TRY(cudaEventRecord(m->evs6, v3));
            BTA_CUDA_TRY(cudaStreamWaitEvent(m->s3, m->evs6, 0));
          }
          BTA_TRY(selinv_sweep_multi(sets->jc.data(), cnt, m->s3, prec, r, r));
          BTA_TRY(selinv_sweep_multi(sets->jp.data(), cnt, m->s4, prec, r, r));
        }
        return BTA_OK;
      });
  // join and combine
  steps.push_back([=]() -> bta_status {
    if (nb > 0) {
      BTA_CUDA_TRY(cudaEventRecord(m->ev3, m->s3));
      BTA_CUDA_TRY(cudaEventRecord(m->ev4, m->s4));
      BTA_CUDA_TRY(cudaStreamWaitEvent(m->s1, m->ev3, 0));
      BTA_CUDA_TRY(cudaStreamWaitEvent(m->s2, m->ev4, 0));
    }
    if (grad) {
      BTA_TRY(selinv_sums(sets->ic.data(), cnt, m->s1));
      BTA_TRY(selinv_sums(sets->ip.data(), cnt, m->s2));
    }
    if (mode < 2) BTA_CUDA_TRY(cudaStreamWaitEvent(m->s1, m->ev5, 0));
    BTA_CUDA_TRY(cudaEventRecord(m->ev1, m->s1));
    BTA_CUDA_TRY(cudaEventRecord(m->ev2, m->s2));
    BTA_CUDA_TRY(cudaStreamWaitEvent(s0, m->ev1, 0));
    BTA_CUDA_TRY(cudaStreamWaitEvent(s0, m->ev2, 0));
    for (int e = 0; e < cnt; ++e) {
      EvalCtx& c = m->ctx[e];
      Reductions r{};
      r.PDc = c.PDc; r.PBc = c.PBc; r.PCc = c.PCc; r.ZTc = c.qc.T;
      r.PDp = c.PDp; r.PBp = c.PBp; r.QD = c.QD; r.QB = c.QB; r.RS = c.RS;
      r.ldc = c.slots_c; r.nldc = m->nslots; r.ldp = c.slots_p; r.nldp = m->nslots;
      r.failc = c.fail; r.failp = c.fail + 1; r.x = c.x; r.red = c.red; r.grad = grad;
      BTA_TRY(launch_finalize(md, m->L, c.coefbuf, r, c.out, s0));
    }
    return BTA_OK;
  });
  return BTA_OK;
}

// Record (issue, or capture) the evaluation of contexts 0..cnt-1.
bta_status record_group(inla_model* m, int mode, int cnt, int prec, int nb, cudaStream_t s0) {
  std::vector<IssueStep> steps;
  BTA_TRY(group_program(m, mode, cnt, prec, nb, s0, steps));
  for (auto& st : steps) BTA_TRY(st());
  return BTA_OK;
}

// Status of one evaluation from its two failure words (parts[6], parts[7]:
// -1, a failing block, or BTA_ERR_TIMEOUT from the task-graph factor) and the
// tensor-core status word: a timeout outranks a non-positive pivot.
bta_status eval_status(const double* parts, int32_t tcs) {
  const double fc = parts[6], fp = parts[7];
  if (tcs == BTA_ERR_TIMEOUT || fc == BTA_ERR_TIMEOUT || fp == BTA_ERR_TIMEOUT)
    return BTA_ERR_TIMEOUT;
  if (fc >= 0 || fp >= 0) return BTA_ERR_NOT_SPD;
  return BTA_OK;
}

bta_status worse(bta_status a, bta_status b) {
  if (a == BTA_ERR_TIMEOUT || b == BTA_ERR_TIMEOUT) return BTA_ERR_TIMEOUT;
  return a != BTA_OK ? a : b;
}

// Run one group (thetas for contexts 0..cnt-1 already in htheta for mode < 2);
// outputs land in hout[e * out_size(d)].
bta_status run_group(inla_model* m, int mode, int cnt, int prec, int use_graph,
                     cudaStream_t stream) {
  const int d = m->d, no = out_size(d);
  const int nb = mode < 2 ? m->reverse_blocks(prec) : m->ctx[0].reverse;
  if (mode < 2)
    for (int e = 0; e < cnt; ++e)
      BTA_CUDA_TRY(cudaMemcpyAsync(m->ctx[e].coefbuf + m->L.theta, m->htheta + (size_t)e * d,
                                   d * sizeof(double), cudaMemcpyHostToDevice, stream));
  if (use_graph) {
    GraphKey* gk = nullptr;
    for (auto& g : m->graphs)
      if (g.mode == mode && g.count == cnt && g.precision == prec && g.reverse == nb) gk = &g;
    if (!gk) {
      if (mode < 2) {
        // one eager evaluation first: it times the tile shapes of the
        // products the graph will hold, which then replays those choices
        TuneScope tune;
        BTA_TRY(record_group(m, mode, cnt, prec, nb, stream));
        BTA_CUDA_TRY(cudaStreamSynchronize(stream));
      }
      const int64_t before = g_launches;
      cudaStream_t cap;
      BTA_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
      BTA_CUDA_TRY(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal));
      bta_status st = record_group(m, mode, cnt, prec, nb, cap);
      cudaGraph_t graph = nullptr;
      cudaError_t e = cudaStreamEndCapture(cap, &graph);
      if (st != BTA_OK) {
        if (graph) cudaGraphDestroy(graph);
        cudaStreamDestroy(cap);
        return st;
      }
      BTA_CUDA_TRY(e);
      cudaGraphExec_t exec = nullptr;
      e = cudaGraphInstantiate(&exec, graph, 0);
      cudaGraphDestroy(graph);
      cudaStreamDestroy(cap);
      BTA_CUDA_TRY(e);
      m->graphs.push_back({mode, cnt, prec, nb, exec, g_launches - before});
      gk = &m->graphs.back();
    }
    BTA_CUDA_TRY(cudaGraphLaunch(gk->exec, stream));
    m->launched += gk->kernels;
  } else {
    const int64_t before = g_launches;
    BTA_TRY(record_group(m, mode, cnt, prec, nb, stream));
    m->launched += g_launches - before;
  }
  for (int e = 0; e < cnt; ++e)
    BTA_CUDA_TRY(cudaMemcpyAsync(m->hout + (size_t)e * no, m->ctx[e].out, no * sizeof(double),
                                 cudaMemcpyDeviceToHost, stream));
  BTA_CUDA_TRY(cudaStreamSynchronize(stream));
  bta_status st = BTA_OK;
  for (int e = 0; e < cnt; ++e) {
    int32_t tcs = 0;   // the tensor-core kernels' status word
    BTA_CUDA_TRY(cudaMemcpy(&tcs, m->ctx[e].fail + 2, sizeof(int32_t), cudaMemcpyDeviceToHost));
    const double* parts = m->hout + (size_t)e * no + 1 + d;
    st = worse(st, eval_status(parts, tcs));
    m->ctx[e].have_factors = mode == 0 ? 1 + prec : 0;   // remembers the factor's precision
    m->ctx[e].reverse = nb;
  }
  m->last.assign(m->hout + (size_t)(cnt - 1) * no, m->hout + (size_t)cnt * no);
  return st;
}

}  // namespace

extern "C" {

const char* bta_status_string(bta_status s) {
  switch (s) {
    case BTA_OK: return "ok";
    case BTA_ERR_ARG: return "invalid argument";
    case BTA_ERR_NOT_SPD: return "matrix not positive definite";
    case BTA_ERR_CUDA: return "CUDA error";
    case BTA_ERR_NOMEM: return "out of device memory";
    case BTA_ERR_TIMEOUT: return "bounded device wait timed out";
    case BTA_ERR_STATE: return "descriptor in the wrong state";
  }
  return "unknown status";
}

void inla_model_destroy(inla_model* m) {
  if (!m) return;
  cudaDeviceSynchronize();
  for (auto& g : m->graphs)
    if (g.exec) cudaGraphExecDestroy(g.exec);
  for (void* p : m->allocs) cudaFree(p);
  if (m->hout) cudaFreeHost(m->hout);
  if (m->htheta) cudaFreeHost(m->htheta);
  if (m->s1) cudaStreamDestroy(m->s1);
  if (m->s2) cudaStreamDestroy(m->s2);
  if (m->s3) cudaStreamDestroy(m->s3);
  if (m->s4) cudaStreamDestroy(m->s4);
  if (m->s5) cudaStreamDestroy(m->s5);
  if (m->s6) cudaStreamDestroy(m->s6);
  if (m->s0) cudaStreamDestroy(m->s0);
  for (cudaEvent_t e : {m->ev0, m->evx, m->ev1, m->ev2, m->evac, m->evap, m->evjc, m->evjp,
                        m->evmc, m->evmp, m->ev3, m->ev4, m->evj, m->evv5, m->evv6, m->evjv,
                        m->evmv, m->evs5, m->evs6, m->ev5})
    if (e) cudaEventDestroy(e);
  delete m;
}

static bta_status model_create_impl(const inla_model_spec* sp, inla_model* m) {
  ModelDev& md = m->md;
  m->lowmem = sp->low_memory != 0;
  const int k = sp->k, ns = sp->ns, nt = sp->nt, a = sp->a;
  if (k < 1 || k > kMaxK || ns < 1 || nt < 1 || a < 0 || a % k || a > 32 || sp->nnz < 1 ||
      !sp->row_ptr || !sp->col || !sp->val_C || !sp->val_G || !sp->val_GG || !sp->m_diag ||
      (nt > 1 && !sp->m_sub) || sp->n_obs < 0 || (sp->n_obs > 0 && (!sp->obs_t || !sp->obs_s ||
      !sp->obs_v || !sp->y || (a > 0 && !sp->obs_cov))))
    return BTA_ERR_ARG;
  md.k = k; md.ns = ns; md.nt = nt; md.a = a; md.a_r = a / k; md.b = k * ns;
  md.ld = pad_ld(md.b); md.d = 4 * k + k * (k - 1) / 2; md.nnz = sp->nnz; md.n_obs = sp->n_obs;
  md.tip_prior = sp->tip_prior > 0 ? sp->tip_prior : 1e-3;
  md.theta_prior_var = sp->theta_prior_var > 0 ? sp->theta_prior_var : 100.0;
  if (md.d > kMaxD) return BTA_ERR_ARG;
  const int ld = md.ld, b = md.b, a_r = md.a_r;
  m->n = nt; m->b = b; m->ld = ld; m->a = a; m->d = md.d;
  // --- spatial pattern
  if (sp->row_ptr[0] != 0 || sp->row_ptr[ns] != sp->nnz) return BTA_ERR_ARG;
  std::vector<int32_t> row_of(sp->nnz);
  for (int s = 0; s < ns; ++s) {
    bool diag = false;
    for (int e = sp->row_ptr[s]; e < sp->row_ptr[s + 1]; ++e) {
      if (sp->col[e] < 0 || sp->col[e] >= ns) return BTA_ERR_ARG;
      row_of[e] = s;
      diag |= sp->col[e] == s;
    }
    if (!diag) return BTA_ERR_ARG;   // the pattern must hold the diagonal
  }
  std::vector<double> val(3 * (size_t)sp->nnz);
  std::memcpy(val.data(), sp->val_C, sp->nnz * sizeof(double));
  std::memcpy(val.data() + sp->nnz, sp->val_G, sp->nnz * sizeof(double));
  std::memcpy(val.data() + 2 * (size_t)sp->nnz, sp->val_GG, sp->nnz * sizeof(double));
  BTA_TRY(upload(m, &md.row_ptr, sp->row_ptr, ns + 1));
  BTA_TRY(upload(m, &md.col, sp->col, sp->nnz));
  BTA_TRY(upload(m, &md.row_of, row_of.data(), sp->nnz));
  BTA_TRY(upload(m, &md.val, val.data(), val.size()));
  md.m_diag_h.assign(sp->m_diag, sp->m_diag + 3 * nt);
  md.m_sub_h.assign(std::max(3 * (nt - 1), 1), 0.0);
  if (nt > 1) std::memcpy(md.m_sub_h.data(), sp->m_sub, 3 * (nt - 1) * sizeof(double));
  BTA_TRY(upload(m, &md.m_diag, md.m_diag_h.data(), md.m_diag_h.size()));
  BTA_TRY(upload(m, &md.m_sub, md.m_sub_h.data(), md.m_sub_h.size()));
  // --- observation-derived, theta-independent pieces (fixed accumulation order)
  std::vector<double> cnt((size_t)nt * ld, 0.0), craw((size_t)nt * a * ld, 0.0),
      traw((size_t)k * a * a, 0.0), rraw((size_t)nt * ld + a, 0.0);
  std::vector<int32_t> lat(std::max<int64_t>(sp->n_obs, 1));
  md.n_per_var.assign(k, 0.0);
  for (int64_t j = 0; j < sp->n_obs; ++j) {
    int t = sp->obs_t[j], s = sp->obs_s[j], v = sp->obs_v[j];
    if (t < 0 || t >= nt || s < 0 || s >= ns || v < 0 || v >= k) return BTA_ERR_ARG;
    int c = v * ns + s;
    int64_t li = (int64_t)t * ld + c;
    lat[j] = (int32_t)li;
    cnt[li] += 1.0;
    rraw[li] += sp->y[j];
    md.n_per_var[v] += 1.0;
    const double* cv = sp->obs_cov + j * a_r;
    for (int i = 0; i < a_r; ++i) {
      int f = v * a_r + i;
      craw[(size_t)t * a * ld + f + (size_t)c * a] += cv[i];
      rraw[(size_t)nt * ld + f] += cv[i] * sp->y[j];
      for (int i2 = 0; i2 < a_r; ++i2)
        traw[(size_t)v * a * a + f + (size_t)(v * a_r + i2) * a] += cv[i] * cv[i2];
    }
  }
  // with no fixed effects (a = 0) the arrow arrays are empty: keep one zero
  // element so that every device array exists
  if (craw.empty()) craw.assign(1, 0.0);
  if (traw.empty()) traw.assign(1, 0.0);
  BTA_TRY(upload(m, &md.cnt, cnt.data(), cnt.size()));
  BTA_TRY(upload(m, &md.craw, craw.data(), craw.size()));
  BTA_TRY(upload(m, &md.traw, traw.data(), traw.size()));
  BTA_TRY(upload(m, &md.rraw, rraw.data(), rraw.size()));
  BTA_TRY(upload(m, &md.obs_lat, lat.data(), lat.size()));
  BTA_TRY(upload(m, &md.obs_v, sp->n_obs ? sp->obs_v : lat.data(), lat.size()));
  std::vector<double> covv((size_t)std::max<int64_t>(sp->n_obs, 1) * std::max(a_r, 1), 0.0),
      yv(std::max<int64_t>(sp->n_obs, 1), 0.0);
  if (sp->n_obs) {
    if (a_r) std::memcpy(covv.data(), sp->obs_cov, sp->n_obs * a_r * sizeof(double));
    std::memcpy(yv.data(), sp->y, sp->n_obs * sizeof(double));
  }
  BTA_TRY(upload(m, &md.obs_cov, covv.data(), covv.size()));
  BTA_TRY(upload(m, &md.y, yv.data(), yv.size()));
  // --- evaluation buffers: one context up front, more on demand
  m->L.init(k, md.d, nt);
  m->nslots = logdet_slots(nt, ld);
  const char* env = std::getenv("BTA_SMALL_WORKSPACES");
  const int form = env ? std::min(std::max(std::atoi(env), 0), kWorkForms - 1) : 0;
  for (int prec : {0, 2})   // (the mixed mode has one form)
    m->small[prec] = std::max(form, m->lowmem && work_bytes(m, prec) > kLowMemoryWork ? 1 : 0);
  BTA_TRY(ensure_ctx(m, 1));
  BTA_CUDA_TRY(cudaMallocHost(&m->hout, (size_t)kMaxBatch * out_size(md.d) * sizeof(double)));
  BTA_CUDA_TRY(cudaMallocHost(&m->htheta, (size_t)kMaxBatch * kMaxD * sizeof(double)));
  BTA_CUDA_TRY(cudaStreamCreateWithFlags(&m->s1, cudaStreamNonBlocking));
  BTA_CUDA_TRY(cudaStreamCreateWithFlags(&m->s2, cudaStreamNonBlocking));
  BTA_CUDA_TRY(cudaStreamCreateWithFlags(&m->s3, cudaStreamNonBlocking));
  BTA_CUDA_TRY(cudaStreamCreateWithFlags(&m->s4, cudaStreamNonBlocking));
  BTA_CUDA_TRY(cudaStreamCreateWithFlags(&m->s5, cudaStreamNonBlocking));
  BTA_CUDA_TRY(cudaStreamCreateWithFlags(&m->s6, cudaStreamNonBlocking));
  BTA_CUDA_TRY(cudaStreamCreateWithFlags(&m->s0, cudaStreamNonBlocking));
  for (cudaEvent_t* e : {&m->ev0, &m->evx, &m->ev1, &m->ev2, &m->evac, &m->evap, &m->evjc,
                         &m->evjp, &m->evmc, &m->evmp, &m->ev3, &m->ev4, &m->evj, &m->evv5,
                         &m->evv6, &m->evjv, &m->evmv, &m->evs5, &m->evs6, &m->ev5})
    BTA_CUDA_TRY(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
  BTA_CUDA_TRY(cudaDeviceSynchronize());
  return BTA_OK;
}

bta_status inla_model_create(const inla_model_spec* spec, inla_model** out) {
  if (!spec || !out) return BTA_ERR_ARG;
  *out = nullptr;
  inla_model* m = new (std::nothrow) inla_model();
  if (!m) return BTA_ERR_NOMEM;
  bta_status st = model_create_impl(spec, m);
  if (st != BTA_OK) {
    inla_model_destroy(m);
    return st;
  }
  *out = m;
  return BTA_OK;
}

bta_status inla_model_dims(const inla_model* m, int32_t* d, int32_t* b, int32_t* ld, int32_t* n,
                           int32_t* a) {
  if (!m) return BTA_ERR_ARG;
  if (d) *d = m->d;
  if (b) *b = m->b;
  if (ld) *ld = m->ld;
  if (n) *n = m->n;
  if (a) *a = m->a;
  return BTA_OK;
}

static bool desc_ok(const bta_desc* q, int need_arrow) {
  if (!q || q->n < 1 || q->b < 1 || q->ld < q->b || q->ld % kPad || q->a < 0 || q->a > 32 ||
      !q->D || (q->n > 1 && !q->B))
    return false;
  if (q->a > 0 && (!q->C || !q->T)) return false;
  (void)need_arrow;
  return true;
}

bta_status bta_assemble(inla_model* m, const double* theta, int32_t which, bta_desc* out,
                        double* rhs, cudaStream_t stream) {
  if (!m || !theta || !out || (which != 0 && which != 1)) return BTA_ERR_ARG;
  if (!finite_theta(theta, m->d)) return BTA_ERR_ARG;
  if (out->n != m->n || out->b != m->b || out->ld != m->ld ||
      out->a != (which ? m->a : 0) || !desc_ok(out, which))
    return BTA_ERR_ARG;
  double* cb = nullptr;
  BTA_CUDA_TRY(cudaMallocAsync(&cb, m->L.total * sizeof(double), stream));
  BTA_CUDA_TRY(cudaMemcpyAsync(cb + m->L.theta, theta, m->d * sizeof(double),
                               cudaMemcpyHostToDevice, stream));
  bta_status st = launch_coef(m->md, m->L, cb, stream);
  if (st == BTA_OK) st = launch_assemble(m->md, m->L, cb, which, *out, which ? rhs : nullptr,
                                         stream);
  cudaFreeAsync(cb, stream);
  if (st == BTA_OK) out->state = BTA_STATE_ASSEMBLED;
  return st;
}

bta_status bta_factor(bta_desc* q, double* rhs_inout, double* logdet, int32_t* fail_block,
                      int32_t precision, cudaStream_t stream) {
  if (!desc_ok(q, 0) || !logdet || !fail_block || precision < 0 || precision > 2)
    return BTA_ERR_ARG;
  if (q->state != BTA_STATE_ASSEMBLED) return BTA_ERR_STATE;
  const int nsl = logdet_slots(q->n, q->ld);
  const size_t wsb = SweepWs::bytes(q->ld, q->a);
  const int ld = q->ld;
  // tensor-core modes: operand copies of the b x b products, 256-byte aligned; the residue
  // planes of fewer moduli at once where all of them do not fit the device
  const size_t head = (wsb + nsl * sizeof(double) + 255) / 256 * 256;
  uint8_t* buf = nullptr;
  SweepWs ws;
  cudaError_t e = cudaSuccess;
  for (int group : {kOzakiModuli, kOzakiSmallGroup}) {
    const size_t tcb = precision ? sweep_tc_ws_bytes(ld, q->a, precision, group) : 0;
    e = cudaMallocAsync(reinterpret_cast<void**>(&buf), head + tcb, stream);
    ws.tcgroup = group;
    if (e != cudaErrorMemoryAllocation || precision != 2) break;
    if (group != kOzakiSmallGroup) cudaGetLastError();
  }
  BTA_CUDA_TRY(e);
  ws.carve(reinterpret_cast<double*>(buf), ld, q->a);
  double* slots = reinterpret_cast<double*>(buf) + wsb / sizeof(double);
  if (precision) {
    ws.tc = buf + head;
    ws.tcstat = fail_block;   // a tensor-core timeout lands in the failure word
  }
  BTA_CUDA_TRY(cudaMemsetAsync(fail_block, 0xff, sizeof(int32_t), stream));
  bta_status st = factor_sweep(*q, rhs_inout, slots, fail_block, ws, stream, precision);
  if (st == BTA_OK) st = sum_slots(slots, nsl, logdet, 0, stream);
  cudaFreeAsync(buf, stream);
  if (st == BTA_OK) q->state = BTA_STATE_FACTORED;
  return st;
}

bta_status bta_solve(const bta_desc* L, double* z_inout, int32_t lower, int32_t refine,
                     const bta_desc* Q_or_null, cudaStream_t stream) {
  if (!desc_ok(L, 0) || !z_inout || refine < 0 || refine > 1) return BTA_ERR_ARG;
  if (refine) {   // needs r (lower = 1) and the assembled matrix of the same shape
    const bta_desc* Q = Q_or_null;
    if (!lower || !desc_ok(Q, 0) || Q->n != L->n || Q->b != L->b || Q->ld != L->ld ||
        Q->a != L->a || Q->D == L->D)
      return BTA_ERR_ARG;
    if (Q->state != BTA_STATE_ASSEMBLED) return BTA_ERR_STATE;
  }
  if (L->state != BTA_STATE_FACTORED) return BTA_ERR_STATE;
  const size_t wsb = SweepWs::bytes(L->ld, L->a);
  const size_t nv = (size_t)L->n * L->ld + L->a;
  double* buf = nullptr;
  BTA_CUDA_TRY(cudaMallocAsync(&buf, wsb + (refine ? 2 * nv * sizeof(double) : 0), stream));
  SweepWs ws;
  ws.carve(buf, L->ld, L->a);
  double* r = buf + wsb / sizeof(double);   // refinement: r, then the correction
  double* dx = r + nv;
  bta_status st = BTA_OK;
  if (refine)
    st = copy_block(z_inout, (int)nv, r, (int)nv, (int)nv, 1, 1.0, stream);
  SweepItem it, di;
  it.q = *L; it.ws = ws; it.vec = z_inout;
  di = it;
  di.vec = dx;
  if (st == BTA_OK && lower) st = lower_solve(it, stream);
  if (st == BTA_OK) st = upper_solve_multi(&it, 1, stream);
  if (st == BTA_OK && refine) {
    // one step of iterative refinement in FP64 (Eqs. 3-5 on the residual):
    // x += Q^{-1} (r - Q x) with the factor L of Q
    st = copy_block(r, (int)nv, dx, (int)nv, (int)nv, 1, 1.0, stream);
    if (st == BTA_OK) st = bta_residual(*Q_or_null, z_inout, dx, stream);
    if (st == BTA_OK) st = lower_solve(di, stream);
    if (st == BTA_OK) st = upper_solve_multi(&di, 1, stream);
    if (st == BTA_OK) st = launch_axpy((int64_t)nv, 1.0, dx, z_inout, stream);
  }
  cudaFreeAsync(buf, stream);
  return st;
}

bta_status bta_set_wait_limit(int64_t limit_ns, int32_t stall) {
  if (limit_ns < 0 || (limit_ns > 0 && limit_ns < 1000000) || limit_ns > 60000000000ll ||
      (stall != 0 && stall != 1))
    return BTA_ERR_ARG;
  g_dag_wait_ns = limit_ns ? (unsigned long long)limit_ns : 2000000000ull;
  g_dag_stall = stall;
  return BTA_OK;
}

bta_status bta_selinv(bta_desc* L, inla_model* m, const double* theta, int32_t which,
                      double* trace_terms, cudaStream_t stream) {
  if (!desc_ok(L, 0)) return BTA_ERR_ARG;
  if (L->state != BTA_STATE_FACTORED) return BTA_ERR_STATE;
  const bool fused = m && trace_terms;
  if (fused) {
    if (!theta || !finite_theta(theta, m->d) || (which != 0 && which != 1)) return BTA_ERR_ARG;
    if (L->n != m->n || L->ld != m->ld || L->a != (which ? m->a : 0)) return BTA_ERR_ARG;
  }
  size_t wsb = SweepWs::bytes(L->ld, L->a);
  double* buf = nullptr;
  BTA_CUDA_TRY(cudaMallocAsync(&buf, wsb, stream));
  SweepWs ws;
  ws.carve(buf, L->ld, L->a);
  bta_status st = BTA_OK;
  if (!fused) {
    st = selinv_sweep(*L, ws, nullptr, stream);
  } else {
    const ModelDev& md = m->md;
    const size_t pblk = (size_t)md.k * md.k * pattern_chunks(md) * kNP;
    const size_t nPD = md.nt * pblk, nPB = std::max(md.nt - 1, 1) * pblk;
    const size_t nPC = std::max<size_t>((size_t)md.nt * md.k * arrow_chunks(md), 1);
    const size_t nRS = (size_t)kMaxK * resid_chunks(md);
    double* rb = nullptr;
    const size_t nZ0 = std::max(nPD + nPB, (size_t)md.nt * md.ld + md.a);
    size_t total = m->L.total + nPD + nPB + nPC + nZ0 + nRS + kRedDoubles + out_size(md.d) + 4;
    BTA_CUDA_TRY(cudaMallocAsync(&rb, total * sizeof(double), stream));
    double* cb = rb;
    double* PD = cb + m->L.total;
    double* PB = PD + nPD;
    double* PC = PB + nPB;
    double* Z0 = PC + nPC;           // zero reductions for the other matrix / quad forms
    double* RS = Z0 + nZ0;
    double* red = RS + nRS;
    double* o = red + kRedDoubles;
    int32_t* fl = reinterpret_cast<int32_t*>(o + out_size(md.d));
    BTA_CUDA_TRY(cudaMemsetAsync(rb, 0, total * sizeof(double), stream));
    BTA_CUDA_TRY(cudaMemsetAsync(fl, 0xff, 2 * sizeof(int32_t), stream));
    BTA_CUDA_TRY(cudaMemcpyAsync(cb + m->L.theta, theta, md.d * sizeof(double),
                                 cudaMemcpyHostToDevice, stream));
    st = launch_coef(md, m->L, cb, stream);
    SelinvFuse fz;
    fz.md = &md; fz.counts = which; fz.PD = PD; fz.PB = PB; fz.PC = which ? PC : nullptr;
    if (st == BTA_OK) st = selinv_sweep(*L, ws, &fz, stream);
    if (st == BTA_OK) {
      // Reuse the final combination with the other matrix's sums at zero:
      // Phase A = -1/2 tr(Q_c^-1 dQ_c), Phase C = +1/2 tr(Q_p^-1 dQ_p).
      Reductions r{};
      r.PDc = which ? PD : Z0; r.PBc = which ? PB : Z0 + nPD; r.PCc = which ? PC : Z0;
      r.ZTc = which ? L->T : Z0;
      r.PDp = which ? Z0 : PD; r.PBp = which ? Z0 + nPD : PB;
      r.QD = Z0; r.QB = Z0 + nPD; r.RS = RS;
      r.ldc = Z0; r.nldc = 1; r.ldp = Z0; r.nldp = 1; r.failc = fl; r.failp = fl + 1;
      r.x = Z0; r.red = red; r.grad = 1;
      ModelDev mz = md;
      mz.a = which ? md.a : 0;
      st = launch_finalize(mz, m->L, cb, r, o, stream);
      if (st == BTA_OK) {
        // phases at o + 1 + d + kOutParts: A (d), B (d), C (d)
        const double* ph = o + 1 + md.d + kOutParts;
        st = copy_block(which ? ph : ph + 2 * md.d, md.d, trace_terms, md.d, md.d, 1,
                        which ? -2.0 : 2.0, stream);
      }
    }
    cudaFreeAsync(rb, stream);
  }
  cudaFreeAsync(buf, stream);
  if (st == BTA_OK) L->state = BTA_STATE_SELINV;
  return st;
}

bta_status inla_value_and_grad(inla_model* m, const double* theta, int32_t batch, double* f,
                               double* grad, const inla_opts* opts, cudaStream_t stream) {
  if (!m || !theta || !f || batch < 1) return BTA_ERR_ARG;
  const int prec = opts ? opts->precision : 0;
  if (prec < 0 || prec > 2) return BTA_ERR_ARG;
  if (prec == 1 && m->lowmem) return BTA_ERR_ARG;   // its refinement solves read the B blocks
  for (int i = 0; i < batch; ++i)
    if (!finite_theta(theta + (size_t)i * m->d, m->d)) return BTA_ERR_ARG;
  const int use_graph = opts ? opts->use_graph : 1;
  int group = opts && opts->streams > 1 ? opts->streams : 1;
  group = std::min(group, std::min<int>(batch, kMaxBatch / 2));
  BTA_TRY(ensure_ctx(m, group));
  BTA_TRY(ensure_workspaces(m, group, prec));
  const int mode = grad ? 1 : 0;
  const int d = m->d, no = out_size(d);
  bta_status st = BTA_OK;
  for (int i0 = 0; i0 < batch; i0 += group) {
    const int cnt = std::min(group, batch - i0);
    std::memcpy(m->htheta, theta + (size_t)i0 * d, (size_t)cnt * d * sizeof(double));
    bta_status s1 = run_group(m, mode, cnt, prec, use_graph, stream);
    if (s1 != BTA_OK && s1 != BTA_ERR_NOT_SPD && s1 != BTA_ERR_TIMEOUT) return s1;
    st = worse(st, s1);
    for (int e = 0; e < cnt; ++e) {
      const double* o = m->hout + (size_t)e * no;
      f[i0 + e] = o[0];
      if (grad)
        for (int j = 0; j < d; ++j) grad[(size_t)(i0 + e) * d + j] = o[1 + j];
    }
  }
  return st;
}

bta_status inla_backward(inla_model* m, double* grad, int32_t use_graph, cudaStream_t stream) {
  if (!m || !grad) return BTA_ERR_ARG;
  if (m->ctx.empty() || !m->ctx[0].have_factors) return BTA_ERR_STATE;
  for (size_t e = 1; e < m->ctx.size(); ++e) m->ctx[e].have_factors = 0;
  bta_status st = run_group(m, 2, 1, m->ctx[0].have_factors - 1, use_graph, stream);
  for (int j = 0; j < m->d; ++j) grad[j] = m->last[1 + j];
  return st;
}

bta_status bta_gemm(int32_t M, int32_t N, int32_t K, double alpha, const double* A, int32_t lda,
                    int32_t transA, const double* B, int32_t ldb, int32_t transB, double beta,
                    double* Cm, int32_t ldc, cudaStream_t stream) {
  if (M < 0 || N < 0 || K < 0 || !A || !B || !Cm) return BTA_ERR_ARG;
  Gemm g;
  g.M = M; g.N = N; g.K = K; g.alpha = alpha; g.beta = beta;
  g.A = A; g.lda = lda; g.transA = transA ? 1 : 0;
  g.B = B; g.ldb = ldb; g.transB = transB ? 1 : 0;
  g.C = Cm; g.ldc = ldc; g.Cin = Cm; g.ldcin = ldc;
  return gemm_f64(g, stream);
}

bta_status bta_gemm_mixed(int32_t M, int32_t N, int32_t K, double alpha, const double* A,
                          int32_t lda, int32_t transA, const double* B, int32_t ldb,
                          int32_t transB, double beta, double* Cm, int32_t ldc, int32_t* status,
                          cudaStream_t stream) {
  if (M < 0 || N < 0 || K < 1 || !A || !B || !Cm) return BTA_ERR_ARG;
  Gemm g;
  g.M = M; g.N = N; g.K = K; g.alpha = alpha; g.beta = beta;
  g.A = A; g.lda = lda; g.transA = transA ? 1 : 0;
  g.B = B; g.ldb = ldb; g.transB = transB ? 1 : 0;
  g.C = Cm; g.ldc = ldc; g.Cin = Cm; g.ldcin = ldc;
  void* ws = nullptr;
  BTA_CUDA_TRY(cudaMallocAsync(&ws, tc_gemm_ws_bytes(M, N, K), stream));
  bta_status st = tc_gemm_mixed(g, ws, status, stream);
  cudaFreeAsync(ws, stream);
  return st;
}

// An emulated product in panels of the result, whose workspaces (84 bytes an entry, with
// the operands' planes) then stay below 13 GiB: a result of 90000 columns as a whole would
// take 227 GB for its residues.  Panels of 16384 rows and columns cost one more split of the
// operands each, under 1 % of their products; where not even those fit the device, smaller
// ones, at last with the planes of four moduli at once.  The bits do not depend on it.  A
// result that overlaps an operand is not split: its panels would overwrite what others read.
// kernel_ms (optional): the product kernels' time, which is waited for.
static bta_status emulated_panels(const Gemm& g, int32_t* status, float* kernel_ms,
                                  const cudaEvent_t* marks, cudaStream_t stream) {
  auto span = [](const double* p, int rows, int cols, int ld) {
    return std::make_pair(p, p + (int64_t)(cols - 1) * ld + rows);
  };
  const auto c = span(g.C, g.M, g.N, g.ldc);
  auto clear = [&](std::pair<const double*, const double*> x) {
    return x.second <= c.first || c.second <= x.first;
  };
  const bool split = clear(g.transA ? span(g.A, g.K, g.M, g.lda) : span(g.A, g.M, g.K, g.lda)) &&
                     clear(g.transB ? span(g.B, g.N, g.K, g.ldb) : span(g.B, g.K, g.N, g.ldb));
  struct Form {
    int panel, group;
  };
  void* ws = nullptr;
  Form form{};
  cudaError_t e = cudaErrorMemoryAllocation;
  for (Form f : {Form{16384, kOzakiModuli}, Form{4096, kOzakiModuli},
                 Form{1024, kOzakiSmallGroup}}) {
    if (!split) f.panel = INT_MAX;
    e = cudaMallocAsync(&ws, ozaki_ws_bytes(std::min(g.M, f.panel), std::min(g.N, f.panel), g.K,
                                            f.group), stream);
    form = f;
    if (e != cudaErrorMemoryAllocation) break;
    cudaGetLastError();
  }
  if (e == cudaErrorMemoryAllocation) return BTA_ERR_NOMEM;
  BTA_CUDA_TRY(e);
  bta_status st = BTA_OK;
  if (kernel_ms) *kernel_ms = 0.0f;
  for (int64_t n0 = 0; n0 < g.N && st == BTA_OK; n0 += form.panel)
    for (int64_t m0 = 0; m0 < g.M && st == BTA_OK; m0 += form.panel) {
      Gemm q = g;
      q.M = (int)std::min<int64_t>(form.panel, g.M - m0);
      q.N = (int)std::min<int64_t>(form.panel, g.N - n0);
      q.A += g.transA ? m0 * g.lda : m0;
      q.B += g.transB ? n0 : n0 * g.ldb;
      q.C += m0 + n0 * g.ldc;
      q.Cin = q.C;
      st = ozaki_gemm(q, ws, status, stream, marks, form.group);
      float ms = 0.0f;
      if (st == BTA_OK && kernel_ms) {
        if (cudaEventSynchronize(marks[1]) != cudaSuccess ||
            cudaEventElapsedTime(&ms, marks[0], marks[1]) != cudaSuccess)
          st = BTA_ERR_CUDA;
        *kernel_ms += ms;
      }
    }
  cudaFreeAsync(ws, stream);
  return st;
}

bta_status bta_gemm_emulated(int32_t M, int32_t N, int32_t K, double alpha, const double* A,
                             int32_t lda, int32_t transA, const double* B, int32_t ldb,
                             int32_t transB, double beta, double* Cm, int32_t ldc,
                             int32_t slices, int32_t* status, cudaStream_t stream) {
  if (M < 0 || N < 0 || K < 1 || K > 5120 || !A || !B || !Cm || slices < 6 || slices > 8)
    return BTA_ERR_ARG;
  Gemm g;
  g.M = M; g.N = N; g.K = K; g.alpha = alpha; g.beta = beta;
  g.A = A; g.lda = lda; g.transA = transA ? 1 : 0;
  g.B = B; g.ldb = ldb; g.transB = transB ? 1 : 0;
  g.C = Cm; g.ldc = ldc; g.Cin = Cm; g.ldcin = ldc;
  if (M == 0 || N == 0) return BTA_OK;
  return emulated_panels(g, status, nullptr, nullptr, stream);
}

bta_status bta_gemm_emulated_timed(int32_t M, int32_t N, int32_t K, double alpha,
                                   const double* A, int32_t lda, int32_t transA, const double* B,
                                   int32_t ldb, int32_t transB, double beta, double* Cm,
                                   int32_t ldc, int32_t slices, int32_t* status,
                                   float* kernel_ms, cudaStream_t stream) {
  if (M < 1 || N < 1 || K < 1 || K > 5120 || !A || !B || !Cm || slices < 6 || slices > 8 ||
      !kernel_ms)
    return BTA_ERR_ARG;
  Gemm g;
  g.M = M; g.N = N; g.K = K; g.alpha = alpha; g.beta = beta;
  g.A = A; g.lda = lda; g.transA = transA ? 1 : 0;
  g.B = B; g.ldb = ldb; g.transB = transB ? 1 : 0;
  g.C = Cm; g.ldc = ldc; g.Cin = Cm; g.ldcin = ldc;
  cudaEvent_t marks[2] = {nullptr, nullptr};
  BTA_CUDA_TRY(cudaEventCreate(&marks[0]));
  BTA_CUDA_TRY(cudaEventCreate(&marks[1]));
  const bta_status st = emulated_panels(g, status, kernel_ms, marks, stream);
  cudaEventDestroy(marks[0]);
  cudaEventDestroy(marks[1]);
  return st;
}

bta_status inla_batch_create(inla_model* const* models, int32_t count, inla_batch** out) {
  if (!models || !out || count < 1) return BTA_ERR_ARG;
  *out = nullptr;
  inla_batch* b = new (std::nothrow) inla_batch();
  if (!b) return BTA_ERR_NOMEM;
  for (int i = 0; i < count; ++i) {
    if (!models[i]) { delete b; return BTA_ERR_ARG; }
    for (int j = 0; j < i; ++j)
      if (models[j] == models[i]) { delete b; return BTA_ERR_ARG; }
    b->models.push_back(models[i]);
  }
  if (cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess) {
    delete b;
    return BTA_ERR_CUDA;
  }
  *out = b;
  return BTA_OK;
}

void inla_batch_destroy(inla_batch* b) {
  if (!b) return;
  cudaDeviceSynchronize();
  for (auto& row : b->exec)
    for (auto& e : row)
      if (e) cudaGraphExecDestroy(e);
  if (b->fork) cudaEventDestroy(b->fork);
  delete b;
}

// Record every model's evaluation (theta upload, sweeps, result download)
// as branches forked from s0.  The models' issue steps are taken round-robin
// (step j of every model, then step j + 1), so their operations are created
// interleaved and every model's streams start together.
static bta_status record_batch(inla_batch* b, int grad, int prec, cudaStream_t s0) {
  BTA_CUDA_TRY(cudaEventRecord(b->fork, s0));
  const size_t nm = b->models.size();
  std::vector<std::vector<IssueStep>> progs(nm);
  size_t longest = 0;
  for (size_t k = 0; k < nm; ++k) {
    inla_model* m = b->models[k];
    BTA_CUDA_TRY(cudaStreamWaitEvent(m->s0, b->fork, 0));
    BTA_CUDA_TRY(cudaMemcpyAsync(m->ctx[0].coefbuf + m->L.theta, m->htheta,
                                 m->d * sizeof(double), cudaMemcpyHostToDevice, m->s0));
    BTA_TRY(group_program(m, grad, 1, prec, b->reverse[grad][prec][k], m->s0, progs[k]));
    longest = std::max(longest, progs[k].size());
  }
  for (size_t j = 0; j < longest; ++j)
    for (size_t k = 0; k < nm; ++k)
      if (j < progs[k].size()) BTA_TRY(progs[k][j]());
  for (inla_model* m : b->models) {
    BTA_CUDA_TRY(cudaMemcpyAsync(m->hout, m->ctx[0].out, out_size(m->d) * sizeof(double),
                                 cudaMemcpyDeviceToHost, m->s0));
    BTA_CUDA_TRY(cudaEventRecord(m->evj, m->s0));
    BTA_CUDA_TRY(cudaStreamWaitEvent(s0, m->evj, 0));
  }
  return BTA_OK;
}

bta_status inla_batch_value_and_grad(inla_batch* b, const double* theta, int32_t ldt, double* f,
                                     double* grad, const inla_opts* opts, cudaStream_t stream) {
  if (!b || !theta || !f || ldt < 1) return BTA_ERR_ARG;
  const int prec = opts ? opts->precision : 0;
  if (prec < 0 || prec > 2) return BTA_ERR_ARG;
  const int g = grad ? 1 : 0;
  const int nm = (int)b->models.size();
  for (int i = 0; i < nm; ++i)   // mixed mode's refinement solves read the B blocks
    if (prec == 1 && b->models[i]->lowmem) return BTA_ERR_ARG;
  for (int i = 0; i < nm; ++i) {
    inla_model* m = b->models[i];
    if (m->d > ldt || !finite_theta(theta + (size_t)i * ldt, m->d)) return BTA_ERR_ARG;
    std::memcpy(m->htheta, theta + (size_t)i * ldt, m->d * sizeof(double));
  }
  if (!b->exec[g][prec]) {
    b->reverse[g][prec].clear();
    for (inla_model* m : b->models) {
      BTA_TRY(ensure_workspaces(m, 1, prec));
      b->reverse[g][prec].push_back(m->reverse_blocks(prec));
    }
    {  // an eager run first times the products' tile shapes (see run_group)
      TuneScope tune;
      BTA_TRY(record_batch(b, g, prec, stream));
      BTA_CUDA_TRY(cudaStreamSynchronize(stream));
    }
    const int64_t before = g_launches;
    cudaStream_t cap;
    BTA_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    BTA_CUDA_TRY(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal));
    bta_status st = record_batch(b, g, prec, cap);
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(cap, &graph);
    if (st != BTA_OK) {
      if (graph) cudaGraphDestroy(graph);
      cudaStreamDestroy(cap);
      return st;
    }
    BTA_CUDA_TRY(e);
    e = cudaGraphInstantiate(&b->exec[g][prec], graph, 0);
    cudaGraphDestroy(graph);
    cudaStreamDestroy(cap);
    BTA_CUDA_TRY(e);
    b->kernels[g][prec] = g_launches - before;
  }
  BTA_CUDA_TRY(cudaGraphLaunch(b->exec[g][prec], stream));
  BTA_CUDA_TRY(cudaStreamSynchronize(stream));
  bta_status st = BTA_OK;
  for (int i = 0; i < nm; ++i) {
    inla_model* m = b->models[i];
    const int no = out_size(m->d);
    int32_t tcs = 0;
    BTA_CUDA_TRY(cudaMemcpy(&tcs, m->ctx[0].fail + 2, sizeof(int32_t), cudaMemcpyDeviceToHost));
    m->last.assign(m->hout, m->hout + no);
    m->ctx[0].have_factors = g ? 0 : 1 + prec;
    m->ctx[0].reverse = b->reverse[g][prec][i];
    m->launched += b->kernels[g][prec] / nm;
    f[i] = m->hout[0];
    if (grad)
      for (int j = 0; j < m->d; ++j) grad[(size_t)i * ldt + j] = m->hout[1 + j];
    st = worse(st, eval_status(m->hout + 1 + m->d, tcs));
  }
  return st;
}

bta_status inla_hessian(inla_model* m, const double* theta, double h, double* H, double* grad0,
                        const inla_opts* opts, cudaStream_t stream) {
  if (!m || !theta || !H || !(h > 0.0) || !finite_theta(theta, m->d)) return BTA_ERR_ARG;
  const int d = m->d;
  // rows: theta, then theta + h e_j, theta - h e_j for every j (Eq. 13)
  std::vector<double> pts((size_t)(2 * d + 1) * d), f(2 * d + 1), g((size_t)(2 * d + 1) * d);
  for (int r = 0; r < 2 * d + 1; ++r)
    for (int j = 0; j < d; ++j) pts[(size_t)r * d + j] = theta[j];
  for (int j = 0; j < d; ++j) {
    pts[(size_t)(1 + 2 * j) * d + j] += h;
    pts[(size_t)(2 + 2 * j) * d + j] -= h;
  }
  inla_opts o = opts ? *opts : inla_opts{0, 1, 1, 0};
  if (o.streams < 1) o.streams = 1;
  bta_status st = inla_value_and_grad(m, pts.data(), 2 * d + 1, f.data(), g.data(), &o, stream);
  if (st != BTA_OK) return st;
  for (int j = 0; j < d; ++j)
    for (int i = 0; i < d; ++i)   // column j: central difference of the gradient along e_j
      H[(size_t)i * d + j] = (g[(size_t)(1 + 2 * j) * d + i] - g[(size_t)(2 + 2 * j) * d + i]) /
                             (2.0 * h);
  if (grad0)
    for (int i = 0; i < d; ++i) grad0[i] = g[i];
  return BTA_OK;
}

bta_status inla_last_parts(const inla_model* m, double* parts, double* phases) {
  if (!m || m->last.empty()) return BTA_ERR_STATE;
  const double* p = m->last.data() + 1 + m->d;
  if (parts)
    for (int i = 0; i < kOutParts; ++i) parts[i] = p[i];
  if (phases)
    for (int i = 0; i < 4 * m->d; ++i) phases[i] = p[kOutParts + i];
  return BTA_OK;
}

bta_status inla_copy_mode(const inla_model* m, double* dst, cudaStream_t stream) {
  if (!m || !dst) return BTA_ERR_ARG;
  if (m->ctx.empty()) return BTA_ERR_STATE;
  BTA_CUDA_TRY(cudaMemcpyAsync(dst, m->ctx[0].x, ((size_t)m->n * m->ld + m->a) * sizeof(double),
                               cudaMemcpyDeviceToDevice, stream));
  return BTA_OK;
}

int64_t inla_kernel_launches(const inla_model* m) { return m ? m->launched : g_launches; }

}  // extern "C"
