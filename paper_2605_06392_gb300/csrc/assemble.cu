// Assembly of the BTA blocks of Q_p(theta) and Q_c(theta) (Section II-A,
// computational structure; Eq. 10 for the coregionalised super-blocks) and
// the closed-form theta-derivatives of their Kronecker coefficients
// (Eqs. 11-12), all on the device.
//
// Block expansion used everywhere:  for time blocks (t, t') with t' in
// {t, t-1} and variable pair (p, q),
//     Q^(pq)(t, t') = sum_j Mj[t, t'] sum_s coef[pq][j][s] S_s,
// with S_s in {Cm, G, GG} and, per variable m with unit scale,
//     u_m[0] = (kappa^4, 2 kappa^2, 1)        (M0 (x) K0)
//     u_m[1] = (2 kappa^3 gamma, 2 kappa gamma, 0)   (2 kappa gamma M1 (x) K1)
//     u_m[2] = (1, 0, 0)                      (M2 (x) Cm)
//     coef[pq][j][s] = sum_m W_pq^(m) u_m[j][s]   (k > 1),  e^{theta_1} u[j][s] (k = 1),
// W_pq^(m) = (Lambda^{-1})_{mp} (Lambda^{-1})_{mq}.
#include "model.cuh"

namespace bta {
namespace {

__device__ void unit_terms(double kap, double gam, double u[kNJ][kNS], double dk[kNJ][kNS],
                           double dg[kNJ][kNS]) {
  double k2 = kap * kap, k3 = k2 * kap, k4 = k2 * k2;
  for (int j = 0; j < kNJ; ++j)
    for (int s = 0; s < kNS; ++s) u[j][s] = dk[j][s] = dg[j][s] = 0.0;
  u[0][0] = k4;            dk[0][0] = 4 * k4;
  u[0][1] = 2 * k2;        dk[0][1] = 4 * k2;
  u[0][2] = 1.0;
  u[1][0] = 2 * k3 * gam;  dk[1][0] = 6 * k3 * gam;  dg[1][0] = 2 * k3 * gam;
  u[1][1] = 2 * kap * gam; dk[1][1] = 2 * kap * gam; dg[1][1] = 2 * kap * gam;
  u[2][0] = 1.0;
}

struct CoefArgs {
  int k, d, nt;
  const double* m_diag;
  const double* m_sub;
  CoefLayout L;
};

// One CTA: the scalars (exponentials, Lambda^{-1}) by a few threads, then every
// coefficient, derivative and block coefficient by a thread of its own, its terms summed
// in the order of m (or j).  One thread for all of them took 190 us at k = 3, nt = 5
// (72 clocks a dependent FP64 operation), now 11 us.
constexpr int kCoefThreads = 512;
__global__ void __launch_bounds__(kCoefThreads) coef_kernel(CoefArgs a, double* buf) {
  const int k = a.k, d = a.d, kk = k * k, tid = threadIdx.x;
  const CoefLayout& L = a.L;
  const double* th = buf + L.theta;
  double* tau = buf + L.tau;
  double* coef = buf + L.coef;
  double* dcoef = buf + L.dcoef;
  __shared__ double u[kMaxK][kNJ][kNS], dk[kMaxK][kNJ][kNS], dg[kMaxK][kNJ][kNS];
  __shared__ double Lam[kMaxK][kMaxK], Li[kMaxK][kMaxK];
  __shared__ double C[kMaxK * kMaxK * kNJ * kNS];
  const int nc = k * (k - 1) / 2;
  if (k == 1) {
    if (tid == 0) {
      unit_terms(exp(th[1]), exp(th[2]), u[0], dk[0], dg[0]);
      Lam[0][0] = exp(th[0]);   // the scale
    }
    if (tid == 32) tau[0] = exp(th[3]);
  } else {
    if (tid < k) unit_terms(exp(th[tid]), exp(th[k + tid]), u[tid], dk[tid], dg[tid]);
    if (tid >= 32 && tid < 32 + k) tau[tid - 32] = exp(th[3 * k + nc + tid - 32]);
    if (tid >= 64 && tid < 64 + kk) {   // Lambda (lower)
      const int p = (tid - 64) / k, q = (tid - 64) % k;
      Lam[p][q] = p == q ? exp(th[2 * k + p]) : p > q ? th[3 * k + p * (p - 1) / 2 + q] : 0.0;
    }
    __syncthreads();
    if (tid < k) {   // column tid of its inverse by forward substitution
      for (int i = 0; i < k; ++i) Li[i][tid] = 0.0;
      Li[tid][tid] = 1.0 / Lam[tid][tid];
      for (int i = tid + 1; i < k; ++i) {
        double s = 0.0;
        for (int r = tid; r < i; ++r) s += Lam[i][r] * Li[r][tid];
        Li[i][tid] = -s / Lam[i][i];
      }
    }
  }
  __syncthreads();
  const int nterm = kk * kNJ * kNS;
  for (int e = tid; e < nterm; e += kCoefThreads) {
    const int pq = e / (kNJ * kNS), j = (e / kNS) % kNJ, s = e % kNS, p = pq / k, q = pq % k;
    double c = 0.0;
    if (k == 1) c = Lam[0][0] * u[0][j][s];
    else
      for (int m = 0; m < k; ++m) c += Li[m][p] * Li[m][q] * u[m][j][s];
    coef[e] = C[e] = c;
  }
  for (int e = tid; e < d * nterm; e += kCoefThreads) {
    const int t = e / nterm, pq = e / (kNJ * kNS) % kk, j = (e / kNS) % kNJ, s = e % kNS;
    const int p = pq / k, q = pq % k;
    double v = 0.0;
    if (k == 1) {
      if (t < 3) v = Lam[0][0] * (t == 0 ? u : t == 1 ? dk : dg)[0][j][s];
    } else if (t < 2 * k) {   // d / d log kappa_m, d / d log gamma_m (Eq. 11)
      const int m = t % k;
      v = Li[m][p] * Li[m][q] * (t < k ? dk : dg)[m][j][s];
    } else if (t < 3 * k + nc) {
      // coupling-type parameters (Eq. 12): dLambda^{-1} = -Li E Li
      const int c = t - 2 * k;
      int er = c, ec = c;
      double ew = 1.0;
      if (c < k) ew = Lam[c][c];
      else {
        er = 1;
        ec = c - k;
        while (ec >= er) ec -= er++;
      }
      for (int m = 0; m < k; ++m) {
        const double dLp = -ew * Li[m][er] * Li[ec][p];
        const double dLq = -ew * Li[m][er] * Li[ec][q];
        v += (dLp * Li[m][q] + Li[m][p] * dLq) * u[m][j][s];
      }
    }
    dcoef[e] = v;
  }
  __syncthreads();
  // Per-block expansion coefficients.
  double* aD = buf + L.alphaD;
  double* aB = buf + L.alphaB;
  for (int e = tid; e < a.nt * kk * kNS; e += kCoefThreads) {
    const int t = e / (kk * kNS), pq = e / kNS % kk, s = e % kNS;
    double vd = 0.0, vb = 0.0;
    for (int j = 0; j < kNJ; ++j) {
      const double c = C[(pq * kNJ + j) * kNS + s];
      vd += a.m_diag[j * a.nt + t] * c;
      if (t + 1 < a.nt) vb += a.m_sub[j * (a.nt - 1) + t] * c;
    }
    aD[e] = vd;
    if (t + 1 < a.nt) aB[e] = vb;
  }
}

struct AsmArgs {
  int k, ns, b, ld, nnz, cond, diag;
  int t0;                 // time block of output block 0 (coefficients, counts)
  const int32_t* row_ptr;
  const int32_t* col;
  const double* val;      // [kNS][nnz]
  const double* alpha;    // [nblk][kk][kNS]
  const double* tau;
  const double* cnt;      // [nt*ld]
};

// One CTA per column c of output block blockIdx.y (time block t0 + blockIdx.y):
// zero-fill, then scatter the stencil.
__global__ void __launch_bounds__(256) assemble_kernel(AsmArgs a, double* out) {
  const int c = blockIdx.x, t = a.t0 + blockIdx.y;
  const int ld = a.ld;
  double* colp = out + ((int64_t)blockIdx.y * ld + c) * ld;
  if (reinterpret_cast<uintptr_t>(colp) % 16) {   // a caller's blocks on an 8-byte boundary
    for (int r = threadIdx.x; r < ld; r += blockDim.x) colp[r] = 0.0;
  } else {
    double2* col2 = reinterpret_cast<double2*>(colp);
    for (int r = threadIdx.x; r < ld / 2; r += blockDim.x) col2[r] = make_double2(0.0, 0.0);
  }
  __syncthreads();
  if (c >= a.b) {
    if (a.diag && threadIdx.x == 0) colp[c] = 1.0;
    return;
  }
  const int q = c / a.ns, s2 = c % a.ns;
  const int e0 = a.row_ptr[s2], e1 = a.row_ptr[s2 + 1];
  const int kk = a.k * a.k;
  const double* al = a.alpha + (int64_t)t * kk * kNS;
  const int len = e1 - e0;
  for (int w = threadIdx.x; w < len * a.k; w += blockDim.x) {
    int p = w / len, e = e0 + w % len;
    int s1 = a.col[e];
    const double* ap = al + (p * a.k + q) * kNS;
    double v = ap[0] * a.val[e] + ap[1] * a.val[a.nnz + e] + ap[2] * a.val[2 * a.nnz + e];
    int r = p * a.ns + s1;
    if (a.cond && a.diag && r == c) v += a.tau[p] * a.cnt[(int64_t)t * ld + r];
    colp[r] = v;
  }
}

__global__ void assemble_arrow(int nt, int a, int ld, int ns, int a_r, const double* tau,
                               const double* craw, double* C) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t total = (int64_t)nt * a * ld;
  if (i >= total) return;
  int f = (int)(i % a);
  C[i] = tau[f / a_r] * craw[i];
}

__global__ void assemble_tip(int a, int k, double tip, const double* tau, const double* traw,
                             double* T) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a * a) return;
  double v = (i % a == i / a) ? tip : 0.0;
  for (int m = 0; m < k; ++m) v += tau[m] * traw[(int64_t)m * a * a + i];
  T[i] = v;
}

__global__ void assemble_rhs(int nt, int ld, int ns, int b, int a, int a_r, const double* tau,
                             const double* rraw, double* r) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t lat = (int64_t)nt * ld;
  if (i >= lat + a) return;
  int v;
  if (i < lat) {
    int row = (int)(i % ld);
    if (row >= b) { r[i] = 0.0; return; }
    v = row / ns;
  } else {
    v = (int)(i - lat) / a_r;
  }
  r[i] = tau[v] * rraw[i];
}

}  // namespace

bta_status launch_coef(const ModelDev& md, const CoefLayout& L, double* coefbuf, cudaStream_t s) {
  CoefArgs a{md.k, md.d, md.nt, md.m_diag, md.m_sub, L};
  coef_kernel<<<1, kCoefThreads, 0, s>>>(a, coefbuf);
  BTA_LAUNCHED();
  return BTA_OK;
}

bta_status launch_rhs(const ModelDev& md, const CoefLayout& L, const double* coefbuf, double* rhs,
                      cudaStream_t s) {
  const int64_t tot = (int64_t)md.nt * md.ld + md.a;
  assemble_rhs<<<cdiv(tot, 256), 256, 0, s>>>(md.nt, md.ld, md.ns, md.b, md.a, md.a_r,
                                               coefbuf + L.tau, md.rraw, rhs);
  BTA_LAUNCHED();
  return BTA_OK;
}

bta_status launch_assemble(const ModelDev& md, const CoefLayout& L, const double* coefbuf,
                           int cond, const bta_desc& q, double* rhs, cudaStream_t s) {
  const int ld = md.ld;
  AsmArgs a{md.k, md.ns, md.b, ld, md.nnz, cond, 1, 0, md.row_ptr, md.col, md.val,
            coefbuf + L.alphaD, coefbuf + L.tau, md.cnt};
  assemble_kernel<<<dim3(ld, md.nt), 256, 0, s>>>(a, q.D);
  BTA_LAUNCHED();
  if (md.nt > 1 && q.B) {   // no B storage: the sweeps assemble B_i per step
    a.diag = 0;
    a.alpha = coefbuf + L.alphaB;
    assemble_kernel<<<dim3(ld, md.nt - 1), 256, 0, s>>>(a, q.B);
    BTA_LAUNCHED();
  }
  if (cond && md.a > 0) {
    int64_t tot = (int64_t)md.nt * md.a * ld;
    assemble_arrow<<<cdiv(tot, 256), 256, 0, s>>>(md.nt, md.a, ld, md.ns, md.a_r,
                                                  coefbuf + L.tau, md.craw, q.C);
    BTA_LAUNCHED();
    assemble_tip<<<cdiv(md.a * md.a, 256), 256, 0, s>>>(md.a, md.k, md.tip_prior,
                                                        coefbuf + L.tau, md.traw, q.T);
    BTA_LAUNCHED();
  }
  if (cond && rhs) {
    int64_t tot = (int64_t)md.nt * ld + md.a;
    assemble_rhs<<<cdiv(tot, 256), 256, 0, s>>>(md.nt, ld, md.ns, md.b, md.a, md.a_r,
                                                 coefbuf + L.tau, md.rraw, rhs);
    BTA_LAUNCHED();
  }
  return BTA_OK;
}

bta_status launch_assemble_b(const ModelDev& md, const CoefLayout& L, const double* coefbuf,
                             int i, double* dst, cudaStream_t s) {
  if (i < 0 || i >= md.nt - 1) return BTA_ERR_ARG;
  AsmArgs a{md.k, md.ns, md.b, md.ld, md.nnz, 0, 0, i, md.row_ptr, md.col, md.val,
            coefbuf + L.alphaB, coefbuf + L.tau, md.cnt};
  assemble_kernel<<<dim3(md.ld, 1), 256, 0, s>>>(a, dst);
  BTA_LAUNCHED();
  return BTA_OK;
}

}  // namespace bta
