"""Sizes at which the kernels of the sweeps change their path or end raggedly.

Products in residues (bta_gemm_emulated): an operand entry is rounded to bits = 56 (55 for
K > 4847) binary places below its row's power of two, so it is off by at most 2^-bits times
the row's largest entry; two operands and K terms give K 2^(1 - bits) max|a_i| max|b_j|.
Added to that are the roundings of the result and of the FP64 reference, at most
(K + 4) 2^-53 (|A| |B| + |C0|).

Evaluations: relative 1e-10 against the oracle (FP64 and emulated FP64), as elsewhere."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_06392_gb300 import build
    build.build()
    import paper_2605_06392_gb300 as P
    return P


# tiles of 128 (up to 8 units an SM: 81 tiles) and of 256; slabs of 64, two a stage; chunks of
# 256; blocks of 16 rows; partial maxima up to K = 1024; 56 bits up to K = 4847
@pytest.mark.parametrize("M,N,K", [
    (1, 1, 1), (16, 17, 63), (127, 129, 64), (128, 128, 65), (257, 383, 257), (33, 500, 1024),
    (500, 33, 1025), (140, 150, 4847), (140, 150, 4848), (96, 97, 5120), (1152, 1152, 70),
    (1153, 1152, 70), (1300, 1030, 321),
])
@pytest.mark.parametrize("transA,transB", [(False, False), (True, True), (False, True)])
def test_residue_products(P, M, N, K, transA, transB):
    import torch
    g = torch.Generator().manual_seed(M + 5 * N + 11 * K)
    A = torch.randn((M, K) if transA else (K, M), generator=g, dtype=torch.float64)
    B = torch.randn((K, N) if transB else (N, K), generator=g, dtype=torch.float64)
    C0 = torch.randn((N, M), generator=g, dtype=torch.float64)
    a = (A if transA else A.T).numpy()
    b = (B if transB else B.T).numpy()
    c0 = C0.numpy().T
    for alpha, beta in ((1.0, 0.0), (-1.0, 1.0), (0.75, -1.5)):
        C = C0.clone().cuda()
        st = P.bta_gemm_emulated(A.cuda(), B.cuda(), C, alpha=alpha, beta=beta, transA=transA,
                                 transB=transB)
        torch.cuda.synchronize()
        assert int(st.item()) == 0
        ref = alpha * (a @ b) + beta * c0
        bits = 56 if K <= 4847 else 55
        bound = (K * 2.0 ** (1 - bits) * np.max(np.abs(a), axis=1)[:, None]
                 * np.max(np.abs(b), axis=0)[None, :]
                 + (K + 4) * 2.0 ** -53 * (np.abs(a) @ np.abs(b) + 2.0 * np.abs(c0)))
        assert np.all(np.abs(C.cpu().numpy().T - ref) <= bound), (alpha, beta)


def _errs(P, prob, precision, low):
    from oracle import bta
    m = P.InlaModel(prob, low_memory=low)
    fv, _ = m.value_and_grad(prob.theta, grad=False, precision=precision)
    f, g = m.value_and_grad(prob.theta, precision=precision)
    x = m.mode().cpu().numpy()
    m.close()
    assert fv == f
    o = bta.evaluate(prob)
    scale = np.maximum(np.abs(o.grad), np.abs(o.phase_a) + np.abs(o.phase_b) + np.abs(o.phase_c))
    return (abs(f - o.f) / abs(o.f), float(np.max(np.abs(g - o.grad) / scale)),
            float(np.max(np.abs(x - o.x)) / np.max(np.abs(o.x))))


# the two ends' legs (one leg below three blocks, an even and an odd middle), the arrow's
# cluster kernel (8 and 16 rows a group, above 16 the general product), and the blocks at
# which a product and the one whose operand planes it shares take different tiles (1152)
@pytest.mark.parametrize("over", [
    dict(nt=1), dict(nt=2), dict(nt=3), dict(nt=4), dict(nt=5), dict(nt=7),
    dict(nt=4, a=0), dict(nt=4, a=8), dict(nt=5, a=9), dict(nt=3, a=16), dict(nt=4, a=17),
    dict(nx=31, ny=32, nt=3, n_obs=1500), dict(nx=36, ny=32, nt=3, n_obs=1500),
], ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()))
@pytest.mark.parametrize("precision,low", [(0, False), (2, False), (0, True), (2, True)])
def test_legs_and_arrow(P, over, precision, low):
    err = _errs(P, workloads.make_problem("st_tiny", **over), precision, low)
    assert max(err) <= 1e-10, err


@pytest.mark.parametrize("over", [dict(nt=2), dict(nt=4), dict(nt=5), dict(nt=4, a=17)],
                         ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()))
def test_legs_mixed(P, over):
    ef, eg, ex = _errs(P, workloads.make_problem("st_tiny", **over), 1, False)
    assert ef <= 1e-6 and eg <= 1e-4 and ex <= 1e-8, (ef, eg, ex)


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("nx,ny", [(8, 8), (13, 11), (24, 25)])
def test_factor_of_unaligned_blocks(P, nx, ny, precision):
    """Diagonal blocks on 8-byte boundaries take the task graph's register loads: the same
    bits as on 16-byte ones."""
    import torch
    m = P.InlaModel(workloads.make_problem("st_tiny", nx=nx, ny=ny, nt=3, n_obs=800))
    th = workloads.make_problem("st_tiny").theta
    src = P.BtaMatrix(m.n, m.b, m.a, m.ld)
    rhs = torch.zeros(m.n * m.ld + m.a, dtype=torch.float64, device="cuda")
    P.bta_assemble(m, th, 1, src, rhs=rhs)
    out = []
    for off in (0, 1):
        q = P.BtaMatrix(m.n, m.b, m.a, m.ld)
        buf = torch.zeros(q.D.numel() + off, dtype=torch.float64, device="cuda")
        q.D = buf[off:].view(q.D.shape)
        for name in ("D", "B", "C", "T"):
            getattr(q, name).copy_(getattr(src, name))
        q.desc.D = q.D.data_ptr()
        q.desc.state = src.desc.state
        x = rhs.clone()
        logdet, fail = P.bta_factor(q, rhs=x, precision=precision)
        torch.cuda.synchronize()
        assert int(fail.item()) == -1
        out.append([t.cpu() for t in (logdet, x, q.D, q.B, q.C, q.T)])
    m.close()
    for u, v in zip(*out):
        assert torch.equal(u, v)
