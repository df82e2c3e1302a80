"""Evaluations in the smaller workspaces (one leg per matrix, the products' planes of seven
or four moduli at once): the same bar as elsewhere, relative 1e-10 against the oracle on f, every
gradient component and x*; low-memory models take them by size."""
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


def _check(m, prob, precision):
    from oracle import bta
    f, g = m.value_and_grad(prob.theta, precision=precision)
    x = m.mode().cpu().numpy()
    fv, _ = m.value_and_grad(prob.theta, grad=False, precision=precision)
    assert fv == f
    o = bta.evaluate(prob)
    scale = np.maximum(np.abs(o.grad), np.abs(o.phase_a) + np.abs(o.phase_b) + np.abs(o.phase_c))
    err = (abs(f - o.f) / abs(o.f), float(np.max(np.abs(g - o.grad) / scale)),
           float(np.max(np.abs(x - o.x)) / np.max(np.abs(o.x))))
    assert max(err) <= 1e-10, err
    return f, g


# partial exponent maxima up to K = 1024, atomic ones above; tiles of 128 and 256; an arrow
# beside the blocks, none, and one too wide for the cluster kernel
@pytest.mark.parametrize("over", [
    dict(nt=1), dict(nt=4), dict(nt=4, a=0), dict(nt=3, a=17), dict(nx=13, ny=11, nt=5),
    dict(nx=24, ny=25, nt=3, n_obs=1500), dict(nx=35, ny=32, nt=3, n_obs=2000),
], ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()))
@pytest.mark.parametrize("precision,low,form", [(0, False, 1), (2, False, 1), (2, False, 2),
                                                (0, True, 1), (2, True, 2)])
def test_small_workspaces_against_oracle(P, monkeypatch, over, precision, low, form):
    prob = workloads.make_problem("st_tiny", **over)
    monkeypatch.setenv("BTA_SMALL_WORKSPACES", str(form))
    m = P.InlaModel(prob, low_memory=low)
    _check(m, prob, precision)
    m.close()


def test_low_memory_of_a_large_block(P):
    prob = workloads.make_problem("st_tiny", nx=40, ny=35, nt=3, n_obs=2000)
    m = P.InlaModel(prob, low_memory=True)
    _check(m, prob, 2)
    m.close()


def test_modes_share_a_model(P):
    """Workspaces come with the first evaluation of a mode; the others' results stay."""
    import torch
    prob = workloads.make_problem("st_tiny", nx=20, ny=18, nt=5)
    m = P.InlaModel(prob)
    first = [m.value_and_grad(prob.theta, precision=p) for p in (2, 1, 0)]
    th = torch.tensor(prob.theta, dtype=torch.float64, requires_grad=True)
    P.inla_objective(th, m).backward()
    again = [m.value_and_grad(prob.theta, precision=p) for p in (0, 1, 2)][::-1]
    m.close()
    fresh = []
    for p in (2, 1, 0):
        m = P.InlaModel(prob)
        fresh.append(m.value_and_grad(prob.theta, precision=p))
        m.close()
    for (f0, g0), (f1, g1), (f2, g2) in zip(first, again, fresh):
        assert f0 == f1 == f2
        assert np.array_equal(g0, g1) and np.array_equal(g0, g2)
    assert np.array_equal(th.grad.numpy(), first[2][1])


@pytest.mark.parametrize("M,N,K,transA,transB", [(64, 16500, 96, False, False),
                                                 (70, 16400, 1030, True, True),
                                                 (16390, 130, 64, False, True)])
def test_panels_of_a_large_product(P, M, N, K, transA, transB):
    """Panels of 16384 rows and columns: the bits of products of the parts, whose operands'
    rows and columns are the same."""
    import torch
    g = torch.Generator().manual_seed(M + N)
    A = torch.randn((M, K) if transA else (K, M), generator=g, dtype=torch.float64).cuda()
    B = torch.randn((K, N) if transB else (N, K), generator=g, dtype=torch.float64).cuda()
    C0 = torch.randn((N, M), generator=g, dtype=torch.float64).cuda()
    whole = C0.clone()
    assert int(P.bta_gemm_emulated(A, B, whole, alpha=0.5, beta=-1.0, transA=transA,
                                   transB=transB).item()) == 0
    h = N // 2
    for lo, hi in ((0, h), (h, N)) if N > M else ((0, N),):
        r = (M // 2, M - M // 2) if M > N else (M,)
        m0 = 0
        for m in r:
            a = A[m0:m0 + m] if transA else A[:, m0:m0 + m]
            b = B[:, lo:hi] if transB else B[lo:hi]
            c = C0[lo:hi, m0:m0 + m].contiguous()
            P.bta_gemm_emulated(a.contiguous(), b.contiguous(), c, alpha=0.5, beta=-1.0,
                                transA=transA, transB=transB)
            torch.cuda.synchronize()
            assert torch.equal(whole[lo:hi, m0:m0 + m], c)
            m0 += m


def test_slices_select_no_other_arithmetic(P):
    """slices (6..8) states the accuracy asked for: one product serves all."""
    import torch
    g = torch.Generator().manual_seed(1)
    A = torch.randn(300, 200, generator=g, dtype=torch.float64).cuda()
    B = torch.randn(250, 300, generator=g, dtype=torch.float64).cuda()
    out = []
    for slices in (6, 7, 8):
        C = torch.zeros(250, 200, dtype=torch.float64, device="cuda")
        P.bta_gemm_emulated(A, B, C, slices=slices)
        out.append(C.cpu())
    ref = (B.cpu() @ A.cpu())
    bound = 300 * 2.0 ** -55 * A.abs().amax(0)[None, :].cpu() * B.abs().amax(1)[:, None].cpu() \
        + 304 * 2.0 ** -53 * (B.abs() @ A.abs()).cpu()
    assert torch.equal(out[0], out[1]) and torch.equal(out[1], out[2])
    assert bool(((out[2] - ref).abs() <= bound).all())
