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
