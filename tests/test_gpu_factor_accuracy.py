"""Precision of the factor's small parts: diagonal blocks and tip."""
import numpy as np
import pytest

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


def _factor(P, D, T=None, rhs=None, precision=0):
    """The factor of one diagonal block D and a tip T without coupling: (logdet, D, T, rhs)."""
    import torch
    b, a = D.shape[0], 0 if T is None else T.shape[0]
    ld = (b + 31) // 32 * 32
    q = P.BtaMatrix(1, b, a, ld)
    full = np.eye(ld)
    full[:b, :b] = D
    q.D.copy_(torch.from_numpy(full).cuda().reshape(q.D.shape))   # symmetric
    if a:
        q.C.zero_()
        q.T.copy_(torch.from_numpy(T).cuda().reshape(q.T.shape))
    q.desc.state = 1
    x = None if rhs is None else torch.from_numpy(rhs).cuda()
    logdet, fail = P.bta_factor(q, rhs=x, precision=precision)
    torch.cuda.synchronize()
    assert int(fail.item()) == -1
    return (logdet.cpu().numpy(), np.tril(q.D.cpu().numpy().reshape(ld, ld).T), q,
            None if x is None else x.cpu().numpy())


@pytest.mark.parametrize("b", [40, 64, 192, 512])
@pytest.mark.parametrize("precision", [1, 2])
def test_graded_blocks_up_to_512_rows_as_in_fp64(P, b, precision):
    """Rows from 1e-6 to 1e6: the tensor-core modes factor such a block with FP64 tile
    products, to the same bits as the FP64 mode."""
    rng = np.random.default_rng(b)
    s = 10.0 ** rng.uniform(-6, 6, b)
    g = rng.standard_normal((b, b + 8))
    D = g @ g.T / b + 0.05 * np.eye(b)
    D = 0.5 * (D + D.T) * np.outer(s, s)
    ref = _factor(P, D)
    got = _factor(P, D, precision=precision)
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])


@pytest.mark.parametrize("a", [1, 7, 32])
def test_tip_divides_by_its_pivots(P, a):
    """Correctly rounded quotients in the tip's factor and solves (a rounded reciprocal
    would cost a second rounding): a diagonal tip's solutions and a first column of L_T are
    those of IEEE division and square root."""
    import torch
    rng = np.random.default_rng(a)
    eye = np.eye(32)
    for _ in range(8):
        t = np.exp(rng.uniform(-9, 9, a))
        r = np.concatenate([np.zeros(32), rng.standard_normal(a)])
        _, _, q, z = _factor(P, eye, np.diag(t), r)
        z_ref = r[32:] / np.sqrt(t)
        assert np.array_equal(z[32:], z_ref)
        x = torch.from_numpy(z).cuda()
        P.bta_solve(q, x)
        assert np.array_equal(x.cpu().numpy()[32:], z_ref / np.sqrt(t))
        zl = torch.from_numpy(r).cuda()                  # the lower solve on its own
        P.bta_solve(q, zl, lower=True)
        assert np.array_equal(zl.cpu().numpy(), x.cpu().numpy())
        T = np.diag(np.full(a, 1e3))
        T[0, 0] = np.exp(rng.uniform(-1, 1))
        T[1:, 0] = T[0, 1:] = rng.standard_normal(a - 1)
        _, _, q, _ = _factor(P, eye, T)
        L = q.T.cpu().numpy().reshape(a, a).T            # column-major
        assert np.array_equal(L[1:, 0], T[1:, 0] / np.sqrt(T[0, 0]))
