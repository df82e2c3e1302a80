"""Host code of the library on a CUDA runtime without a GPU (fakecuda)."""
import ctypes as C

import pytest

import workloads
from fakecuda import Stream, load


@pytest.fixture
def fake(tmp_path_factory, monkeypatch):
    return load(tmp_path_factory.mktemp("fakecuda")).install(monkeypatch)


def _ptr(x):
    return C.c_void_p(x << 8)


def _factor(fake, n, b, a, precision, noalloc=False):
    from paper_2605_06392_gb300._capi import bta_desc
    ld = (b + 31) // 32 * 32
    q = bta_desc(n=n, b=b, a=a, ld=ld, D=1 << 30, B=1 << 31, C=1 << 32, T=1 << 33, state=1)
    if noalloc:
        return fake.lib.bta_factor_noalloc(C.byref(q), None, _ptr(1), _ptr(2), None)
    return fake.lib.bta_factor(C.byref(q), None, _ptr(1), _ptr(2), precision, None)


# ---- several devices in one process ------------------------------------------
@pytest.mark.parametrize("call", [
    lambda f: _factor(f, 2, 64, 0, 0), lambda f: _factor(f, 2, 64, 0, 0, noalloc=True),
    lambda f: _factor(f, 2, 1024, 0, 1), lambda f: _factor(f, 2, 1024, 0, 2),
    lambda f: f.lib.bta_gemm_mixed(64, 64, 64, 1.0, _ptr(1), 64, 0, _ptr(1), 64, 0, 0.0, _ptr(1),
                                   64, None, None),
    lambda f: f.lib.bta_gemm_emulated(64, 64, 64, 1.0, _ptr(1), 64, 0, _ptr(1), 64, 0, 0.0,
                                      _ptr(1), 64, 8, None, None),
    lambda f: f.lib.bta_gemm_emulated(2048, 2048, 64, 1.0, _ptr(1), 2048, 0, _ptr(1), 2048, 0,
                                      0.0, _ptr(1), 2048, 8, None, None),
], ids=["fp64", "noalloc", "mixed", "emulated", "gemm_mixed", "gemm_emulated", "gemm_pairs"])
def test_kernel_attributes_on_every_device(fake, call):
    """The limit on a kernel's dynamic shared memory belongs to a device."""
    for dev in (0, 3, 0, 70):
        fake.device(dev)
        assert call(fake) == 0, dev


# ---- the task graph's grid ----------------------------------------------------
def _leaves(fake):
    """(rows, matrices, CTAs, bulk tasks yield) of the task graphs launched."""
    return [(32 * fake.head(i, 0), fake.head(i, 2), grid[0], fake.head(i, 10))
            for name, grid, i in fake.launches() if "potrf_dag_kernel" in name]


def _evaluate(fake, precision, count=1, grad=False, low_memory=False, **over):
    """Task graphs of an evaluation of `count` thetas together."""
    import numpy as np

    import paper_2605_06392_gb300 as P
    prob = workloads.make_problem("st_tiny", **over)
    m = P.InlaModel(prob, low_memory=low_memory)
    fake.reset()
    m.value_and_grad(np.array([prob.theta] * count), grad=grad, use_graph=False, concurrent=count,
                     precision=precision, stream=Stream())
    got = _leaves(fake)
    m.close()
    assert got
    return got


@pytest.mark.parametrize("nx", [4, 8, 12, 16])
@pytest.mark.parametrize("count", [1, 2])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_a_yielding_grid_has_a_free_cta(fake, precision, count, nx):
    """Bulk tasks that yield wait for the chain on their SM, which waits for them: with two
    CTAs an SM, at least one CTA must lie outside the chains' SMs."""
    for rows, matrices, ctas, yields in _evaluate(fake, precision, count, nx=nx):
        assert not yields or ctas > 2 * matrices, (rows, matrices, ctas)


@pytest.mark.parametrize("count", [1, 4, 16])
@pytest.mark.parametrize("precision", [1, 2])
def test_every_matrix_of_a_set_brings_its_ctas(fake, precision, count):
    """A set's bulk tasks grow with its matrices: so do the CTAs, up to the SMs."""
    for rows, matrices, ctas, _ in _evaluate(fake, precision, count, nx=24, ny=25):
        assert matrices == count and ctas >= min(152, count * rows // 16), (rows, ctas)


# ---- diagonal factors in the tensor-core modes -------------------------------
@pytest.mark.parametrize("b", [32, 64, 192, 480, 512])
@pytest.mark.parametrize("precision", [1, 2])
def test_blocks_up_to_512_rows_keep_fp64_tile_products(fake, b, precision):
    """potrf_dag_kernel<false>: emulated tile products (<true>) begin above 512 rows."""
    assert _factor(fake, 2, b, 0, precision) == 0
    names = [n for n, _, _ in fake.launches() if "potrf_dag_kernel" in n]
    assert len(names) == 2 and all("ILb0E" in n for n in names), names


# ---- workspaces ---------------------------------------------------------------
def _pad(n, m):
    return (n + m - 1) // m * m


LD, A, NT = 2080, 4, 5
BLOCK = 8 * LD * LD
PLANE = _pad(LD + A, 256) * _pad(LD + A, 256)   # entries of a product's padded operand


def _model(low=False):
    import paper_2605_06392_gb300 as P
    prob = workloads.make_problem("st_tiny", nx=65, ny=32, nt=NT, a=A, n_obs=400)
    return prob, P.InlaModel(prob, low_memory=low)


def _run(m, prob, precision, count=1, **kw):
    import numpy as np
    th = np.array([prob.theta] * count)
    return m.value_and_grad(th, use_graph=False, precision=precision, concurrent=count,
                            stream=Stream(), **kw)


def _work_of(fake, precision, low):
    """Bytes of a model that has been evaluated, beside its matrices' blocks."""
    before = fake.live()
    prob, m = _model(low)
    _run(m, prob, precision)
    work = fake.live() - before - 2 * (NT + (0 if low else NT - 1)) * BLOCK
    m.close()
    assert fake.live() == before
    return work


@pytest.mark.parametrize("precision,low,want", [
    # legs of three blocks each; the products' planes: two operands' and the result's, of 14
    # moduli (low memory: of 7, and one leg a matrix); TF32: high and low parts of two
    (0, False, 4 * 3 * BLOCK),
    (1, False, 2 * (3 * BLOCK + 16 * LD * LD)),
    (2, False, 4 * (3 * BLOCK + 84 * PLANE)),
    (0, True, 4 * 3 * BLOCK),
    (2, True, 2 * (3 * BLOCK + 56 * PLANE)),
])
def test_workspaces_follow_legs_and_mode(fake, precision, low, want):
    work = _work_of(fake, precision, low)
    half = 84 * _pad(_pad(LD, 64) // 2, 256) ** 2       # the diagonal factor's products
    if precision == 1:
        want = max(want, 2 * (3 * BLOCK + half))
    assert work <= want + 0.02 * want + (4 << 20), work / want


def test_large_models_of_every_mode_fit_where_they_did(fake):
    """b = 4800: an evaluation finds a form that fits into what two legs of four blocks and
    40 bytes an entry once took."""
    import paper_2605_06392_gb300 as P
    prob = workloads.make_problem("coreg_production", nt=4, n_obs=600)
    blk, once = 8 * 4800 ** 2, 2 * (4 * 8 * 4800 ** 2 + 40 * 4864 ** 2)
    for precision, low in ((0, False), (1, False), (2, False), (0, True), (2, True)):
        before = fake.live()
        m = P.InlaModel(prob, low_memory=low)
        fake.reset(limit=before + 2 * (4 + (0 if low else 3)) * blk + once + (48 << 20))
        for grad in (False, True):
            f, _ = m.value_and_grad(prob.theta, use_graph=False, precision=precision, grad=grad,
                                    stream=Stream())
        m.close()
        assert fake.live() == before


def test_out_of_memory_leaves_the_model_as_it_was(fake):
    from paper_2605_06392_gb300._capi import BtaError
    prob, m = _model()
    _run(m, prob, 0)
    live = fake.live()
    fake.reset(limit=live + 80 * PLANE)             # less than the small form's 2 x 44
    with pytest.raises(BtaError, match="memory"):
        _run(m, prob, 2)
    with pytest.raises(BtaError, match="memory"):
        _run(m, prob, 0, count=2)                   # a second context does not fit either
    assert fake.live() == live
    _run(m, prob, 0)
    fake.reset(limit=live + 90 * PLANE)
    _run(m, prob, 2)                                # now the small form does
    m.close()


def test_reverse_pass_takes_the_order_of_its_factor(fake):
    """A value by two legs a matrix, then by one (a set that finds no room for two): each
    reverse pass runs in the order of the factors held, whatever a failed call tried since."""
    import numpy as np

    def legs(m):
        fake.reset()
        g = np.zeros(m.d)
        assert fake.lib.inla_backward(m.handle, g.ctypes.data_as(C.POINTER(C.c_double)), 0,
                                      None) == 0
        return len(fake.streams() - {0})

    from paper_2605_06392_gb300._capi import BtaError
    prob, m = _model()
    second = (2 * (2 * NT - 1) + 6) * BLOCK         # another context, without its planes
    for room, streams in ((second + 60 * PLANE, 4), (second + 2 * 46 * PLANE, 2)):
        _run(m, prob, 2, grad=False)
        assert legs(m) == 4
        _run(m, prob, 2, grad=False)
        fake.reset(limit=fake.live() + room)
        if streams == 4:
            with pytest.raises(BtaError, match="memory"):
                _run(m, prob, 2, count=2, grad=False)
        else:
            _run(m, prob, 2, count=2, grad=False)
        assert legs(m) == streams
    m.close()


# ---- emulated products beyond one panel ---------------------------------------
def _gemm(fake, M, N, K, transA=0, transB=0, A=1 << 40, B=1 << 42, Cm=1 << 44):
    return fake.lib.bta_gemm_emulated(M, N, K, 1.0, C.c_void_p(A), K if transA else M, transA,
                                      C.c_void_p(B), N if transB else K, transB, 0.0,
                                      C.c_void_p(Cm), M, 8, None, None)


@pytest.mark.parametrize("M,N,K", [(90000, 90000, 512), (1500000, 64, 5120), (64, 1500000, 5120)])
def test_large_emulated_products_need_no_more_room(fake, M, N, K):
    """Beside their operands such products took 16 bytes an operand entry and 8 a result's."""
    room = 16 * (M + N) * K + 8 * M * N
    fake.reset(limit=room)
    assert _gemm(fake, M, N, K) == 0
    assert fake.peak() <= room and fake.live() == 0


@pytest.mark.parametrize("M,N,K", [(300, 200, 64), (5000, 3000, 256), (4096, 4096, 5120)])
def test_emulated_products_under_a_full_device(fake, M, N, K):
    assert _gemm(fake, M, N, K) == 0
    once = max(16 * (M + N) * K + 8 * M * N, 32 << 20)
    fake.reset(limit=once)
    assert _gemm(fake, M, N, K) == 0
    assert _gemm(fake, M, N, K, 1, 1) == 0
    fake.reset(limit=1 << 20)
    assert _gemm(fake, M, N, K) == -4
    assert fake.lib.bta_gemm(8, 8, 8, 1.0, _ptr(1), 8, 0, _ptr(1), 8, 0, 0.0, _ptr(1), 8,
                             None) == 0                          # no error left behind


def test_a_result_in_place_of_an_operand_is_not_split(fake):
    n = 4000
    fake.reset()
    assert _gemm(fake, n, n, n, Cm=1 << 40) == 0
    whole = fake.peak()
    fake.reset(limit=whole // 2)
    assert _gemm(fake, n, n, n, Cm=1 << 40) == -4
    assert _gemm(fake, n, n, n) == 0
