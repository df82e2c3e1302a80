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
