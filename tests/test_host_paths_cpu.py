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
