"""The library's host code on a CUDA runtime without a GPU (runtime.cpp): which kernels it
launches, with which grids, and how much device memory it asks for."""
import ctypes as C
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


class Stream:
    cuda_stream = 0


class FakeCuda:
    """libbta on the test runtime; install(monkeypatch) puts it behind the Python binding."""

    def __init__(self, path):
        from paper_2605_06392_gb300 import _capi
        self.lib = C.CDLL(path)
        for name, (res, args) in _capi.SIGNATURES.items():
            getattr(self.lib, name).restype = res
            getattr(self.lib, name).argtypes = args
        self.lib.fake_reset.argtypes = [C.c_size_t]
        self.lib.fake_live.restype = self.lib.fake_peak.restype = C.c_size_t
        self.lib.fake_launch_name.restype = C.c_char_p
        self.lib.fake_launch_grid.restype = C.c_uint
        self.lib.fake_launch_stream.restype = C.c_size_t

    def install(self, monkeypatch):
        import torch

        from paper_2605_06392_gb300 import _capi
        monkeypatch.setattr(_capi, "_lib", self.lib)
        monkeypatch.setattr(torch.cuda, "init", lambda: None)
        self.lib.fake_set_device(0)
        self.reset()
        return self

    def reset(self, limit=2 ** 64 - 1):
        self.lib.fake_reset(limit)

    def device(self, d):
        self.lib.fake_set_device(d)

    def live(self):
        return self.lib.fake_live()

    def peak(self):
        return self.lib.fake_peak()

    def launches(self):
        """[(mangled kernel name, grid, index)] since the last reset."""
        return [(self.lib.fake_launch_name(i).decode(),
                 tuple(self.lib.fake_launch_grid(i, d) for d in range(3)), i)
                for i in range(self.lib.fake_launches())]

    def streams(self):
        """Streams that took launches since the last reset."""
        return {self.lib.fake_launch_stream(i) for i in range(self.lib.fake_launches())}

    def head(self, i, k):
        """Int k of launch i's first argument (task-graph kernels)."""
        return self.lib.fake_launch_head(i, k)


_fake = None


def load(tmp):
    """Link the library's objects with the test runtime (once a process)."""
    global _fake
    if _fake is None:
        from paper_2605_06392_gb300 import build
        build.build()
        objs = [os.path.join(build.OUT, os.path.basename(s)[:-3] + ".o")
                for s in build._sources()]
        cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
        so = os.path.join(str(tmp), "libbta_fake.so")
        subprocess.run([shutil.which("g++"), "-shared", "-fPIC", "-O1", "-std=c++17",
                        "-I", os.path.join(cuda, "include"), os.path.join(HERE, "runtime.cpp"),
                        *objs, "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", so], check=True)
        _fake = FakeCuda(so)
    return _fake
