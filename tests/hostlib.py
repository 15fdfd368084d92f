"""The library's host code on a CUDA runtime without a GPU (fake_cudart.cpp):
what it launches, copies and orders, from its log."""
import ctypes
import glob
import importlib
import mmap
import os
import shutil
import subprocess

import inputs
from paper_1908_08557_gb300 import binding

build = importlib.import_module("paper_1908_08557_gb300.build")  # the package's name `build` is its function
CUDA = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
STREAM = 0x77  # the caller's stream


class HostLib:
    def __init__(self, tmp):
        objs = lambda: sorted(glob.glob(os.path.join(build.BUILD, "*.o")))  # noqa: E731
        build.build()
        if len(objs()) != len(build.sources()):
            build.build(force=True)
        so = os.path.join(str(tmp), "libmhd_host.so")
        fake = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fake_cudart.cpp")
        r = subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(CUDA, "include"),
                            fake] + objs() + ["-o", so], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        self.lib = ctypes.CDLL(so)
        self.lib.fake_log.restype = ctypes.c_char_p
        for f in ("mhd_workspace_bytes", "mhd_gran_workspace_bytes", "mhd_tape_bytes"):
            getattr(self.lib, f).restype = ctypes.c_size_t
        self.lib.mhd_last_error.restype = ctypes.c_char_p
        self.keep = []

    def log(self):
        return [ln.split() for ln in self.lib.fake_log().decode().splitlines()]

    def clear(self):
        self.lib.fake_clear()

    def memory(self, nbytes, foreign=False):
        """Zeroed "device" memory, 256-byte aligned; pages are taken when touched."""
        m = mmap.mmap(-1, nbytes + 256, flags=mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS | 0x4000)  # MAP_NORESERVE
        self.keep.append(m)
        p = (ctypes.addressof(ctypes.c_char.from_buffer(m)) + 255) // 256 * 256
        if foreign:
            self.lib.fake_foreign(ctypes.c_void_p(p), ctypes.c_size_t(nbytes))
        return p

    def handle(self, nx, ny, nz, precision, adjoint=False, **over):
        p = inputs.scheme_params(nx, ny, nz, **over)
        q = binding.make_params(p, precision, adjoint=adjoint)
        n = self.lib.mhd_workspace_bytes(ctypes.byref(q))
        assert n
        state = self.memory(8 * nx * ny * nz * precision // 8)
        lr = (ctypes.c_double * (nz + 6))()
        h = ctypes.c_void_p()
        rc = self.lib.mhd_create(ctypes.byref(q), ctypes.c_void_p(self.memory(n)), ctypes.c_size_t(n),
                                 ctypes.c_void_p(state), 0, lr, lr, ctypes.c_void_p(STREAM), ctypes.byref(h))
        assert rc == 0, self.lib.mhd_last_error(None)
        self.keep.append(q)
        return h

    def ok(self, rc, h):
        assert rc == 0, self.lib.mhd_last_error(h)
