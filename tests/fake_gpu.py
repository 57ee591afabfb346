"""The library linked with fake_cudart.c: its host logic on a machine without a GPU, with failures at chosen calls."""
import ctypes
import importlib
import mmap
import os
import subprocess

import numpy as np

MAP_NORESERVE = 0x4000  # of Linux; not in the mmap module
HERE = os.path.dirname(os.path.abspath(__file__))


def load(B, directory):
    """The library on the fake runtime, built in `directory`; its functions take and return what B.lib's do."""
    build = importlib.import_module("paper_2112_02574_gb300.build")
    objdir = os.path.join(build.LIBDIR, "obj")
    objs = [os.path.join(objdir, os.path.basename(s) + ".o") for s in build._sources()]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    fake, lib = (os.path.join(directory, n) for n in ("fake_cudart.o", "libsc_fake.so"))
    for cmd in ([build.NVCC, "-Xcompiler", "-fPIC", "-c", os.path.join(HERE, "fake_cudart.c"), "-o", fake],
                [build.NVCC, *build.ARCH, "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", lib, *objs, fake]):
        subprocess.run(cmd, check=True, capture_output=True)
    L = ctypes.CDLL(lib)
    for n in B.declared_symbols():
        f, real = getattr(L, n), getattr(B.lib, n)
        f.restype, f.argtypes = real.restype, real.argtypes
    L.fake_call.restype = ctypes.c_char_p
    L.fake_fail.argtypes = [ctypes.c_char_p, ctypes.c_int]
    L.fake_reset()
    return L


def calls(L):
    """Names of the kernels launched (and "graph launch") since the last fake_reset."""
    return [L.fake_call(k).decode() for k in range(L.fake_calls())]


def buffer(nbytes):
    """"Device" memory, page aligned; pages that nothing touches take no memory."""
    m = mmap.mmap(-1, nbytes, flags=mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS | MAP_NORESERVE)
    v = np.frombuffer(m, dtype=np.uint8)
    return v, ctypes.c_void_p(v.ctypes.data)


class Context:
    """A context on the fake runtime; ws_bytes: the workspace handed to sc_create (the library's size by default)."""

    def __init__(self, L, params, ws_bytes=None):
        self.L, n = L, params.nx * params.ny * params.nz
        self.fields, f = buffer(16 * n)
        need = L.sc_workspace_bytes(ctypes.byref(params)) if ws_bytes is None else ws_bytes
        self.ws, w = buffer(need)
        self.ctx = ctypes.c_void_p()
        self.status = L.sc_create(ctypes.byref(params), f, ctypes.c_void_p(f.value + 8 * n), w, need, None,
                                  ctypes.byref(self.ctx))
        self.out = buffer(40 * n)

    def moments(self):
        n = self.fields.size // 16
        p = self.out[1].value
        return self.L.sc_moments(self.ctx, ctypes.c_void_p(p), ctypes.c_void_p(p + 8 * n), None)


class Batch:
    """A batch on the fake runtime."""

    def __init__(self, L, params, ws_bytes=None):
        self.L, n = L, len(params)
        arr = (type(params[0]) * n)(*params)
        self.keep = [buffer(16 * p.nx * p.ny * p.nz) for p in params]
        ptr = [(ctypes.c_void_p * n)(*(k[1].value for k in self.keep)) for _ in range(2)]
        need = L.sc_batch_workspace_bytes(n, arr) if ws_bytes is None else ws_bytes
        self.ws, w = buffer(need)
        self.handle = ctypes.c_void_p()
        self.status = L.sc_batch_create(n, arr, ptr[0], ptr[1], w, need, None, ctypes.byref(self.handle))

    def member(self, k):
        return ctypes.c_void_p(self.L.sc_batch_member(self.handle, k))
