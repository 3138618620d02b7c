"""The library's host code on the CPU: its objects linked against the runtime
of fake_cuda.cpp (device memory is host memory, kernels are counted)."""
import ctypes
import os
import subprocess

import numpy as np

import paper_2607_20211_gb300 as drsf

HERE = os.path.dirname(os.path.abspath(__file__))
_lib = None


def load(tmp):
    """The library over the fake runtime (built once per session, in `tmp`)."""
    global _lib
    if _lib is not None:
        return _lib
    bld = drsf._build_mod
    drsf.build()
    objs = [os.path.join(bld.BUILD, os.path.basename(src)[:-3] + ".o") for src in bld.sources()]
    if not all(map(os.path.exists, objs)):
        drsf.build(force=True)
    out = os.path.join(str(tmp), "libdrsf_fake.so")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(bld._nvcc())))
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-O1", "-fvisibility=hidden", "-Wl,-Bsymbolic",
                    "-I", os.path.join(cuda, "include"), os.path.join(HERE, "fake_cuda.cpp"),
                    *objs, "-o", out], check=True)
    lib = ctypes.CDLL(out)
    vp, i32, i64, u32 = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64, ctypes.c_uint32
    lib.drsf_create.argtypes = [i32, vp, i64, vp, u32, vp, ctypes.POINTER(ctypes.c_void_p)]
    for name in ("drsf_apply", "drsf_apply_host"):
        getattr(lib, name).argtypes = [vp, ctypes.c_int, vp, i64, vp]
    lib.drsf_apply_grouped.argtypes = [vp, ctypes.c_int, vp, i64, i32, vp, vp, vp]
    lib.drsf_apply_batched.argtypes = [vp, ctypes.c_int, vp, i64, i32, vp, vp, vp, i32, vp]
    lib.drsf_reserve.argtypes = [vp, i64, vp]
    lib.drsf_sync.argtypes = [vp, vp]
    lib.drsf_destroy.argtypes = [vp]
    lib.fake_capture.argtypes = [vp]
    lib.fake_room.argtypes = [i64]
    lib.fake_launches.argtypes = [ctypes.c_char_p]
    for name in ("waits", "pinned", "forbidden", "recorded_copies", "held", "launches"):
        getattr(lib, "fake_" + name).restype = i64
    _lib = lib
    return lib


class Handle:
    """A handle over `n` vertices and no edges, on stream 77."""
    STREAM = 77

    def __init__(self, lib, n=1000):
        self.lib, self.n = lib, n
        self.parent = np.arange(n, dtype=np.int32)
        h = ctypes.c_void_p()
        assert lib.drsf_create(n, None, 0, self.parent.ctypes.data, 0, self.STREAM, ctypes.byref(h)) == drsf.OK
        self.h = h

    def batch(self, k):
        self.b = np.zeros((max(k, 1), 2), np.int32)
        return self.b.ctypes.data

    def apply(self, op, k, host=False):
        f = self.lib.drsf_apply_host if host else self.lib.drsf_apply
        return f(self.h, op, self.batch(k), k, self.STREAM)

    def grouped(self, op, k, graphs=2):
        vo = np.linspace(0, self.n, graphs + 1).astype(np.int64)
        bo = np.linspace(0, k, graphs + 1).astype(np.int64)
        return self.lib.drsf_apply_grouped(self.h, op, self.batch(k), k, graphs, vo.ctypes.data, bo.ctypes.data,
                                           self.STREAM)

    def batched(self, op, k, graphs=2):
        vo = np.linspace(0, self.n, graphs + 1).astype(np.int64)
        bo = np.linspace(0, k, graphs + 1).astype(np.int64)
        cl = (drsf.BatchedClass * 1)(drsf.BatchedClass(2 ** 31 - 1, 256, 0, 1))
        return self.lib.drsf_apply_batched(self.h, op, self.batch(k), k, graphs, vo.ctypes.data, bo.ctypes.data,
                                           ctypes.cast(cl, ctypes.c_void_p), 1, self.STREAM)

    def close(self):
        self.lib.fake_capture(None)
        self.lib.fake_room(-1)
        self.lib.drsf_destroy(self.h)
