"""libgpm's host code on a stand-in CUDA runtime (fake_cudart.cpp): the
compiled objects of the library, linked against it into a library of their
own.  Kernels do nothing and every count is zero; what is checked is what the
host asks of the runtime, and what a failing call leaves behind."""
from __future__ import annotations

import ctypes
import glob
import os
import subprocess

import numpy as np

from paper_2212_04551_gb300 import build, gpm

HERE = os.path.dirname(os.path.abspath(__file__))


def link(folder) -> "FakeGpu":
    build.build()
    lib = os.path.join(str(folder), "libgpm_fake.so")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    # (-Bsymbolic: the stand-in's functions, whatever runtime the process has loaded)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cudart.cpp"), *sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o"))),
                    "-lpthread", "-o", lib], check=True, capture_output=True, text=True)
    return FakeGpu(lib)


class FakeGpu:
    def __init__(self, path):
        self.lib = ctypes.CDLL(path)
        for name, (res, args) in gpm.SIGNATURES.items():
            f = getattr(self.lib, name)
            f.restype, f.argtypes = res, args
        vp, ci, sz = ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t
        for name, res, args in [("fake_reset", None, []), ("fake_fail", None, [ctypes.c_char_p, ci]),
                                ("fake_failed", ci, []), ("fake_calls", ci, [ctypes.c_char_p]), ("fake_memory_limit", None, [sz]),
                                ("fake_memory_in_use", sz, []), ("fake_violations", ci, []),
                                ("fake_log", ctypes.c_char_p, []), ("fake_clear_log", None, []),
                                ("fake_on_event_record", None, [vp]), ("fake_stream", vp, [ci])]:
            f = getattr(self.lib, name)
            f.restype, f.argtypes = res, args
        self.lib.fake_reset()

    def log(self):
        """(kernel, blocks, threads, shared bytes) of every launch since the last call."""
        lines = self.lib.fake_log().decode().splitlines()
        self.lib.fake_clear_log()
        return [(x[0], *map(int, x[1:])) for x in (line.split() for line in lines)]

    def error(self):
        return (self.lib.gpm_last_error() or b"").decode()

    def graph(self, indptr, indices, stream=None, flags=gpm.GPM_SKIP_VALIDATE):
        indptr = np.ascontiguousarray(indptr, np.int32)
        indices = np.ascontiguousarray(indices, np.int32)
        out = ctypes.c_void_p()
        st = self.lib.gpm_graph_create(indptr.ctypes.data, indices.ctypes.data, len(indptr) - 1, flags, stream,
                                       ctypes.byref(out))
        assert st == gpm.GPM_OK, self.error()
        return out

    def batch(self, goff, indptr, indices, stream=None):
        goff, indptr, indices = (np.ascontiguousarray(x, np.int32) for x in (goff, indptr, indices))
        out = ctypes.c_void_p()
        st = self.lib.gpm_batch_create(goff.ctypes.data, indptr.ctypes.data, indices.ctypes.data, len(goff) - 1,
                                       gpm.GPM_SKIP_VALIDATE, stream, ctypes.byref(out))
        assert st == gpm.GPM_OK, self.error()
        return out

    def configure(self, g, batch=False, **kw):
        c = gpm.gpm_config(0, 0, 4, gpm.GPM_ORDER_DEGREE_DESC, 120000, 1, 50, 0, 0, 16, 1, 1, 85)
        for key, val in kw.items():
            setattr(c, key, val)
        st = (self.lib.gpm_batch_set_config if batch else self.lib.gpm_set_config)(g, ctypes.byref(c))
        assert st == gpm.GPM_OK, self.error()

    def motifs(self, g, k):
        counts = np.zeros(853, np.uint64)
        return self.lib.gpm_motif_count(g, k, counts.ctypes.data_as(gpm._u64p), len(counts))

    def cliques(self, g, k_lo, k_hi=None):
        counts = np.zeros(16, np.uint64)
        p = counts.ctypes.data_as(gpm._u64p)
        return self.lib.gpm_clique_count(g, k_lo, p) if k_hi is None else self.lib.gpm_clique_count_range(g, k_lo, k_hi, p)

    def batch_count(self, b, kc, km, graphs):
        c, m = np.zeros(graphs, np.uint64), np.zeros(graphs * 853, np.uint64)
        return self.lib.gpm_batch_count(b, kc, km, c.ctypes.data_as(gpm._u64p), m.ctypes.data_as(gpm._u64p))

    def autotune(self, b, kc, km):
        c, ms = gpm.gpm_config(), ctypes.c_double()
        assert self.lib.gpm_batch_autotune(b, kc, km, 1, ctypes.byref(c), ctypes.byref(ms)) == gpm.GPM_OK, self.error()
        return c
