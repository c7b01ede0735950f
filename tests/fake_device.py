"""The library on two pretended GPUs: its objects linked with tests/fake_cudart.cpp, called through ctypes."""
import ctypes as C
import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build(directory):
    from paper_2410_03462_b200 import build as lib_build
    lib_build.build()
    objs = [os.path.join(lib_build.HERE, "_build", s.replace(".cu", ".o")) for s in lib_build.SOURCES]
    newest = max(os.path.getmtime(os.path.join(lib_build.CSRC, f)) for f in os.listdir(lib_build.CSRC))
    if any(not os.path.exists(o) or os.path.getmtime(o) < newest for o in objs):
        lib_build.build(force=True)
    so = os.path.join(str(directory), "libgrf_host.so")
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                           "-I", lib_build.INCLUDE, "-I", lib_build.CSRC, os.path.join(ROOT, "tests", "fake_cudart.cpp"),
                           *objs, "-ldl", "-o", so])
    return so


class Fake:
    """Sizes that the kernels report are set with `report`; NNZ etc. index them."""
    INVALID, NOMEM, TOO_LARGE = -1, -5, -2
    PHI, PSI, DEP_PHI, DEP_PSI, EDGES, PLAN, KEYS, POSITIONS, LONGEST = range(9)

    def __init__(self, so):
        self.lib = C.CDLL(so)
        for name in ("fake_stream", "fake_denominators", "fake_live"):
            getattr(self.lib, name).restype = C.c_size_t if name == "fake_live" else C.c_void_p
        self.lib.fake_capture.argtypes = [C.c_void_p]
        self.lib.fake_log.restype = C.c_char_p
        self.lib.fake_limit.argtypes = [C.c_int, C.c_size_t]
        self.lib.fake_report.argtypes = [C.c_int, C.c_int64]
        self.lib.grf_attn_workspace_bytes.restype = C.c_size_t
        self.lib.fake_reset()

    def report(self, **sizes):
        for name, value in sizes.items():
            self.lib.fake_report(getattr(self, name), value)

    def errors(self):
        return self.lib.fake_errors()

    def log(self):
        return [self.lib.fake_log(i).decode() for i in range(self.lib.fake_log_size())]

    def launched(self, kernel):
        return sum(kernel in x for x in self.log() if x.startswith("launch"))

    def context(self, device=0, stream=None):
        h = C.c_void_p()
        assert self.lib.grf_ctx_create(C.byref(h), device, C.c_void_p(stream)) == 0
        return h

    def sample(self, ctx, N, feat=None, walks=32, length=12):
        """A sample of a graph whose arrays nobody reads; returns (code, object)."""
        h = feat if feat is not None else C.c_void_p()
        f = np.ones(length + 1, np.float32).ctypes.data_as(C.POINTER(C.c_float))
        some = C.c_void_p(4096)
        rc = self.lib.grf_sample(ctx, N, some, some, some, C.c_uint64(1), walks, C.c_float(0.1), length, f, None, C.byref(h))
        return rc, h

    def nnz(self, feat, which=0):
        """(code, non-zeros)"""
        n = C.c_int64(-1)
        return self.lib.grf_features_view(feat, which, None, None, C.byref(n), None, None, None), n.value

    def linear(self, ctx, feat, G, N, m, d, dtype, workspace=None):
        """grf_masked_linear_attn on arrays that nobody reads, with a workspace for one problem if not stated."""
        code = 1 if dtype == "bf16" else 0
        need = workspace or self.lib.grf_attn_workspace_bytes(1, N, m, d, code)
        some = C.c_void_p(4096)
        return self.lib.grf_masked_linear_attn(ctx, feat, G, N, m, d, code, some, some, some, some, None, some,
                                               C.c_size_t(need))

    def step_host(self, ctx, N, G, m, d, walks=32, length=12):
        """grf_step_host in bf16 on a ring of N nodes."""
        rowptr = np.arange(0, 2 * N + 1, 2, dtype=np.int32)
        col = np.stack([np.arange(N) - 1, np.arange(N) + 1], 1).astype(np.int32).ravel() % N
        w = np.full(2 * N, 0.25, np.float32)
        f = np.ones(length + 1, np.float32)
        q, v = np.zeros(G * N * m, np.uint16), np.zeros(G * N * d, np.uint16)
        out = np.zeros_like(v)
        p = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
        return self.lib.grf_step_host(ctx, N, p(rowptr), p(col), p(w), C.c_uint64(1), walks, C.c_float(0.1), length, p(f), None,
                                      G, m, d, 1, p(q), p(q), p(v), p(out))
