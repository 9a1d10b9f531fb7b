"""The library's host code (plans, routing, device memory) compiled by g++ over a fake CUDA runtime
(tests/host/fake_cuda.cpp): what a plan decides and what it asks of the runtime can be tested without a GPU."""
from __future__ import annotations

import ctypes
import os
import shutil
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1812_00904_gb300", "csrc")
CSC, CSR = 0, 1
F64, F32, BF16, F16 = 0, 1, 2, 3


def cuda_include() -> str:
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


class HostLib:
    def __init__(self, directory: str):
        path = os.path.join(directory, "libhost.so")
        srcs = [os.path.join(HERE, "host", "fake_cuda.cpp"), *(os.path.join(CSRC, f) for f in ("api.cu", "devmem.cu"))]
        # (-Bsymbolic: the fake runtime, also where a real one is loaded)
        subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-fPIC", "-shared", "-Wl,--no-undefined", "-Wl,-Bsymbolic", "-I", cuda_include(), "-x", "c++",
                        *srcs, "-lpthread", "-o", path], check=True)
        self.lib = ctypes.CDLL(path)
        self.lib.fake_log.restype = ctypes.c_char_p
        self.lib.fake_alloc.restype = ctypes.c_void_p
        self.lib.fake_alloc.argtypes = [ctypes.c_size_t]
        self.lib.fake_used.restype = ctypes.c_uint64
        self.lib.fake_room.argtypes = [ctypes.c_uint64]
        self.lib.spmv_plan_destroy.argtypes = [ctypes.c_void_p]
        self.lib.spmv_plan_ex.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int64, ctypes.c_int64, ctypes.c_int32,
                                          ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int32,
                                          ctypes.c_int32, ctypes.c_void_p, ctypes.c_uint32, ctypes.c_void_p]
        for name, vectors in (("spmv", 2), ("spvtm", 2), ("spmv_pair", 4), ("spmv_dvalues", 3)):
            getattr(self.lib, name).argtypes = [ctypes.c_void_p] * (vectors + 2)
        self.lib.spmv_batch.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32, ctypes.c_void_p, ctypes.c_int64,
                                        ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p]
        self.lib.spmv_last_error.restype = ctypes.c_char_p
        self.reset()

    def reset(self, sms=152, optin=232448):
        self.lib.fake_reset(sms, optin)

    def log(self):
        return self.lib.fake_log().decode().split("\n")[:-1]

    def device(self, d=None):
        if d is not None:
            self.lib.cudaSetDevice(d)
        cur = ctypes.c_int()
        self.lib.cudaGetDevice(ctypes.byref(cur))
        return cur.value

    def plan(self, n_minor, n_major, nnz, val=F32, flags=0, opts=None, ptr=None):
        """A CSC plan of nnz nonzeros spread evenly over n_major columns (or as ptr says)."""
        if ptr is None:
            ptr = (np.arange(n_major + 1, dtype=np.int64) * nnz // n_major).astype(np.int32)
        p = self.lib.fake_alloc(4 * len(ptr))
        ctypes.memmove(p, np.ascontiguousarray(ptr, dtype=np.int32).ctypes.data, 4 * len(ptr))
        out = ctypes.c_void_p()
        st = self.lib.spmv_plan_ex(ctypes.byref(out), n_minor, n_major, nnz, CSC, p, 0x10000, 0x20000, val,
                                   F64 if val == F64 else F32, None, flags, opts)
        assert st == 0, self.lib.spmv_last_error().decode()
        return out

    def launches(self, plan, call, *extra):
        """The kernels that a call on device vectors launches: [(name, warps of a CTA, CTAs)]."""
        self.log()
        vectors = {"spmv": 2, "spvtm": 2, "spmv_pair": 4, "spmv_dvalues": 3}
        if call == "batch":
            op, k, ld_in, ld_out = extra
            st = self.lib.spmv_batch(plan, op, k, 0x100000, ld_in, 0x200000, ld_out, None)
        else:
            st = getattr(self.lib, call)(plan, *(0x100000 * (i + 1) for i in range(vectors[call])), None)
        assert st == 0, self.lib.spmv_last_error().decode()
        return [(" ".join(w[:-2]), int(w[-2]), int(w[-1])) for w in (line.split() for line in self.log())
                if len(w) > 2 and w[-1].isdigit() and w[-2].isdigit()]

    def close(self, plan):
        self.lib.spmv_plan_destroy(plan)
