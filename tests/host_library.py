"""The library's own host code over fake_cudart.cpp: which kernels a call
launches, which workspace it asks for and what it returns when a CUDA call
fails, without a GPU.  Kernels do not run, so records are not looked at."""
import ctypes
import glob
import os
import subprocess

import numpy as np

from paper_1510_01041_gb300 import build, lms

HERE = os.path.dirname(os.path.abspath(__file__))


class Host:
    def __init__(self, path):
        self.lib = ctypes.CDLL(path)
        self.lib.fake_launch_name.restype = ctypes.c_char_p
        for f in ("fake_frees", "fake_held", "fake_limit"):
            getattr(self.lib, f).restype = ctypes.c_longlong
        self.lib.lms_workspace_size.restype = ctypes.c_size_t
        self.lib.lms_workspace_size.argtypes = [ctypes.c_int64, ctypes.c_int32, ctypes.c_void_p]
        self.x = np.arange(65536, dtype=np.int64).astype(np.int16)
        self.xf = self.x.astype(np.float32)
        self.rec = np.zeros(4096, lms.RESULT_DTYPE)
        self.stats = np.zeros(64, np.int64)

    def set(self, knob, v):
        self.lib.fake_set(knob.encode(), ctypes.c_longlong(v))

    def kernels(self):
        """Names of the kernels launched since the last call."""
        names = [self.lib.fake_launch_name(k).decode() for k in range(self.lib.fake_launches())]
        self.lib.fake_clear()
        return names

    @staticmethod
    def _opt(algorithm, sweepers=0, buckets=0, seed_mode="quantiles"):
        return lms.options(algorithm, sweepers, buckets, seed_mode)

    def fit(self, n, h=0, algorithm="auto", dtype=lms.LMS_I16, host=False, **opt):
        o = self._opt(algorithm, **opt)
        p = ctypes.c_void_p((self.x if dtype == lms.LMS_I16 else self.xf).ctypes.data)
        f = self.lib.lms_fit_host if host else self.lib.lms_fit
        return f(p, p, ctypes.c_int64(n), ctypes.c_int64(h), dtype, ctypes.byref(o),
                 ctypes.c_void_p(self.rec.ctypes.data), None)

    def fit_bnb(self, n, h=0, stats=False, **opt):
        o = self._opt("bnb", **opt)
        p = ctypes.c_void_p(self.x.ctypes.data)
        return self.lib.lms_fit_bnb(p, p, ctypes.c_int64(n), ctypes.c_int64(h), None, ctypes.byref(o),
                                    ctypes.c_void_p(self.rec.ctypes.data),
                                    ctypes.c_void_p(self.stats.ctypes.data) if stats else None, None)

    def workspace_size(self, n, dtype=lms.LMS_I16, algorithm="auto", **opt):
        o = self._opt(algorithm, **opt)
        return self.lib.lms_workspace_size(n, dtype, ctypes.byref(o))

    def set_workspace(self, p, size):
        return self.lib.lms_set_workspace(p, ctypes.c_size_t(size))

    def plan(self, sizes, h=None, plain_max_n=0, streams=0, bnb_min_n=0):
        off = np.zeros(len(sizes) + 1, np.int64)
        off[1:] = np.cumsum(sizes)
        hh = None if h is None else np.ascontiguousarray(h, np.int32)
        handle = ctypes.c_void_p()
        rc = self.lib.lms_batch_plan_create_ex(ctypes.c_void_p(off.ctypes.data), ctypes.c_int64(len(sizes)),
                                               ctypes.c_void_p(hh.ctypes.data) if hh is not None else None,
                                               plain_max_n, streams, bnb_min_n, ctypes.byref(handle))
        return rc, handle, off

    def fit_batched(self, plan, off):
        p = ctypes.c_void_p(self.x.ctypes.data)
        return self.lib.lms_fit_batched(plan, p, p, ctypes.c_void_p(off.ctypes.data),
                                        ctypes.c_void_p(self.rec.ctypes.data), None)


def load(folder):
    """Links the built objects to the stand-in runtime (bound to itself: another runtime may be loaded); a fresh library
    with its own state in `folder`."""
    build.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    path = os.path.join(str(folder), "liblms_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"), "-o", path,
                    os.path.join(HERE, "fake_cudart.cpp"), *sorted(glob.glob(os.path.join(build.OUT, "*.o")))],
                   check=True)
    return Host(path)
