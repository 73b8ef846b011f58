"""The one-kernel branch-and-bound (direct.cuh) built for the host: the
kernel's own code run by one thread (direct_host.h), with counters of its
phases, on sets of any form, without a GPU.  Barriers and races are not
covered; answers, give-ups, loops and the amount of work are."""
import ctypes
import os
import re
import subprocess

import numpy as np

from paper_1510_01041_gb300 import lms

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1510_01041_gb300", "csrc")
MODES = ("tree", "pairs", "event", "exact", "candidates")

ENTRY = """
template <bool F> static void host_fit(DirectArgs &a, int HC, int PM, int LRUN, float leaf)
{
    TeamShape s;
    s.PM = PM; s.LC = LRUN + PM; s.HC = HC; s.Q = min(PM, 128) - 1; s.leaf = leaf;
    s.ptsn = 0; s.dupw = 2048; s.sortw = 16LL * 65536; s.C = 1;
    a.nsets = 1;
    a.algo = LMS_ALGO_SWEEP;
    a.bnb_min = 0x7fffffff;
    a.shape = s;
    std::vector<long long> mem(team_bytes(s) / 8 + 64);
    a.mem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(mem.data()) + 255) & ~(uintptr_t)255);
    memset(host_count, 0, sizeof host_count);
    if (PM == 256) k_direct<1, 1, 1024, 4096, 256, 64, true, F>(a);
    else k_direct<1, 1, 1024, 1024, 64, 32, true, F>(a);
}
extern "C" void host_i16(const short *x, const short *y, int n, int h, int batch, lms_result *out, long long *count)
{
    DirectArgs a = {};
    a.x = x; a.y = y; a.n = n; a.h = h; a.out = out;
    int done = -1;
    if (batch == 2) { a.set_done = &done; a.small_max = n; }
    if (batch) host_fit<false>(a, 2048, 64, 32, 256.0f);
    else host_fit<false>(a, 4096, 256, 64, 256.0f);
    host_count[0][7] = done;
    memcpy(count, host_count, sizeof host_count);
}
extern "C" int host_f32(const float *x, const float *y, int n, int h, lms_result *out, long long *count)
{
    int done = 0;
    DirectArgs a = {};
    a.xf = x; a.yf = y; a.n = n; a.h = h; a.out = out; a.done = &done;
    host_fit<true>(a, n <= 2048 ? 4096 : 16384, 256, 64, 256.0f);
    memcpy(count, host_count, sizeof host_count);
    return done;
}
"""


def source():
    common = open(os.path.join(CSRC, "common.cuh")).read()
    a, b = common.index("// Ascending bitonic sort of P = IPT"), common.index("// A range's start order (global")
    common = common[:a] + common[b:]          # its sorting helpers: direct_host.h has them
    direct = open(os.path.join(CSRC, "direct.cuh")).read()
    direct = direct[:direct.index("// ------------------------------------------------------------------ host\n")]
    for name, body in (("unsigned cluster_ctas()", "return 1;"), ("unsigned cluster_rank()", "return 0;"),
                       ("unsigned smem_size()", "return sizeof(dsm);"), ("void cluster_meet()", ""),
                       ("void group_meet(int id)", "")):
        i = direct.index(name)
        j, k = direct.index("{", i), direct.index("\n}", i)
        direct = direct[:j] + "{" + body + direct[k:]
    direct = direct.replace("    extern __shared__ __align__(16) unsigned char dsm[];\n", "")
    text = common + direct
    text = re.sub(r"#include.*\n|#pragma once\n", "", text)
    return ('#include "direct_host.h"\n#include "lms.h"\n'
            "static unsigned char dsm[1 << 20] __attribute__((aligned(16)));\n" + text + "}\n}\nusing namespace lms;\nusing namespace lms::direct;\n"
            + ENTRY)


class Direct:
    def __init__(self, path):
        self.lib = ctypes.CDLL(path)

    def _run(self, f, x, y, h, *extra):
        rec = np.zeros(1, lms.RESULT_DTYPE)
        count = np.zeros((2, 8), np.int64)
        p = [ctypes.c_void_p(a.ctypes.data) for a in (x, y, rec, count)]
        done = f(p[0], p[1], x.size, h or x.size // 2 + 1, *extra, p[2], p[3])
        calls = dict(zip(MODES, count[0].tolist()))
        calls["phases"] = sum(calls[m] for m in MODES[:4])
        calls["done"] = int(count[0, 7])
        calls.update({m + "_sum": v for m, v in zip(MODES, count[1].tolist())})
        return done, rec[0], calls

    def i16(self, x, y, h=0, batch=0):
        """The record and the counters of one fit: in the shape of small single fits (batch 0), of a batch's sets (1), of
        its small sets, which may be left to the plain kernel (2; then calls["done"] is 0)."""
        x, y = (np.ascontiguousarray(v, dtype=np.int16) for v in (x, y))
        return self._run(self.lib.host_i16, x, y, h, int(batch))[1:]

    def f32(self, x, y, h=0):
        """Whether the attempt finished, its record and its counters."""
        x, y = (np.ascontiguousarray(v, dtype=np.float32) for v in (x, y))
        return self._run(self.lib.host_f32, x, y, h)


def load(folder):
    src, lib = os.path.join(str(folder), "direct_host.cpp"), os.path.join(str(folder), "libdirect_host.so")
    with open(src, "w") as f:
        f.write(source())
    subprocess.run(["g++", "-std=c++17", "-O2", "-w", "-shared", "-fPIC", "-fno-strict-aliasing", "-I", HERE, "-I",
                    os.path.join(ROOT, "include"), "-o", lib, src], check=True)
    return Direct(lib)
