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
// The distinct slopes of a leaf listed by `parts` CTAs, each with the points in another order (as their cells may have
// them): slope keys, or order words for float points.  Returns how many were listed, -1 if they did not fit.
static TeamMem list_memory(std::vector<long long> &keys, std::vector<unsigned> &den)
{
    TeamMem m = {};
    keys.resize(1 << 20);
    den.resize(1 << 20);
    m.lkey = keys.data();
    m.lden = den.data();
    return m;
}
extern "C" int host_list_i16(const int *pts, int n, long long A, long long B, int xr, int yr, int parts, long long *out)
{
    std::vector<long long> keys;
    std::vector<unsigned> den;
    TeamMem m = list_memory(keys, den);
    Box bx = {0, 0, -xr, xr, -yr, yr, 0};
    DNode lf = {A, B, 1, 0, 0.0f, 0};
    int nlist = 0, over = 0, warp[32];
    for (int part = 0; part < parts; ++part)
        if (!list_pairs<1>(pts + (long long)part * n, n, nullptr, lf, bx, 1024, dsm, warp, m, &nlist, &over, 1 << 20,
                           part, parts))
            return -1;
    memcpy(out, keys.data(), sizeof(long long) * nlist);
    return over ? -1 : nlist;
}
extern "C" int host_list_f32(const float *xy, int n, long long A, long long B, int parts, long long *out)
{
    std::vector<long long> keys;
    std::vector<unsigned> den;
    TeamMem m = list_memory(keys, den);
    int nlist = 0, over = 0, warp[32];
    for (int part = 0; part < parts; ++part) {
        const float *x = xy + 2LL * part * n, *y = x + n;
        FloatSet f{};
        Box bx;
        long long red[8];
        if (!float_box<1>(x, y, n, f, bx, red)) return -1;
        std::vector<int2> pts(n);
        for (int k = 0; k < n; ++k)
            pts[k] = make_int2(__double2int_rn((x[k] - f.xc) * f.sx), __double2int_rn((y[k] - f.yc) * f.sy));
        list_pairs_f32<1>(pts.data(), n, A, B, bx, f, 1024, dsm, warp, m, &nlist, &over, 1 << 20, part, parts);
    }
    memcpy(out, keys.data(), sizeof(long long) * nlist);
    return over ? -1 : nlist;
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

    def listed_i16(self, x, y, lo, hi, parts, seed=0):
        """Slope keys of a leaf [lo, hi) listed by `parts` CTAs with the points in another order each."""
        rng = np.random.default_rng(seed)
        order = [rng.permutation(x.size) for _ in range(parts)]
        pts = np.concatenate([(y[o].astype(np.int32) << 16) | (x[o].astype(np.int32) & 0xffff) for o in order])
        pts = np.ascontiguousarray(pts, np.int32)
        out = np.zeros(1 << 20, np.int64)
        n = self.lib.host_list_i16(ctypes.c_void_p(pts.ctypes.data), x.size, ctypes.c_int64(lo), ctypes.c_int64(hi),
                                   int(np.abs(x).max()), int(np.abs(y).max()), parts, ctypes.c_void_p(out.ctypes.data))
        assert n >= 0
        return set(out[:n].tolist())

    def listed_f32(self, x, y, lo, hi, parts, seed=0):
        """The same for float points and scaled slope keys: the slopes, as doubles.  Seed None: one order (cells of many
        points are shared by the points' indices, which are the same in every CTA)."""
        rng = np.random.default_rng(seed)
        order = [np.arange(x.size) if seed is None else rng.permutation(x.size) for _ in range(parts)]
        xy = np.concatenate([np.concatenate([np.float32(x[o]), np.float32(y[o])]) for o in order])
        out = np.zeros(1 << 20, np.int64)
        n = self.lib.host_list_f32(ctypes.c_void_p(xy.ctypes.data), x.size, ctypes.c_int64(lo), ctypes.c_int64(hi), parts,
                                   ctypes.c_void_p(out.ctypes.data))
        assert n >= 0
        w = out[:n]
        return set(np.where(w < 0, w ^ 0x7fffffffffffffff, w).view(np.float64).tolist())


def load(folder):
    src, lib = os.path.join(str(folder), "direct_host.cpp"), os.path.join(str(folder), "libdirect_host.so")
    with open(src, "w") as f:
        f.write(source())
    subprocess.run(["g++", "-std=c++17", "-O2", "-w", "-shared", "-fPIC", "-fno-strict-aliasing", "-I", HERE, "-I",
                    os.path.join(ROOT, "include"), "-o", lib, src], check=True)
    return Direct(lib)
