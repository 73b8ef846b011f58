"""The one-kernel branch-and-bound at the edges of its dispatch: the largest
set, small sets by fit_bnb, order statistics around its limit, sets of a
batch on both sides of every rule, forms where slopes or widths repeat, float
coordinates with ties and far from the origin, and graphs captured before fits
of the same size by other routes."""
import json
import os

import numpy as np
import pytest

from direct_sets import points
from paper_1510_01041_gb300 import datagen
from test_direct_host import best_line

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "lms_large.json")
F = ("status", "w_num", "w_den", "s_num", "s_den", "t_num", "t_den", "i", "j", "theta1", "theta2", "med_sq")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_01041_gb300 import build, lms
    build.build()
    return lms


def cuda(x, y, dtype=np.int16):
    return tuple(torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).cuda() for a in (x, y))


def rec(L, out):
    r = L.decode(out)[0]
    return tuple(r[k] for k in F)


# ---------------------------------------------------------------- captured graphs
@pytest.mark.parametrize("n", [2048, 8192])
def test_graph_replays_after_other_routes(L, n):
    """A fit captured in a graph, then fits of the same n with statistics, by the sweep and with a small order
    statistic: none of them moves the workspace, and the graph replays on new points."""
    x, y = cuda(*points("sloped", n, 1))
    small = cuda(*points("sloped", 600, 1))   # every route once: the kernels' own memory is allocated
    for run in (lambda a, b: L.fit_bnb(a, b, stats=True), lambda a, b: L.fit_bnb(a, b, 37, stats=False), L.fit,
                lambda a, b: L.fit(a, b, 0, "sweep"), lambda a, b: L.fit(a, b, 37)):
        run(*small)
    torch.cuda.synchronize()
    out = torch.zeros(L.RESULT_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    L.fit_bnb(x, y, stats=False, out=out)
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            L.fit_bnb(x, y, stats=False, out=out, stream=s)
    held = torch.cuda.mem_get_info()[0]
    L.fit_bnb(x, y, stats=True)
    L.fit_bnb(x, y, n // 16, stats=False)
    L.fit(x, y)
    L.fit(x, y, 0, "sweep")
    L.fit(x, y, n // 16)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == held
    x2, y2 = cuda(*points("line", n, 2))
    x.copy_(x2)
    y.copy_(y2)
    g.replay()
    torch.cuda.synchronize()
    assert rec(L, out) == rec(L, L.fit(x2, y2, 0, "sweep"))


# ---------------------------------------------------------------- single int16 fits
def test_largest_set_equals_oracle(L):
    with open(GOLDEN) as f:
        case = json.load(f)["cases"]["sloped_n65536_s65"]
    x, y = cuda(*datagen.sloped(case["n"], case["seed"], case["outlier_frac"])[:2])
    want = tuple(case[k] for k in F)
    assert rec(L, L.fit(x, y)) == want
    assert rec(L, L.fit_bnb(x, y, stats=False)[0]) == want
    assert rec(L, L.pretrained().fit(x, y, stats=False)[0]) == want


@pytest.mark.parametrize("kind", ["full", "columns", "rows", "vertical", "lattice", "collinear", "two_lines",
                                  "duplicates", "equal_x"])
def test_points_in_global_memory(L, kind):
    """Above 16384 points: the forms of test_gpu_direct and more against the staged branch-and-bound."""
    x, y = cuda(*points(kind, 17000, 5))
    for h in (0, 12750):
        assert rec(L, L.fit_bnb(x, y, h, stats=False)[0]) == rec(L, L.fit_bnb(x, y, h)[0]), h


@pytest.mark.parametrize("kind", ["line", "full", "vertical", "lattice", "duplicates", "digital"])
def test_small_sets_and_seeds_equal_oracle(L, orc, kind):
    for n in (2, 3, 17, 64, 300, 512):
        x, y = points(kind, n, 7 * n)
        x, y = x.astype(np.int16), y.astype(np.int16)
        X, Y = cuda(x, y)
        for h in sorted({n // 8, n // 8 + 1, n // 2 + 1, int(0.75 * n) + 1, n} & set(range(1, n + 1))):
            o = orc.lms_i16(x, y, h, "brute" if n <= 160 else "sweep")
            for seed in (None, 0.7, -40.0):
                sd = None if seed is None else torch.tensor([seed], dtype=torch.float32, device="cuda")
                got = rec(L, L.fit_bnb(X, Y, h, sd, stats=False)[0])
                assert got == tuple(getattr(o, k) for k in F), (kind, n, h, seed, got, o)


@pytest.mark.parametrize("kind", ["line", "rows", "digital", "collinear", "two_lines", "vertical", "duplicates"])
def test_order_statistic_at_the_limits(L, kind):
    for n in (513, 2048, 2049):
        X, Y = cuda(*points(kind, n, n))
        for h in (n // 8, n // 8 + 1, n // 4, n // 4 + 1, n // 3, n // 3 + 1, n):
            assert rec(L, L.fit(X, Y, h)) == rec(L, L.fit(X, Y, h, "sweep")), (kind, n, h)


# ---------------------------------------------------------------- batches
@pytest.mark.parametrize("options", [{}, {"plain_max_n": 256}, {"bnb_min_n": -1}, {"bnb_min_n": 512, "streams": 3}])
def test_batch_rules_equal_sweep(L, options):
    """Sizes and order statistics on both sides of every rule, sets of more than 4096 points among them."""
    kinds = ("line", "random", "columns", "duplicates", "lattice", "two_lines")
    sizes = [64, 65, 96, 97, 128, 129, 160, 161, 200, 256, 257, 511, 512, 1024, 1025, 4096, 4097]
    sets, h = [], []
    for k, n in enumerate(sizes):
        for q, hh in enumerate((0, n // 8, n // 8 + 1, n // 4, n // 3 + 1, int(0.75 * n))):
            if n > 1025 and q > 2:
                continue
            sets.append(points(kinds[(k + q) % len(kinds)], n, 31 * n + q))
            h.append(hh)
    off = np.zeros(len(sets) + 1, np.int64)
    off[1:] = np.cumsum([len(s[0]) for s in sets])
    X, Y = cuda(np.concatenate([s[0] for s in sets]), np.concatenate([s[1] for s in sets]))
    plan = L.BatchPlan(off, np.array(h, np.int32), **options)
    res = L.decode(plan.fit(X, Y, torch.from_numpy(off).cuda()))
    for k, r in enumerate(res):
        a, b = int(off[k]), int(off[k + 1])
        assert tuple(r[f] for f in F) == rec(L, L.fit(X[a:b], Y[a:b], h[k], "sweep")), (k, b - a, h[k], options)


# ---------------------------------------------------------------- float sets
@pytest.mark.parametrize("kind", ["line", "columns", "rows", "lattice", "digital", "collinear", "two_lines", "vertical",
                                  "duplicates"])
def test_float_ties_equal_sweep_arithmetic(L, kind):
    """Integer coordinates as floats.  Where the one kernel finishes, its record is the first of all pair slopes with
    slopes and projections computed in double; the sweep, which may compute a window's two projections one event
    earlier or later, has the same width up to that rounding (2^-51 of the largest terms of a projection)."""
    for n in (16, 64, 160, 300):
        x, y = points(kind, n, 5 * n)
        X, Y = cuda(x, y, np.float32)
        for h in (0, int(0.75 * n)):
            a, b = L.decode(L.fit(X, Y, h))[0], L.decode(L.fit(X, Y, h, "sweep"))[0]
            w, s, t, pair = best_line(np.float32(x), np.float32(y), h)
            size = float(np.abs(y).max() + 2 * max(abs(s), abs(b["theta1"])) * np.abs(x).max())
            for r in (a, b):
                assert r["status"] == 0 and abs(2 * np.sqrt(r["med_sq"]) - w) <= 2.0 ** -50 * size, (n, h, r, w)


@pytest.mark.parametrize("kind", ["line", "rows", "digital", "collinear", "two_lines", "lattice"])
@pytest.mark.parametrize("n", [512, 2048, 2049, 4096])
def test_float_shared_slopes_equal_sweep(L, kind, n):
    x, y = points(kind, n, n)
    X, Y = cuda(x, y, np.float32)
    a, b = L.decode(L.fit(X, Y))[0], L.decode(L.fit(X, Y, 0, "sweep"))[0]
    size = float(np.abs(y).max() + 2 * max(abs(a["theta1"]), abs(b["theta1"])) * np.abs(x).max())
    assert a["status"] == b["status"] == 0
    assert abs(2 * np.sqrt(a["med_sq"]) - 2 * np.sqrt(b["med_sq"])) <= 2.0 ** -50 * size, (a, b)
    # the reported line attains the reported width
    res = np.sort(np.abs(np.float64(y) - a["theta1"] * np.float64(x) - a["theta2"]))[n // 2]
    assert abs(res - np.sqrt(a["med_sq"])) <= 2.0 ** -50 * size


@pytest.mark.parametrize("offset", [1e3, 1e5, 1e7])
def test_float_far_from_the_origin(L, offset):
    """The record of sets whose projections round by up to grid steps: the widths of both paths and of all pair slopes
    in double differ by that rounding alone."""
    rng = np.random.default_rng(int(offset))
    for n in (40, 150, 290):
        x, y = (np.float32(offset + 3 * rng.normal(size=n)) for _ in range(2))
        X, Y = cuda(x, y, np.float32)
        for h in (0, int(0.8 * n)):
            w = best_line(x, y, h)[0]
            for algorithm in ("auto", "sweep"):
                r = L.decode(L.fit(X, Y, h, algorithm))[0]
                size = float(np.abs(y).max() + 2 * abs(r["theta1"]) * np.abs(x).max())
                assert abs(2 * np.sqrt(r["med_sq"]) - w) <= 2.0 ** -50 * size, (n, h, algorithm, r, w)
