"""The one-kernel branch-and-bound (direct.cu) equals the plain sweep bit for
bit: single fits at the edges of its launch shapes, batches at the edges of
its sort and table sizes, and data that its interval test cannot prune early
(lattices, few columns, near-vertical clusters, duplicate points, the full
int16 range, no outliers), with several order statistics."""
import numpy as np
import pytest

from paper_1510_01041_gb300 import datagen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F = ("status", "w_num", "w_den", "s_num", "s_den", "t_num", "t_den", "i", "j", "theta1", "theta2", "med_sq")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_01041_gb300 import build, lms
    build.build()
    return lms


def cuda(x, y):
    return tuple(torch.from_numpy(np.ascontiguousarray(a, dtype=np.int16)).cuda() for a in (x, y))


def points(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "line":
        return datagen.line_with_outliers(n, seed, 0.4)
    if kind == "sloped":
        return datagen.sloped(n, seed, 0.45, 1.5)[:2]
    if kind == "pure":
        return datagen.sloped(n, seed, 0.0, 1.5)[:2]
    if kind == "random":
        return datagen.line_with_outliers(n, seed, 1.0)
    if kind == "full":
        return rng.integers(-32768, 32768, n), rng.integers(-32768, 32768, n)
    if kind == "columns":
        return rng.integers(0, 3, n), rng.integers(-30000, 30000, n)
    if kind == "vertical":
        return np.where(rng.random(n) < 0.6, rng.integers(-2, 3, n), rng.integers(-9000, 9000, n)), \
            rng.integers(-16000, 16000, n)
    if kind == "lattice":
        return rng.integers(-20, 20, n), rng.integers(-20, 20, n)
    if kind == "equal_x":
        return np.full(n, 7), rng.integers(-500, 500, n)
    assert kind == "duplicates"
    same = rng.random(n) < 0.7
    return np.where(same, 5, rng.integers(-300, 300, n)), np.where(same, -8, rng.integers(-300, 300, n))


KINDS = ("line", "sloped", "pure", "random", "full", "columns", "vertical", "lattice", "equal_x", "duplicates")


@pytest.mark.parametrize("kind", KINDS)
def test_single_equals_sweep(L, kind):
    for n, hf in ((513, 0), (1025, 0.75), (2048, 0), (2049, 0.3), (8193, 0)):
        x, y = cuda(*points(kind, n, n))
        h = int(hf * n)
        a = L.decode(L.fit(x, y, h))[0]
        b = L.decode(L.fit(x, y, h, "sweep"))[0]
        assert a == b, (kind, n, h, a, b)


@pytest.mark.parametrize("kind,n", [("line", 16384), ("sloped", 16385), ("random", 20000), ("pure", 32768)])
def test_large_equals_branch_and_bound(L, kind, n):
    """Without statistics fit_bnb is the one kernel; with them the staged branch-and-bound."""
    x, y = cuda(*points(kind, n, 3))
    a = L.decode(L.fit_bnb(x, y, stats=False)[0])[0]
    b = L.decode(L.fit_bnb(x, y)[0])[0]
    assert a == b, (kind, n, a, b)


def test_batch_equals_sweep(L):
    sizes = [257, 258, 300, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096]
    sets = [points(k, n, 11 * n + s) for s, k in enumerate(KINDS) for n in sizes if n <= 1025 or k in KINDS[:4]]
    off = np.zeros(len(sets) + 1, np.int64)
    off[1:] = np.cumsum([len(s[0]) for s in sets])
    X, Y = cuda(np.concatenate([s[0] for s in sets]), np.concatenate([s[1] for s in sets]))
    h = np.array([0 if k % 3 else max(2, 2 * len(s[0]) // 3) for k, s in enumerate(sets)], np.int32)
    plan = L.BatchPlan(off, h)
    res = L.decode(plan.fit(X, Y, torch.from_numpy(off).cuda()))
    for k, r in enumerate(res):
        a, b = int(off[k]), int(off[k + 1])
        want = L.decode(L.fit(X[a:b], Y[a:b], int(h[k]), "sweep"))[0]
        assert tuple(r[f] for f in F) == tuple(want[f] for f in F), (k, b - a, r, want)
        assert r["algorithm"] == L.ALGOS["bnb" if b - a >= 512 else "sweep"]


@pytest.mark.parametrize("n", [15, 16, 17, 64, 511, 2048, 2049, 4096, 4097])
def test_float_equals_sweep(L, n):
    """The float form (grid points, scores in double) finds the sweep's line: the same pair, and a width that
    differs by the rounding of double projections only (2^-53 of their size, at most 1e-9 of the width here)."""
    rng = np.random.default_rng(n)
    cases = [datagen.gaussian_f32(n, n, f) for f in (0.4, 0.0, 1.0)]
    cases += [(rng.standard_cauchy(n), rng.standard_cauchy(n)), (np.full(n, 3.0), rng.normal(size=n)),
              (3 + 1e-6 * rng.normal(size=n), rng.normal(size=n)),
              (rng.normal(size=n) * 1e-9, rng.normal(size=n) * 1e9),
              (np.append(rng.normal(size=n - 1), np.inf), rng.normal(size=n))]
    for k, (x, y) in enumerate(cases):
        X, Y = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda() for a in (x, y))
        for h in (0, int(0.75 * n)):
            a, b = L.decode(L.fit(X, Y, h))[0], L.decode(L.fit(X, Y, h, "sweep"))[0]
            assert a["status"] == b["status"] and a["algorithm"] == b["algorithm"], (k, n, h, a, b)
            if a["status"] == 0:
                assert (a["i"], a["j"], a["theta1"]) == (b["i"], b["j"], b["theta1"]), (k, n, h, a, b)
                assert a["med_sq"] == pytest.approx(b["med_sq"], rel=1e-9), (k, n, h, a, b)
