"""The one-kernel branch-and-bound run on the host (direct_host.py): its
records equal the oracle's, and sets whose pairs share slopes or whose slopes
share widths take no more than a bounded amount of work."""
import numpy as np
import pytest

import direct_host
from direct_sets import points

EXACT = ("status", "w_num", "w_den", "s_num", "s_den", "t_num", "t_den", "i", "j")


@pytest.fixture(scope="module")
def D(tmp_path_factory):
    return direct_host.load(tmp_path_factory.mktemp("direct"))


@pytest.mark.parametrize("kind", ["line", "sloped", "pure", "random", "full", "columns", "rows", "vertical", "lattice",
                                  "digital", "collinear", "two_lines", "equal_x", "duplicates"])
def test_int16_equals_oracle(D, orc, kind):
    for n in (2, 3, 7, 33, 64, 65, 129, 300):
        x, y = points(kind, n, 3 * n)
        x, y = x.astype(np.int16), y.astype(np.int16)
        for h in sorted({1, 2, n // 8 + 1, n // 2 + 1, int(0.75 * n) + 1, n} & set(range(1, n + 1))):
            want = orc.lms_i16(x, y, h, "brute" if n <= 160 else "sweep")
            for batch in (0, 1):
                r, _ = D.i16(x, y, h, batch)
                assert tuple(int(r[k]) for k in EXACT) == tuple(want.exact()), (kind, n, h, batch, r, want)


@pytest.mark.parametrize("parts", [1, 2, 5, 8, 16])
def test_shared_leaf_loses_no_slope(D, parts):
    """CTAs that share a leaf list all its slopes between them, whatever the order of the points inside the cells, which
    differs between CTAs."""
    rng = np.random.default_rng(parts)
    for n in (40, 200, 700):
        x, y = rng.integers(-30000, 30001, n), rng.integers(-30000, 30001, n)
        i, j = np.triu_indices(n, 1)
        ok = x[i] != x[j]
        i, j = i[ok], j[ok]
        dx, dy = x[j] - x[i], y[j] - y[i]
        keys = ((np.where(dx < 0, -dy, dy).astype(object) << 32) // np.abs(dx)).astype(np.int64)
        lo, hi = np.sort(keys)[[keys.size // 2, keys.size // 2 + 300]].tolist()
        want = set(keys[(keys >= lo) & (keys < hi)].tolist())
        for seed in range(4):
            assert D.listed_i16(x, y, lo, hi, parts, seed) == want, (n, seed)
        # float points (the frame scales both axes by powers of two); then half of them on one line, in one cell
        for line in (False, True):
            xf, yf = np.float32(x + rng.random(n)), np.float32(y + rng.random(n))
            if line:
                yf[: n // 2] = np.float32(-0.75) * xf[: n // 2]
            s = np.subtract(yf[j], yf[i], dtype=np.float64) / np.subtract(xf[j], xf[i], dtype=np.float64)
            ex, ey = (np.frexp(np.float64(v.max()) - np.float64(v.min()))[1] for v in (xf, yf))
            scale = 2.0 ** (int(ex) - int(ey) + 29)
            ks = np.unique(s * scale)
            at = max(0, int(np.searchsorted(ks, -0.75 * scale)) - 100) if line else ks.size // 2
            lo, hi = np.floor(ks[[at, min(at + 300, ks.size - 1)]]).astype(np.int64).tolist()
            want = set(s[(s * scale >= lo) & (s * scale < hi)].tolist())
            for seed in (None,) if line else range(4):
                assert D.listed_f32(xf, yf, lo, hi, parts, seed) == want, (n, line, seed)


# The counters of ordinary sets at these sizes: at most 16 phases, 32 candidates a point and leaf, 10 slopes scored.
@pytest.mark.parametrize("kind,n,h", [("duplicates", 2048, 0), ("duplicates", 513, 0), ("two_lines", 4096, 4096),
                                      ("pure", 2048, 267), ("rows", 2048, 0), ("collinear", 4096, 0)])
def test_shared_slopes_take_bounded_work(D, kind, n, h):
    """Duplicates and points on few lines: the candidates of the pair search and the phases stay bounded (the pairs in
    one cell are quadratically many, with few distinct slopes)."""
    _, c = D.i16(*points(kind, n, n), h)
    assert c["phases"] <= 64, c
    assert c["candidates_sum"] <= 4096 * n, c
    assert c["exact_sum"] <= 512, c


def test_shared_widths_are_not_scored_as_fractions(D):
    """Points in few columns: many slopes share the width; only slopes of pairs are scored (they were 253,056
    fractions, most of them no pair's slope)."""
    _, c = D.i16(*points("vertical", 8192, 8192), 6144)
    assert c["exact_sum"] <= 16384 and c["phases"] <= 256, c


@pytest.mark.parametrize("kind", ["line", "sloped", "pure", "random", "full", "digital", "columns", "duplicates",
                                  "vertical", "two_lines"])
def test_small_sets_of_a_batch_end_early(D, orc, kind):
    """Sets of 97 to 256 points finish, or are left to the plain kernel after a bounded number of phases; ordinary ones
    finish."""
    for n in (97, 128, 200, 256):
        for seed in range(6):
            x, y = (v.astype(np.int16) for v in points(kind, n, 100 * n + seed))
            for h in (0, int(0.75 * n), n // 3 + 1):
                r, c = D.i16(x, y, h, 2)
                assert c["phases"] <= 22, (n, seed, h, c)
                if c["done"]:
                    want = orc.lms_i16(x, y, h, "brute" if n <= 128 else "sweep")
                    assert tuple(int(r[k]) for k in EXACT) == tuple(want.exact())
                else:
                    assert kind in ("columns", "duplicates", "vertical", "two_lines", "pure"), (n, seed, h, c)


# ---------------------------------------------------------------- float sets
def best_line(x, y, h):
    """(w, theta1, theta2, pair) of the narrowest window over all pair slopes, computed as the float sweep does:
    slopes and projections in double, the first in the order (w, theta1, theta2, pair)."""
    x, y = x.astype(np.float64), y.astype(np.float64)
    n = x.size
    h = h or n // 2 + 1
    i, j = np.triu_indices(n, 1)
    dx, dy = x[j] - x[i], y[j] - y[i]
    ok = dx != 0
    i, j, dx, dy = i[ok], j[ok], dx[ok], dy[ok]
    s = np.where(dx < 0, -dy, dy) / np.abs(dx)
    best = None
    for k in range(0, s.size, 4096):
        z = np.sort(y[None] - s[k:k + 4096, None] * x[None], axis=1)
        w = z[:, h - 1:] - z[:, :n - h + 1]
        a = w.argmin(axis=1)
        r = np.arange(a.size)
        lo, hi = z[r, a], z[r, a + h - 1]
        for q in np.flatnonzero(w[r, a] == w[r, a].min()):
            c = (hi[q] - lo[q], s[k + q], 0.5 * (lo[q] + hi[q]), (int(i[k + q]), int(j[k + q])))
            best = c if best is None or c < best else best
    return best


def check_float(D, x, y, h):
    done, r, c = D.f32(x, y, h)
    if done:
        w, s, t, pair = best_line(np.float32(x), np.float32(y), h)
        assert (r["theta1"], (r["i"], r["j"])) == (s, pair) and r["theta2"] == t, (x.size, h, r, (w, s, t, pair))
        assert r["med_sq"] == (0.5 * w) * (0.5 * w)
    return done, c


@pytest.mark.parametrize("kind", ["line", "pure", "full", "columns", "rows", "lattice", "digital", "collinear",
                                  "two_lines", "vertical", "duplicates"])
def test_float_equals_sweep_arithmetic(D, kind):
    """Integer coordinates as floats: ties of slopes and widths; an attempt that is given up is the sweep's."""
    for n in (16, 33, 64, 160):
        x, y = points(kind, n, 5 * n)
        for h in (0, int(0.75 * n), int(0.4 * n)):
            check_float(D, x, y, h)


@pytest.mark.parametrize("kind", ["line", "digital", "collinear", "rows", "two_lines"])
@pytest.mark.parametrize("n", [512, 2048])
def test_float_shared_slopes_finish(D, kind, n):
    """Pairs that share a slope are listed once (a leaf of one slope key overflowed its list: 403 phases, given up)."""
    done, _, c = D.f32(*points(kind, n, n))
    assert done and c["phases"] <= 24, c


@pytest.mark.parametrize("offset", [0.0, 1e2, 1e4, 1e5, 1e6, 1e7])
def test_float_far_from_the_origin(D, offset):
    """A common offset of up to the float's precision: the double projections round by up to a few steps of the grid
    that prunes, which no interval may be dropped for."""
    rng = np.random.default_rng(int(offset) + 1)
    finished = 0
    for trial in range(12):
        n = int(rng.integers(24, 120))
        x, y = offset + rng.normal(size=n), rng.normal(size=n) + (offset if trial % 2 else 0)
        x, y = x.astype(np.float32), y.astype(np.float32)
        for h in (0, int(0.8 * n)):
            finished += check_float(D, x, y, h)[0]
    assert finished or offset > 1e6
