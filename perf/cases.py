"""The framework's work as performance cases: one pass of each public entry point at the sizes users call it with.

Sizes and distributions are those of this repository's workloads (the seeded generators in ``datagen``): single
fits from the paper's Table 1 sizes to the scaling workload's largest, the learned and branch-and-bound fits at
n = 8192 and 65536, a batch of uneven sets, Hough detection with exact refinement, and one training gradient of
the set network.
"""
import math

import numpy as np
import torch

from paper_1510_01041_gb300 import datagen, lms

DEVICE = "cuda:0"
HOUGH_THETA, HOUGH_RHO, HOUGH_PEAKS = 1024, 2896, 32
RECORD = lms.RESULT_DTYPE.itemsize


def listed():
    return [
        # a paper-size set fitted on its own (an interactive caller, one line at a time): latency and launches
        {"name": "fit_i16_n128", "kind": "fit", "dtype": "i16", "points": "line", "n": 128, "outliers": 0.4,
         "algorithm": "auto", "h": 0.0},
        # the largest sets of the per-slope kernel, ragged
        {"name": "fit_i16_n509", "kind": "fit", "dtype": "i16", "points": "sloped", "n": 509, "outliers": 0.3,
         "algorithm": "auto", "h": 0.0},
        # the scaling workload: the smallest size, one point off it
        {"name": "fit_i16_n2047", "kind": "fit", "dtype": "i16", "points": "line", "n": 2047, "outliers": 0.4,
         "algorithm": "auto", "h": 0.0},
        # the scaling workload: its middle size
        {"name": "fit_i16_n8192", "kind": "fit", "dtype": "i16", "points": "line", "n": 8192, "outliers": 0.4,
         "algorithm": "auto", "h": 0.0},
        # measured (real-valued) points, an ordinary set
        {"name": "fit_f32_n2048", "kind": "fit", "dtype": "f32", "points": "gaussian", "n": 2048, "outliers": 0.4,
         "algorithm": "auto", "h": 0.0},
        # measured points, the largest set that float input takes
        {"name": "fit_f32_n32768", "kind": "fit", "dtype": "f32", "points": "gaussian", "n": 32768, "outliers": 0.4,
         "algorithm": "auto", "h": 0.0},
        # the headline: the learned-seeded exact fit of points already on the GPU
        {"name": "learned_n8192", "kind": "learned", "n": 8192, "outliers": 0.45, "h": 0.0},
        # the same as a serving loop calls it: points in pinned host memory, the line back in host memory
        {"name": "learned_host_n8192", "kind": "learned_host", "n": 8192, "outliers": 0.45, "h": 0.0},
        # the largest single set
        {"name": "bnb_n65536", "kind": "bnb", "n": 65536, "outliers": 0.45, "h": 0.0},
        # many uneven sets at once, one call on a kept plan
        {"name": "batched_4096", "kind": "batched", "sets": 4096},
        # line detection: votes, peaks, band points and the exact line of every peak
        {"name": "hough_8x2048", "kind": "hough", "images": 8, "size": 2048, "segments": 16, "salt": 0.05,
         "max_points": 0},
        # one gradient of the set network over an ordinary training batch
        {"name": "setnet_backward_128", "kind": "backward", "sets": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit_f32", "bnb", "learned", "learned_host", "batched", "hough", "backward"])
    outliers = round(rng.uniform(0.0, 0.45), 3)
    # the median, or now and then a higher quantile of the residuals (least quantile of squares)
    h = rng.choice([0.0, 0.0, 0.0, 0.75])
    if kind == "fit":
        # "random" points have no line in them, as in the paper's Table 1
        points = rng.choice(["line", "sloped", "sloped", "random"])
        return {"kind": "fit", "dtype": "i16", "points": points, "n": _log_int(rng, 64, 16384),
                "outliers": 1.0 if points == "random" else outliers,
                "algorithm": rng.choice(["auto", "auto", "auto", "sweep"]), "h": h}
    if kind == "fit_f32":
        return {"kind": "fit", "dtype": "f32", "points": "gaussian", "n": _log_int(rng, 64, 32768),
                "outliers": outliers, "algorithm": "auto", "h": h}
    if kind in ("bnb", "learned", "learned_host"):
        return {"kind": kind, "n": _log_int(rng, 256, 65536), "outliers": outliers, "h": h}
    if kind == "batched":
        return {"kind": kind, "sets": _log_int(rng, 16, 4096)}
    if kind == "hough":
        # with max_points a band is subsampled before its fit
        return {"kind": kind, "images": rng.randint(1, 8), "size": rng.choice([512, 720, 1024, 1536, 2048]),
                "segments": rng.randint(4, 16), "salt": round(rng.uniform(0.005, 0.05), 4),
                "max_points": rng.choice([0, 0, 128, 1000])}
    return {"kind": "backward", "sets": _log_int(rng, 8, 256)}


def _points(case, seed):
    n, kind = case["n"], case.get("points", "sloped")
    if kind == "gaussian":
        return datagen.gaussian_f32(n, seed, case["outliers"])
    if kind == "sloped":
        return datagen.sloped(n, seed, case["outliers"], 1.4)[:2]
    return datagen.line_with_outliers(n, seed, case["outliers"])


def _order(case):
    """The order statistic: 0 is the library's default (the upper median)."""
    return max(2, int(math.ceil(case["h"] * case["n"]))) if case["h"] else 0


def _training_sets(case, seed):
    """A training batch as train_setnet draws it: n log-uniform in [256, 8192], up to 45% outliers."""
    st = datagen.Stream(seed)
    sizes = np.floor(256 * 32 ** st.uniform(case["sets"])).astype(np.int64)
    fracs = st.uniform(case["sets"]) * 0.45
    sets, targets = [], np.zeros((case["sets"], 2), dtype=np.float32)
    for k in range(case["sets"]):
        x, y, line = datagen.sloped(int(sizes[k]), seed * 7777 + k, float(fracs[k]), 1.4)
        sets.append((x, y))
        m = math.tan(line["phi"])
        cx, cy, scale = _frame(x, y)
        targets[k] = line["phi"], (line["c"] - cy + m * cx) / scale
    offsets = np.zeros(case["sets"] + 1, dtype=np.int64)
    offsets[1:] = np.cumsum(sizes)
    return np.concatenate([s[0] for s in sets]), np.concatenate([s[1] for s in sets]), offsets, targets


def _frame(x, y):
    x, y = x.astype(np.float64), y.astype(np.float64)
    return (0.5 * (x.min() + x.max()), 0.5 * (y.min() + y.max()),
            max(1.0, 0.5 * max(x.max() - x.min(), y.max() - y.min())))


def _to_gpu(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).to(DEVICE) for a in arrays]


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind in ("fit", "bnb", "learned"):
        s["x"], s["y"] = _to_gpu(*_points(case, seed))
        s["h"] = _order(case)
    elif kind == "learned_host":
        s["x"], s["y"] = [torch.from_numpy(a).pin_memory() for a in _points(case, seed)]
        s["out"] = torch.zeros(RECORD, dtype=torch.uint8).pin_memory()
        s["h"] = _order(case)
    elif kind == "batched":
        x, y, offsets = datagen.batch(case["sets"], seed)
        s["x"], s["y"], s["offsets"] = _to_gpu(x, y, offsets)
        s["plan"] = lms.BatchPlan(offsets)
    elif kind == "hough":
        size = case["size"]
        s["edges"] = _to_gpu(datagen.edge_images(case["images"], seed, size, size, case["segments"],
                                                 size // 10, size * 3 // 4, case["salt"]))[0]
        s["seed"] = seed
    elif kind == "backward":
        s["x"], s["y"], s["offsets"], s["targets"] = _to_gpu(*_training_sets(case, seed))
    if kind in ("learned", "learned_host", "backward"):
        s["net"] = lms.pretrained()
    return s


def run(s):
    kind = s["kind"]
    if kind == "fit":
        out = lms.fit(s["x"], s["y"], s["h"], s["case"]["algorithm"])
        return out if s["case"]["dtype"] == "i16" else _typed(out)
    if kind == "bnb":
        return lms.fit_bnb(s["x"], s["y"], s["h"], stats=False)[0]
    if kind == "learned":
        return s["net"].fit(s["x"], s["y"], s["h"], stats=False)[0]
    if kind == "learned_host":
        return s["net"].fit_host(s["x"], s["y"], s["h"], out=s["out"], stats=False)[0]
    if kind == "batched":
        return s["plan"].fit(s["x"], s["y"], s["offsets"])
    if kind == "hough":
        return _lines(lms.hough_refine(s["edges"], HOUGH_THETA, HOUGH_RHO, HOUGH_PEAKS,
                                       max_points=s["case"]["max_points"], sample_seed=s["seed"]))
    loss, grads = s["net"].backward(s["x"], s["y"], s["offsets"], s["targets"], 1.0)
    return {"loss": loss, "grads": grads}


def _typed(out):
    """A float fit's record: its integers, the line (theta1, theta2, med_sq), the pair, status and algorithm."""
    return {"rational": out[:48].view(torch.int64), "line": out[48:72].view(torch.float64),
            "ids": out[72:].view(torch.int32)}


def _lines(found):
    """Detected lines as two tables: the whole numbers and the real ones."""
    keys = ("theta_index", "rho_index", "votes", "transposed", "npoints", "nfit")
    exact = ("w_num", "w_den", "s_num", "s_den", "t_num", "t_den", "i", "j", "status", "algorithm")
    whole = np.array([[d[k] for k in keys] + [d["fit"][k] for k in exact] for d in found], dtype=np.int64)
    real = np.array([[d["fit"][k] for k in ("theta1", "theta2", "med_sq")] + [d["ols_theta1"], d["ols_theta2"]]
                     for d in found], dtype=np.float64)
    return {"whole": whole, "real": real}


def _mean_set(lo, hi):
    return (hi - lo) / math.log(hi / lo)


def work(case):
    """Inputs read once, results written once; operations: a projection (2) of every point at the answer's slope
    and one sorting step (n log2 n) for a fit, the products and sums of a vote or of the network otherwise."""
    kind = case["kind"]

    def fit_ops(n):
        return 2.0 * n + n * math.log2(n)

    if kind in ("fit", "bnb", "learned", "learned_host"):
        n = case["n"]
        return {"bytes": n * (8 if case.get("dtype") == "f32" else 4) + RECORD, "flops": fit_ops(n)}
    if kind == "batched":
        n = _mean_set(64, 4096)
        return {"bytes": case["sets"] * (4 * n + RECORD + 8), "flops": case["sets"] * fit_ops(n)}
    if kind == "hough":
        pixels = case["images"] * case["size"] ** 2
        edges = pixels * case["salt"] + case["images"] * case["segments"] * 0.425 * case["size"]
        return {"bytes": pixels + case["images"] * HOUGH_PEAKS * 144, "flops": 3.0 * edges * HOUGH_THETA}
    points = case["sets"] * _mean_set(256, 8192)
    return {"bytes": points * 4 + case["sets"] * 16 + 4 * 6498, "flops": 2.0 * 4224 * points}


# ------------------------------------------------------------------ 64-bit values
def exact(case, seed):
    """The float fits and the network's gradient in plain 64-bit torch; the other outputs are whole numbers, or
    (Hough) take one exact fit per peak."""
    if case["kind"] == "fit" and case["dtype"] == "f32":
        x, y = _points(case, seed)
        return {"rational": None, "line": _exact_line(x, y, _order(case) or case["n"] // 2 + 1), "ids": None}
    if case["kind"] == "backward":
        return _exact_gradient(*_training_sets(case, seed))
    return None


def _widths(X, Y, slopes, h):
    """The narrowest window of h projections at each slope: its width and centre."""
    z = torch.sort(Y[None] - slopes[:, None] * X[None], dim=1).values
    w, at = (z[:, h - 1:] - z[:, :z.shape[1] - h + 1]).min(dim=1)
    lo = z.gather(1, at[:, None])[:, 0]
    return w, lo + w / 2


def _in_chunks(fn, n, *slopes):
    step = max(1, (1 << 25) // n)
    parts = [fn(*(s[k:k + step] for s in slopes)) for k in range(0, slopes[0].numel(), step)]
    return [torch.cat(p) for p in zip(*parts)]


def _exact_line(x, y, h):
    """Exact least quantile of squares in float64: slope intervals are bounded below by the hulls of the projections
    over them, dropped when above the best width seen and cut finer; then every pairwise slope in what is left is
    scored."""
    device = DEVICE if torch.cuda.is_available() else "cpu"
    X, Y = (torch.from_numpy(a).to(device, torch.float64) for a in (x, y))
    n = X.numel()
    xs = torch.sort(X).values
    span = float((xs[h - 1:] - xs[:n - h + 1]).min())      # any h points span at least this in x

    def bound(a, b):
        za, zb = Y[None] - a[:, None] * X[None], Y[None] - b[:, None] * X[None]
        lo = torch.sort(torch.minimum(za, zb), dim=1).values
        hi = torch.sort(torch.maximum(za, zb), dim=1).values
        return ((lo[:, h - 1:] - hi[:, :n - h + 1]).min(dim=1).values,)

    angles = torch.linspace(-math.pi / 2, math.pi / 2, 514, dtype=torch.float64, device=device)[1:-1]
    best = float(_in_chunks(lambda s: _widths(X, Y, s, h), n, torch.tan(angles))[0].min())
    steep = (best + float(Y.max() - Y.min())) / span if span > 0 else 1e12   # beyond it w(s) >= |s| span - range(y)
    edges = torch.tan(torch.linspace(-math.atan(steep), math.atan(steep), 513, dtype=torch.float64, device=device))
    a, b = edges[:-1], edges[1:]
    for _ in range(40):
        mids = 0.5 * (a + b)
        best = min(best, float(_in_chunks(lambda s: _widths(X, Y, s, h), n, mids)[0].min()))
        keep = _in_chunks(bound, n, a, b)[0] <= best * (1 + 1e-9)
        a, b = a[keep], b[keep]
        if float((b - a).sum()) * n * n < 2000 or a.numel() > 20000:
            break
        f = torch.arange(5, dtype=torch.float64, device=device) / 4
        cut = a[:, None] + (b - a)[:, None] * f[None]
        a, b = cut[:, :-1].reshape(-1), cut[:, 1:].reshape(-1)
    step = max(1, (1 << 25) // n)
    slopes = []
    for k in range(0, n, step):
        dx = X[None, :] - X[k:k + step, None]
        s = ((Y[None, :] - Y[k:k + step, None]) / dx)[torch.triu(dx != 0, diagonal=k + 1)]
        at = torch.searchsorted(a.contiguous(), s, right=True) - 1
        slopes.append(s[(at >= 0) & (s <= b[at.clamp(min=0)])])
    slopes = torch.unique(torch.cat(slopes))
    w, centre = _in_chunks(lambda s: _widths(X, Y, s, h), n, slopes)
    k = int(w.argmin())
    return torch.stack([slopes[k], centre[k], (w[k] / 2) ** 2]).cpu()


def _exact_gradient(x, y, offsets, targets, lam=1.0):
    """Loss and gradient of the set network with its parameters rounded to bfloat16, in float64 autograd."""
    flat = torch.from_numpy(lms.pretrained().get_params()).to(torch.bfloat16).to(torch.float64).requires_grad_()
    shapes = [(64, 2), (64,), (64, 64), (64,), (32, 64), (32,), (2, 32), (2,)]
    parts = torch.split(flat, [int(np.prod(s)) for s in shapes])
    W1, b1, W2, b2, W3, b3, W4, b4 = [p.reshape(s) for p, s in zip(parts, shapes)]
    loss, sets = 0.0, len(offsets) - 1
    for k in range(sets):
        xs, ys = x[offsets[k]:offsets[k + 1]], y[offsets[k]:offsets[k + 1]]
        cx, cy, scale = _frame(xs, ys)
        p = torch.from_numpy(np.stack([(xs - cx) / scale, (ys - cy) / scale], axis=1))
        g = torch.relu(torch.relu(p @ W1.T + b1) @ W2.T + b2).max(dim=0).values
        e = torch.relu(W3 @ g + b3) @ W4.T + b4 - torch.from_numpy(targets[k]).to(torch.float64)
        loss = loss + (e[0] ** 2 + lam * e[1] ** 2) / sets
    loss.backward()
    return {"loss": loss.detach().reshape(1), "grads": flat.grad}
