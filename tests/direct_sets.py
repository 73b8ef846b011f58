"""Point sets for the tests of the one-kernel branch-and-bound: ordinary
ones, and the forms where many pairs share a slope or many slopes a width."""
import numpy as np

from paper_1510_01041_gb300 import datagen


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
    if kind == "rows":
        return rng.integers(-30000, 30000, n), rng.integers(0, 3, n)
    if kind == "vertical":      # most points in five columns
        return np.where(rng.random(n) < 0.6, rng.integers(-2, 3, n), rng.integers(-9000, 9000, n)), \
            rng.integers(-16000, 16000, n)
    if kind == "lattice":
        return rng.integers(-20, 20, n), rng.integers(-20, 20, n)
    if kind == "digital":       # a digitised line of a 640 x 480 image and noise pixels
        x = rng.integers(-320, 320, n)
        y = np.rint(0.37 * x + 11).astype(int)
        noise = rng.random(n) < 0.2
        y[noise] = rng.integers(-240, 240, noise.sum())
        return x, y
    if kind == "collinear":     # seven in ten on one line
        x = rng.integers(-1000, 1000, n)
        y = 3 * x - 7
        noise = rng.random(n) < 0.3
        y[noise] = rng.integers(-3000, 3000, noise.sum())
        return x, y
    if kind == "two_lines":
        x = rng.integers(-10000, 10000, n)
        return x, np.where(rng.random(n) < 0.5, x // 2 + 5, -x // 3 - 9)
    if kind == "equal_x":
        return np.full(n, 7), rng.integers(-500, 500, n)
    assert kind == "duplicates"
    same = rng.random(n) < 0.7
    return np.where(same, 5, rng.integers(-300, 300, n)), np.where(same, -8, rng.integers(-300, 300, n))
