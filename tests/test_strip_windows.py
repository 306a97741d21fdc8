"""The windows of the strip forward, from its FP32 arithmetic (CPU).

A warp (32 consecutive bins of a view) bounds the rows that its rays touch in a
strip of the image by its first and last ray of the driving axis, at the ends of
the strip's part that any of them covers, with one row of margin; samples inside
a staged window are read without further tests.  That needs the FP32 positions
of the rays in between to stay within a row of the exact, monotone ones: they
err by a few 2^-24 of |f0| <= n + n df, df <= the pixels' aspect, so the strips
serve aspects up to 8 (0.1 rows at 16384 pixels).  At 1e5 the same arithmetic
leaves the window."""
import math

import numpy as np
import pytest

F = np.float32
S, ROWS = 32, 160


def _table(nx, ny, dx, dy, beta, ga, sid):
    """Joseph set-up of the x-driven rays at fan angles ga of the view beta (those of the forward's table)."""
    px, py = sid * math.cos(beta), sid * math.sin(beta)
    slope = np.tan(beta - ga)                      # uy / ux
    cx, cy = 0.5 * (nx - 1), 0.5 * (ny - 1)
    df = dx * slope / dy
    f0 = (py + (-cx * dx - px) * slope) / dy + cy
    a, b = (-1.0 - f0) / df, (ny - f0) / df
    lo, hi = np.floor(np.minimum(a, b)) - 1, np.ceil(np.maximum(a, b)) + 1
    lo, hi = np.maximum(lo, 0), np.minimum(hi, nx - 1)
    hi = np.where(np.abs(slope) <= 1.0, hi, -1)    # the others are y-driven
    return f0.astype(F), df.astype(F), lo.astype(int), hi.astype(int)


def _row(f0h, df, i):
    """Lower row of the sample on driving index i: round to nearest of fma(i, df, f0 - 1/2)."""
    h = (i * df.astype(np.float64) + f0h.astype(np.float64)).astype(F)
    return np.rint(h.astype(np.float64)).astype(np.int64)


def _outside(nx, ny, dx, dy, beta, ga, sid):
    """Largest distance (rows) of a sample outside its warp's window, over the staged windows of one warp."""
    f0, df, lo, hi = _table(nx, ny, dx, dy, beta, ga, sid)
    mine = np.flatnonzero(lo <= hi)
    if not mine.size:
        return 0
    f0h = f0 - F(0.5)
    ends2 = mine[[0, -1]]
    w_lo, w_hi, worst = lo[mine].min(), hi[mine].max(), -10 ** 9
    for i0 in range(w_lo, w_hi + 1, S):
        ia, ib = max(w_lo, i0), min(w_hi, i0 + S - 1)
        ends = np.concatenate([_row(f0h[ends2], df[ends2], i) for i in (ia, ib)])
        w0, w1 = (ends.min() - 1) & ~3, ends.max() + 2
        if w1 - w0 + 1 > ROWS:
            continue
        for i in range(ia, ib + 1):
            q = mine[(lo[mine] <= i) & (i <= hi[mine])]
            if q.size:
                k = _row(f0h[q], df[q], i)
                worst = max(worst, int(w0 - k.min()), int(k.max() + 1 - w1))
    return worst


@pytest.mark.parametrize("n", [64, 1000, 16384])
@pytest.mark.parametrize("aspect", [1.0, 8.0, 0.125])
def test_samples_stay_inside_their_windows(n, aspect):
    rng = np.random.default_rng(n)
    staged = 0
    for _ in range(60 if n < 16384 else 12):
        half = 0.5 * n * math.hypot(aspect, 1.0)
        sid = half * rng.uniform(1.05, 4.0)
        step = min(aspect, 1.0) * 10 ** rng.uniform(-2, 0.5) / sid
        ga = rng.uniform(-0.8, 0.8) * half / sid + np.arange(32) * step
        w = _outside(n, n, aspect, 1.0, rng.uniform(-math.pi, math.pi), ga, sid)
        assert w <= 0
        staged += w > -10 ** 9
    assert staged > 3


def test_extreme_pixels_would_leave_their_windows():
    """Rays that pass a flat image just beyond its last column: one sample each, far from where f0 is taken."""
    n, dx, dy, worst = 16384, 1.0, 1e-5, 0
    for seed in range(40):
        rng = np.random.default_rng(seed)
        beta = rng.uniform(0.3, 0.7)
        sid = 2.0 * n
        px, py = sid * math.cos(beta), sid * math.sin(beta)
        for x in (-(n / 2 + 1) * dx, (n / 2 + 1) * dx):
            to = math.atan2(py, px - x)              # through (x, 0)
            worst = max(worst, _outside(n, n, dx, dy, beta, beta - to + np.arange(32) * 10 ** rng.uniform(-10.5, -9), sid))
    assert worst > 16
