"""The density pass's FP16 filter (csrc/k_density.cu, phase 1) restated in numpy:
a pair within r_c always passes, and few pairs outside do."""
import numpy as np
import pytest

F16 = np.float16
FILT = np.float64(1.0 + 9.0 / 1024.0)


def _fma16(a, b, c):
    """One FP16 fused multiply-add (FP64 holds the exact product and sum)."""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F16)


def _passes(xi, xj, yi, yj, zi, zj):
    d = [(a.astype(np.float64) - b.astype(np.float64)).astype(F16)
         for a, b in ((xi, xj), (yi, yj), (zi, zj))]
    t = np.full(xi.shape, -FILT).astype(F16)
    for c in d:
        t = _fma16(c, c, t)
    return np.signbit(t)


@pytest.mark.parametrize("nc, h", [(3, 4.0 / 3.0 - 1e-9), (4, 1.0), (5, 1.19), (8, 1.0), (9, 1.1),
                                   (2, 1.4999), (1, 1.9999)])
def test_filter_keeps_every_partner(nc, h):
    """Home and candidate in neighbouring cells of edge h (in r_c), in every window
    position of the row: r < 1 passes, and less than 2 % more than those do."""
    rng = np.random.default_rng(int(1000 * h) + nc)
    n = 400_000
    q = rng.integers(0, nc, n)                       # home's column
    cells = [rng.integers(-1, 2, n) if nc > 1 else np.zeros(n, int) for _ in range(3)]
    if nc < 3:                                       # not periodic: stay inside
        cells[0] = np.clip(q + cells[0], 0, nc - 1) - q
    oi = (rng.random((3, n)) - 0.5) * h
    oj = (rng.random((3, n)) - 0.5) * h
    # a third of the pairs just inside the cutoff
    u = rng.normal(size=(3, n))
    u *= (1.0 - 1e-7 * rng.random(n)) / np.linalg.norm(u, axis=0)
    near = np.arange(n) % 3 == 0
    edge = oi - u - np.array(cells) * h
    ok = near & (np.abs(edge) <= 0.5 * h).all(0)
    oj = np.where(ok, edge, oj)
    oi32, oj32 = oi.astype(np.float32), oj.astype(np.float32)
    d = oi32.astype(float) - np.array(cells) * h - oj32.astype(float)
    r2 = (d * d).sum(0)
    # the row of the candidate: its own offset; the home moved by the row's offset
    y = [((oi32[k] - cells[k] * h).astype(np.float32)).astype(F16) for k in (1, 2)]
    yj = [oj32[k].astype(F16) for k in (1, 2)]
    col = q + cells[0]
    across = (col < 0) | (col >= nc)
    col = col % nc
    win_b = ((q + 1) & 3) < 2

    def x16(window_col, off):
        return ((2 * window_col - 3) * np.float32(0.5 * h) + off).astype(np.float32).astype(F16)
    xj_a, xj_b = x16(col & 3, oj32[0]), x16((col + 2) & 3, oj32[0])
    xi_n = np.where(win_b, x16((q + 2) & 3, oi32[0]), x16(q & 3, oi32[0]))
    # across a periodic face: one cell, met from the column beside it
    xi_f = x16((col & 3) + np.where(q == 0, 1, -1), oi32[0])
    xi = np.where(across, xi_f, xi_n).astype(F16)
    xj = np.where(across, xj_a, np.where(win_b, xj_b, xj_a)).astype(F16)
    p = _passes(xi, xj, y[0], yj[0], y[1], yj[1])
    # (at an edge of 1e-7 the FP32 offsets may put the pair outside by their rounding)
    inside = r2 < 1.0
    assert inside.sum() > n // 20
    assert p[inside].all()
    far = r2 > 1.02
    assert not p[far].any()
