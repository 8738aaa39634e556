"""The grid screen's bound for rows without negative operands, emulated on the
CPU: there t_k = s_k, so one bound on the float sums, thr = u + 2 c u with u =
s_min + c s_min + d (the last two steps rounded up), keeps every candidate that
the bracket lo_k <= u keeps."""
import numpy as np

from tests.test_grid_screen import C, D, fma32, rows, truncate_to_float


def up(x):
    """The smallest float >= x (x a float64 of at most two float roundings)."""
    f = np.float32(x)
    return f if np.float64(f) >= x else np.nextafter(f, np.float32(np.inf))


def test_bound_keeps_every_fp64_minimiser_and_every_bracket():
    rng = np.random.default_rng(33)
    for g, f in rows(rng, 5000):
        g, f = np.abs(g), np.abs(f)
        a, b = truncate_to_float(g), truncate_to_float(f)
        s = (a + b).astype(np.float32)
        hi = fma32(np.full_like(s, C), s, s)
        u = up(np.float64(fma32(C, s.min(), s.min())) + np.float64(D))
        assert hi.min() == fma32(C, s.min(), s.min())
        thr = up(np.float64(u) + 2.0 * np.float64(C) * np.float64(u))
        kept = s <= thr
        lo = fma32(np.full_like(s, -C), s, s)
        assert kept[lo <= u].all()
        sums = g + f
        assert kept[sums == sums.min()].all()
