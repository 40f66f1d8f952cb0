"""A patch's existing children are columns times rows of two each, so it has 0, 1, 2 or 4 of them: the level kernels'
averages multiply by 1, 1/2 or 1/4 and never divide by 3."""
import numpy as np
import pytest

import oracle


@pytest.mark.parametrize("W1,H1", [(5, 4), (6, 5), (7, 64), (37, 29), (64, 48), (65, 13), (97, 61), (200, 30), (31, 257), (301, 243)])
def test_never_three(W1, H1):
    g = oracle.geometry(W1, H1, 32, 24)
    flags = oracle.valid_flags(W1, H1, 32, 24)
    for l in range(1, g.L + 1):
        gx, gy = (g.P0x, g.P0y) if l == 1 else (g.Lx, g.Ly)
        ix, iy = np.meshgrid(np.arange(g.Lx), np.arange(g.Ly))
        lo, hi = (-1, 0) if l == 1 else (-(1 << (l - 2)), 1 << (l - 2))
        n = np.zeros(g.Lx * g.Ly, dtype=int)
        for ox in (lo, hi):
            for oy in (lo, hi):
                cx, cy = (ix + ox).ravel(), (iy + oy).ravel()
                inside = (cx >= 0) & (cy >= 0) & (cx < gx) & (cy < gy)
                c = np.where(inside, cy * gx + cx, 0)
                n += inside & (np.asarray(flags[l - 1]).ravel()[c] != 0)
        np.testing.assert_array_equal(n > 0, np.asarray(flags[l]).ravel() != 0)
        assert set(np.unique(n)) <= {0, 1, 2, 4}
