"""The particle tiles that push_tiles gives a grid (a host function of the library): they cover the grid, stay within
the kernels' tile, and a wave of them never holds more rows of cells than a wave of full tiles. A warp takes whole rows
of the tile's full width, so that is what a wave costs, however narrow the tiles are."""
import ctypes

import pytest

P = pytest.importorskip("paper_1401_0838_gb300")


def _tiles(ndim, es, ho, n, spread):
    nt, te = (ctypes.c_int * 3)(), (ctypes.c_int * 3)()
    P.lib()._ZN5picgb10push_tilesEiibiiiiPiS0_(ndim, es, ctypes.c_bool(ho), *n, spread, nt, te)
    return tuple(nt), tuple(te)


@pytest.mark.parametrize("ndim,es,ho", [(d, e, h) for d in (2, 3) for e in (4, 8) for h in (False, True)])
def test_rows_per_wave(ndim, es, ho):
    full = _tiles(ndim, es, ho, (1 << 12, 1 << 12, 1 << 12), 0)[1]
    resident = 152 * (1 if es == 8 else 2 if ndim == 2 else 1 if ho else 3)
    fixed = 40 if es == 4 else 6
    sizes = [3, 8, 13, 24, 32, 44, 45, 64, 100, 129, 301, 512] if ndim == 2 else [5, 13, 24, 32, 44, 48, 70]
    for nx in sizes:
        for ny in [1] if ndim == 2 else sizes:
            for nz in sizes:
                n = (nx, ny, nz)
                nt, te = _tiles(ndim, es, ho, n, 152)
                cost = []
                for t, e in ((nt, te), (tuple(-(-a // b) for a, b in zip(n, full)), full)):
                    assert all(b * c >= a for a, b, c in zip(n, t, e))
                    tiles = t[0] * t[1] * t[2]
                    cost.append(-(-tiles // resident) * (full[0] * e[1] * e[2] + fixed))
                assert all(a <= b for a, b in zip(te, full)) and min(te[0], te[2]) >= 4
                assert cost[0] <= cost[1], (n, te, cost)
