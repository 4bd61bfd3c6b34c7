"""One step from cells holding uneven particle counts, against the FP64 oracle.

The push kernels hand a cell's particles to a few lanes in rounds, so what matters is the counts per
cell and species: none, fewer than the lanes, one more than a full round or item, one species only, all
of a warp's cells empty. Bars as for every one-step parity test: FP64 1e-10, FP32 1e-5."""
import numpy as np
import pytest

import synth
from tests._pic import Pair, make_cfg
from tests.test_gpu_parity import TOL, _coeffs, _compare

pytestmark = pytest.mark.gpu


def _uneven(ndim, nx, ny, nz, seed, gamma=130.0):
    """Particles with per-cell counts walking through 0 .. 19 electrons and 0 .. 17 positrons, and a run of
    empty cells."""
    rng = np.random.default_rng(seed)
    ncell = nx * ny * nz
    c = np.arange(ncell)
    n0, n1 = (c * 7 + c // 3) % 20, (c * 5 + c // 7) % 18
    n0[c % 11 == 0] = 0
    n1[c % 13 == 1] = 0
    n0[40:104] = 0
    n1[40:104] = 0
    cell = np.concatenate([np.repeat(c, n0), np.repeat(c, n1)])
    n = len(cell)
    p = synth.random_particles(ndim, nx, ny, nz, n, seed=seed + 1, gamma=gamma)
    i, j, k = cell % nx, (cell // nx) % ny, cell // (nx * ny)
    p["x"], p["z"] = i + rng.uniform(0, 1, n), k + rng.uniform(0, 1, n)
    p["y"] = j + rng.uniform(0, 1, n) if ndim == 3 else np.zeros(n)
    p["q"] = np.concatenate([-np.ones(n0.sum()), np.ones(n1.sum())])
    return p


# the configured ppc picks the lanes per cell (2D: 4 up to 16 particles per cell and species, else 16; 3D: 2 up
# to 8, then 8, then 16)
@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("ndim,ppc,scheme,order", [(2, 4, 0, 1), (2, 20, 0, 1), (2, 4, 1, 1), (3, 8, 0, 1), (3, 12, 0, 1),
                                                   (3, 20, 1, 1), (2, 4, 0, 3), (2, 4, 1, 3), (2, 4, 2, 3), (2, 4, 2, 1),
                                                   (3, 8, 0, 3), (3, 8, 1, 3), (3, 8, 2, 3), (3, 8, 2, 1)])
def test_step_uneven_cells(ndim, ppc, scheme, order, precision):
    nx, ny, nz = (19, 1, 45) if ndim == 2 else (11, 7, 13)
    cfg = make_cfg(ndim=ndim, nx=nx, ny=ny, nz=nz, dt=0.5, scheme=scheme, precision=precision, ppc=ppc, order=order,
                   cap=24, sigma_perp=1.0 if ndim == 3 else 0.0)
    pair = Pair(cfg, psi=_coeffs(scheme, 0.5), fields=synth.random_fields((nz, ny, nx), seed=3, scale=2e-2, smooth=1),
                part=_uneven(ndim, nx, ny, nz, seed=11))
    try:
        pair.step(1)
        _compare(pair, TOL[precision])
    finally:
        pair.close()
