"""The charge density of pic_charge_residual against the oracle's of the same state at every lanes-per-cell
class of its kernel (32 lanes for a few cells, one for many; ragged last warps), both shapes and dimensions,
with and without per-particle weights, over uneven cells."""
import numpy as np
import pytest

import synth
from tests._pic import P, Pair, make_cfg
from tests.test_gpu_gauss import _oracle_residual

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("order", [1, 3])
@pytest.mark.parametrize("sigma", [0.0, 2.0])
@pytest.mark.parametrize("nx,ny,nz,npart", [(5, 0, 7, 900), (41, 0, 67, 20000), (150, 0, 280, 60000),
                                            (281, 0, 277, 90000), (11, 7, 13, 20000), (44, 43, 42, 90000)])
def test_charge_density(precision, order, sigma, nx, ny, nz, npart):
    ndim = 3 if ny else 2
    cfg = make_cfg(ndim=ndim, nx=nx, ny=max(ny, 1), nz=nz, dt=0.4, precision=precision, order=order, sigma_perp=sigma,
                   cap=128)
    shape = (nz, max(ny, 1), nx)
    pair = Pair(cfg, fields=synth.random_fields(shape, seed=3, scale=2e-2, smooth=1),
                part=synth.random_particles(ndim, nx, max(ny, 1), nz, npart, seed=5, per_particle_weight=sigma > 0))
    try:
        got = P.pic_charge_residual(pair.h)
        want = _oracle_residual(pair, cfg)
    finally:
        pair.close()
    # a node sums a few dozen FP64 terms on either side
    for name, w in zip(("max", "rms", "rho_max"), want):
        assert abs(got[name] - w) <= 1e-12 * want[0], (name, got, want)
