"""Steps on the narrowest grids whose field tiles are staged as boxes, and on ragged ones, against the FP64
oracle: nearly every tile there holds elements outside the grid, on one edge or on two, that are replaced by
their periodic images. Bars as for every one-step parity test: FP64 1e-10, FP32 1e-5."""
import numpy as np
import pytest

import synth
from tests._pic import P, Pair, make_cfg, rel_l2
from tests.test_gpu_parity import TOL, _coeffs, _compare

pytestmark = pytest.mark.gpu


# (ndim, nx, ny, nz, solver): the Yee boxes need 40 x 35 (FP64: 36) cells, the Cole-Karkkainen ones 40 x 37,
# the stencils' 136 x 46 and in 3D 24 x 11 x 11 and 40 x 14 x 22; narrower grids stage their elements singly
@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("ndim,nx,ny,nz,solver", [(2, 36, 1, 35, 0), (2, 40, 1, 35, 0), (2, 44, 1, 37, 0), (2, 40, 1, 37, 1),
                                                  (2, 136, 1, 46, 0), (2, 140, 1, 61, 1), (2, 268, 1, 33, 0),
                                                  (3, 24, 11, 11, 0), (3, 28, 12, 13, 0), (3, 40, 14, 22, 0),
                                                  (3, 44, 19, 25, 0)])
def test_step_on_narrow_grids(ndim, nx, ny, nz, solver, precision):
    cfg = make_cfg(ndim=ndim, nx=nx, ny=ny, nz=nz, dt=0.5, precision=precision, solver=solver,
                   sigma_perp=1.0 if ndim == 3 else 0.0)
    pair = Pair(cfg, psi=_coeffs(0, 0.5), fields=synth.random_fields((nz, ny, nx), seed=5, scale=2e-2, smooth=1),
                part=synth.random_particles(ndim, nx, ny, nz, 3000, seed=6))
    try:
        expect = pair.o.gather_copies()
        pair.step(1)
        outs = [np.zeros(pair.o.shape, dtype=pair.T) for _ in range(6)]
        P.pic_debug_gather_copies(pair.h, P.PIC_HOST, outs)
        for c in range(6):
            assert rel_l2(outs[c], expect[c]) <= TOL[precision], c
        _compare(pair, TOL[precision])
    finally:
        pair.close()
