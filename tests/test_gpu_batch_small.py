"""Batches too small to fill the GPU with full tiles: every run's tiles are spread over its share of the SMs. Against the
FP64 oracle run by run, in 2D and 3D, and in time: a batched step takes no longer than its runs one after another."""
import time

import numpy as np
import pytest

import synth
from tests._pic import P, Pair, make_cfg
from tests.test_gpu_parity import TOL, _compare

pytestmark = pytest.mark.gpu


# one run, uneven runs (a share of less than one SM among them), different lanes per cell; FP32 and FP64
@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("ndim,grids", [(2, [(24, 1, 32, 4)]), (2, [(61, 1, 90, 4), (13, 1, 14, 8), (40, 1, 33, 20)]),
                                        (3, [(13, 11, 17, 8)]), (3, [(20, 16, 24, 8), (7, 6, 9, 2), (12, 13, 10, 12)])])
def test_small_batch_matches_oracle(ndim, grids, scheme, precision):
    cfgs = [make_cfg(ndim=ndim, nx=nx, ny=ny, nz=nz, dt=0.4, scheme=scheme, precision=precision, ppc=ppc)
            for nx, ny, nz, ppc in grids]
    b = P.pic_batch_create(cfgs)
    pairs = []
    try:
        for i, (nx, ny, nz, ppc) in enumerate(grids):
            coeffs = P.pic_compute_correction_coeffs(scheme, 0.4)
            P.pic_batch_set_correction_stencil(b, i, *coeffs)
            pairs.append(Pair(cfgs[i], psi=coeffs, fields=synth.random_fields((nz, ny, nx), seed=i, scale=2e-2, smooth=1),
                              part=synth.random_particles(ndim, nx, ny, nz, 2 * ppc * nx * ny * nz, seed=9 + i),
                              handle=P.pic_batch_run(b, i)))
        P.pic_batch_step(b, 2)
        P.pic_batch_sync(b)
        for pair in pairs:
            pair.o.step(2)
            _compare(pair, TOL[precision])
    finally:
        for pair in pairs:
            pair.close()
        P.pic_batch_destroy(b)


def _time(step, sync):
    best = 1.0
    for _ in range(6):
        sync()
        t0 = time.perf_counter()
        step()
        sync()
        best = min(best, time.perf_counter() - t0)
    return best


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("ndim,grids", [(2, [(24, 1, 32, 8)] * 2), (3, [(16, 16, 16, p) for p in (2, 8, 4, 8)]),
                                        (3, [(32, 32, 32, 8)] * 6)])
def test_small_batch_time(ndim, grids, precision):
    cfgs = [make_cfg(ndim=ndim, nx=nx, ny=ny, nz=nz, dt=0.4, gamma=3.0, precision=precision, ppc=ppc, init_beam=1, u_th=1.0)
            for nx, ny, nz, ppc in grids]
    b = P.pic_batch_create(cfgs)
    try:
        P.pic_batch_step(b, 8)
        together = _time(lambda: P.pic_batch_step(b, 8), lambda: P.pic_batch_sync(b))
    finally:
        P.pic_batch_destroy(b)
    alone = 0.0
    for c in cfgs:
        h = P.pic_create(c)
        try:
            P.pic_step(h, 8)
            alone += _time(lambda: P.pic_step(h, 8), lambda: P.pic_sync(h))
        finally:
            P.pic_destroy(h)
    assert together <= alone, (together, alone)
