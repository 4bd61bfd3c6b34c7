"""Single steps at the ends of the number range."""
import numpy as np
import pytest

from tests._pic import P, make_cfg

pytestmark = pytest.mark.gpu
FN = ("ex", "ey", "ez", "bx", "by", "bz")


def _handle(ndim, precision, order=1, scheme=0, cells=None, species=None, mom=None, fields=None, sigma=0.0, w=None,
            nx=24, nz=32, targets=3):
    """A handle with particles at the middle of the given cells, momenta mom[3] relative to the drift (gamma = 130)."""
    T = np.float32 if precision == 0 else np.float64
    ny = 10 if ndim == 3 else 1
    cfg = make_cfg(ndim=ndim, nx=nx, ny=ny, nz=nz, dt=0.5, precision=precision, order=order, scheme=scheme, ppc=1,
                   sigma_perp=sigma, targets=targets)
    cfg.diag_every = 1
    n = len(cells)
    part = {"cell": np.asarray(cells, np.int32), "species": np.asarray(species, np.int32), "id": np.arange(n, dtype=np.uint32),
            "ox": np.full(n, 0.5, T), "oy": np.full(n, 0.5, T) if ndim == 3 else None, "oz": np.full(n, 0.5, T),
            "w": np.full(n, w, T) if w is not None else None}
    for k, v in zip(("dux", "duy", "duz"), mom):
        part[k] = np.full(n, v, T)
    f = {k: np.zeros((nz, ny, nx), T) for k in FN}
    for k, v in (fields or {}).items():
        f[k][...] = v
    h = P.pic_create(cfg)
    P.pic_set_state(h, P.make_state(P.PIC_HOST, f, part))
    return h, cfg, T


@pytest.mark.parametrize("ndim,order,scheme", [(2, 1, 0), (2, 3, 0), (3, 1, 0), (3, 3, 0)])
def test_kinetic_record_past_fp32(ndim, order, scheme):
    # a thread's sum stays below 3.4e38, a warp's does not; the record is FP64 from there on. An electron and a
    # positron on the same spot: no net current
    nx, ny, nz = 24, 10 if ndim == 3 else 1, 32
    cell = np.tile(np.arange(nx * ny * nz), 2)
    species = np.repeat([0, 1], nx * ny * nz)
    w = 5e35 if ndim == 2 else 2.5e35
    h, cfg, T = _handle(ndim, 0, order, scheme, cell, species, (0, 0, 0), sigma=1.0, w=w)
    try:
        P.pic_step(h, 1)
        e = P.pic_energy_history(h, 4)[-1]
    finally:
        P.pic_destroy(h)
    want = len(cell) * float(T(w)) * 129.0
    assert want > 3.4e38 * 8
    assert abs(e["k"] - want) <= 1e-5 * want, e
