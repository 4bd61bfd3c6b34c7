"""Single steps at the ends of the number range: recorded kinetic energies past FP32's range, rotations by
fields so strong that (1 + t^2) nears it, momenta whose square leaves it, and fields that are not finite where no
particle is."""
import numpy as np
import pytest

from tests._pic import P, make_cfg

pytestmark = pytest.mark.gpu
FN = ("ex", "ey", "ez", "bx", "by", "bz")
# the pushes that read a window of nodes: cubic shapes, and the momentum-conserving gather
WINDOW = [(2, 3, 0), (2, 3, 1), (2, 3, 2), (2, 1, 2), (3, 3, 0), (3, 3, 1), (3, 3, 2), (3, 1, 2)]


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


def _momenta(h, n, T):
    out = {k: np.zeros(n, T) for k in ("dux", "duy", "duz", "oz")}
    out.update({k: np.zeros(n, np.int32) for k in ("cell", "species")}, id=np.zeros(n, np.uint32))
    s = P.make_state(P.PIC_HOST, None, out)
    s.np = n
    P.pic_get_state(h, s)
    order = np.argsort(out["id"])
    return {k: v[order] for k, v in out.items()}


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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ndim,order,scheme", WINDOW)
def test_rotation_by_a_very_strong_field(ndim, order, scheme, precision):
    # t = dt/2 B / gamma with t^2 past the FP32 estimates' range (a reciprocal of more than 2^126): the rotation
    # about B tends to half a turn, u perpendicular to B changes sign
    t = 1.25e19 if precision == 0 else 1e25
    cells, species = [5 * 24 + 7] * 2, [0, 1]
    h, cfg, T = _handle(ndim, precision, order, scheme, cells, species, (3.0, 0.25, 0.0), {"by": t * 130.0 / 0.25})
    u0 = float(T(np.sqrt(130.0 ** 2 - 1)))
    try:
        P.pic_step(h, 1)
        P.pic_sync(h)
        m = _momenta(h, 2, T)
    finally:
        P.pic_destroy(h)
    tol = 1e-5 if precision == 0 else 1e-10
    assert np.abs(m["duz"] + u0 + u0).max() <= tol * u0, m  # u_z = u0 + duz -> -u0
    assert np.abs(m["dux"] + 3.0).max() <= tol * u0, m
    assert np.abs(m["duy"] - 0.25).max() <= tol * u0, m


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ndim,order,scheme", WINDOW)
def test_momenta_past_fp32_squares(ndim, order, scheme, precision):
    # FP64: u = 1e25 moves at the speed of light. FP32: u^2 is infinite and the velocity comes out zero, which is no
    # error of the step
    h, cfg, T = _handle(ndim, precision, order, scheme, [5 * 24 + 7] * 2, [0, 1], (0.0, 0.0, 1e25))
    try:
        P.pic_step(h, 1)
        P.pic_sync(h)
        m = _momenta(h, 2, T)
    finally:
        P.pic_destroy(h)
    assert (m["duz"] == T(1e25)).all(), m
    k = m["cell"] // (24 * (10 if ndim == 3 else 1))
    z0 = 5 // (10 if ndim == 3 else 1)
    assert np.abs(k + m["oz"] - (z0 + (1.0 if precision else 0.5))).max() <= 1e-12, m


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ndim,order,scheme", WINDOW + [(2, 1, 0), (2, 1, 1), (3, 1, 0)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_bad_fields_without_particles(ndim, order, scheme, precision, bad):
    # particles in cells x = 0 of some rows, a bad value seven cells on in the same rows, filters off: no particle
    # reads it, and the cells beside it, which share the particles' warps, are empty
    nx, ny, nz = 24, 10 if ndim == 3 else 1, 32
    rows = np.arange(ny * nz) * nx
    cells, species = np.tile(rows, 2), np.repeat([0, 1], len(rows))
    f = np.zeros((nz, ny, nx))
    f[:, :, 7] = bad
    want, got = [], None
    for fields in ({}, {"ex": f, "ez": f, "by": f}):
        h, cfg, T = _handle(ndim, precision, order, scheme, cells, species, (0.1, 0.2, 0.3), fields, targets=0)
        try:
            P.pic_step(h, 1)
            P.pic_sync(h)
            m = _momenta(h, len(cells), T)
            m["k"] = P.pic_energy_history(h, 4)[-1]["k"]
            want.append(m)
        finally:
            P.pic_destroy(h)
    a, b = want
    for k in ("dux", "duy", "duz", "oz", "cell"):
        np.testing.assert_array_equal(a[k], b[k])
    assert abs(a["k"] - b["k"]) <= 1e-6 * abs(a["k"])
