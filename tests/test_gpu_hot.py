"""Cubic steps of hot loads, where many particles step back or cross a transverse face and deposit past the register
window: against the FP64 oracle (bars as for every one-step parity test, FP64 1e-10, FP32 1e-5), and in time."""
import time

import numpy as np
import pytest

import synth
from tests._pic import P, Pair, make_cfg
from tests.test_gpu_parity import TOL, _coeffs, _compare

pytestmark = pytest.mark.gpu


def _hot(nx, nz, n, seed, spread, gamma, back=False):
    p = synth.random_particles(2, nx, 1, nz, n, seed=seed, gamma=gamma, spread=spread, weight=1e-3)
    if back:  # everyone steps back in z from the lower half of its cell: all deposits leave the window
        p["uz"] = -np.abs(p["uz"]) - 1.0
        p["z"] = np.floor(p["z"]) + 0.3 * (p["z"] % 1.0)
    return p


# a few far deposits per item, about half, and every slot of full items; with and without weights
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("scheme", [0, 1, 2])
@pytest.mark.parametrize("spread,back,sigma", [(0.3, False, 0.0), (3.0, False, 2.0), (1.0, True, 0.0), (1.0, True, 2.0)])
def test_hot_step_matches_oracle(precision, scheme, spread, back, sigma):
    nx, nz, n = 19, 37, 19 * 37 * 24
    cfg = make_cfg(nx=nx, nz=nz, dt=0.6, gamma=2.0, scheme=scheme, precision=precision, ppc=12, order=3, sigma_perp=sigma,
                   track_ids=1, cap=48)
    pair = Pair(cfg, psi=_coeffs(scheme, 0.5), fields=synth.random_fields((nz, 1, nx), seed=3, scale=2e-2, smooth=1),
                part=_hot(nx, nz, n, 5, spread, 2.0, back))
    try:
        pair.step(1)
        _compare(pair, TOL[precision])
    finally:
        pair.close()


def test_hot_step_time():
    # a relativistically hot load, an eighth of whose particles deposit past the window, takes no more than three times
    # a step of a cold one; one far deposit costs about as much as the rest of a particle's step
    t = []
    for spread in (1e-4, 1.0):
        nx, nz = 256, 512
        cfg = make_cfg(nx=nx, nz=nz, dt=0.5, gamma=3.0, precision=0, ppc=8, order=3)
        h = P.pic_create(cfg)
        try:
            rng = np.random.default_rng(1)
            m = nx * nz * 8
            part = {"cell": np.tile(np.repeat(np.arange(nx * nz), 8), 2).astype(np.int32),
                    "species": np.repeat([0, 1], m).astype(np.int32), "oy": None, "w": None, "id": np.arange(2 * m, dtype=np.uint32)}
            for k in ("ox", "oz"):
                part[k] = np.tile(rng.uniform(0, 0.999, m).astype(np.float32), 2)
            for k in ("dux", "duy", "duz"):
                part[k] = (spread * rng.standard_normal(2 * m)).astype(np.float32)
            P.pic_set_state(h, P.make_state(P.PIC_HOST, None, part))
            best = 1.0
            for _ in range(5):
                P.pic_sync(h)
                t0 = time.perf_counter()
                P.pic_step(h, 8)
                P.pic_sync(h)
                best = min(best, time.perf_counter() - t0)
            t.append(best)
        finally:
            P.pic_destroy(h)
    assert t[1] <= 3 * t[0], t
