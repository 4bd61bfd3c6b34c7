"""The adjoint makes room for the particles its bins cannot hold: a run whose particles focus past the bins and part
again, so that the state at its end fits. The forward pass grows the bins at its checkpoints, the backward pass
where it sees particles wait; neither pushes them from the spill list in every pass that follows."""
import numpy as np
import pytest

from tests._pic import P, make_cfg

pytestmark = pytest.mark.gpu


def _focus(nx, nz, ppc, T, steps, dt=0.5, width=5):
    """Neutral pairs that drift along x into every fifth column at step steps / 2, without fields, and apart again."""
    rng = np.random.default_rng(1)
    cell = np.repeat(np.arange(nx * nz), ppc)
    i, ox = cell % nx, rng.uniform(0.05, 0.95, len(cell))
    v = (i // width * width + width / 2 + 0.8 * (ox - 0.5) - (i + ox)) / (steps / 2) / dt
    p = {"cell": np.tile(cell, 2).astype(np.int32), "species": np.repeat([0, 1], len(cell)).astype(np.int32),
         "id": np.arange(2 * len(cell), dtype=np.uint32), "oy": None, "w": None, "ox": np.tile(ox, 2).astype(T),
         "oz": np.tile(rng.uniform(0.05, 0.95, len(cell)), 2).astype(T), "dux": np.tile(v / np.sqrt(1 - v * v), 2).astype(T)}
    p["duy"], p["duz"] = np.zeros(2 * len(cell), T), np.zeros(2 * len(cell), T)
    return p


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("every", [1, 3, 12])
def test_bins_grow(precision, every):
    # 8 per cell and species in bins of 16; at step 6 a fifth of the cells hold 40
    nx, nz, steps = 255, 256, 12
    T = np.float64 if precision else np.float32
    h = P.pic_create(make_cfg(nx=nx, nz=nz, dt=0.5, gamma=1.0, precision=precision, ppc=8, cap=16))
    try:
        part = _focus(nx, nz, 8, T, steps)
        P.pic_set_state(h, P.make_state(P.PIC_HOST, None, part))
        P.pic_adjoint_forward(h, steps, every)
        cap = P.pic_bin_stats(h)[0]
        assert every > 6 or cap >= 40, cap  # checkpoints at the focus, or the last before it
        spilled = [P.pic_bin_stats(h)[1]]
        for _ in range(4):
            P.pic_adjoint_backward(h, 1.0)
            spilled.append(P.pic_bin_stats(h)[1])
        # the first passes may still find the bins too small; from then on every particle has its slot
        assert spilled[4] == spilled[3], (cap, spilled)
        assert P.pic_num_particles(h) == len(part["cell"])
    finally:
        P.pic_destroy(h)


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("every", [1, 3, 12])
def test_gradient_with_waiting_particles(precision, every):
    # the tape takes the particles that wait from the spill list: the same gradient as with room for all of them
    nx, nz, steps = 25, 24, 12
    T = np.float64 if precision else np.float32
    rng = np.random.default_rng(2)
    fields = {n: (2e-2 * rng.standard_normal((nz, 1, nx))).astype(T) for n in ("ex", "ey", "ez", "bx", "by", "bz")}
    part, out = _focus(nx, nz, 8, T, steps), []
    for cap in (16, 128):
        h = P.pic_create(make_cfg(nx=nx, nz=nz, dt=0.5, gamma=1.0, precision=precision, ppc=8, cap=cap))
        try:
            P.pic_set_correction_stencil(h, *P.pic_compute_correction_coeffs(0, 0.5))
            P.pic_set_state(h, P.make_state(P.PIC_HOST, fields, part))
            w = P.pic_adjoint_forward(h, steps, every)
            out.append(np.concatenate([[w], *P.pic_adjoint_backward(h, 1.0)]))
            assert (P.pic_bin_stats(h)[1] > 0) == (cap == 16)
            assert P.pic_num_particles(h) == len(part["cell"])
        finally:
            P.pic_destroy(h)
    a, b = out
    # the same sums in another order, through 12 steps
    assert np.abs(a[1:] - b[1:]).max() <= (1e-11 if precision else 1e-3) * np.abs(b[1:]).max()
    assert abs(a[0] - b[0]) <= (1e-11 if precision else 1e-4) * abs(b[0])
