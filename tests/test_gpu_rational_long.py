"""The exact rational multiplier on z-lines that fill shared memory, one to a block, at the last length that fits and
at the first that does not (a thread per line), against the operator's symbol Psi_E / Psi_B in FFT space."""
import numpy as np
import pytest

from tests._pic import P, make_cfg, rel_l2
from tests.test_gpu_parity import TOL

pytestmark = pytest.mark.gpu

# one to four factors, real and in conjugate pairs
FACTORS = [((1.0, 5.0),), ((1.0, 0.5, 0.8),), ((1.0, -0.9), (1.0, 30.0), (1.0, 0.5, 0.8))]


# 12,801 cells take more than half of the 200 KB a block may have; 25,568 all of them
@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("factors", range(len(FACTORS)))
@pytest.mark.parametrize("nz", [12801, 25568, 25600])
def test_long_lines(precision, factors, nz):
    psi_b = np.ones(1)
    for f in FACTORS[factors]:
        psi_b = np.convolve(psi_b, f)
    psi_e = np.array([1.0, 0.1, 0.0, 0.0, 0.0])
    T = np.float64 if precision else np.float32
    nx = 3
    rng = np.random.default_rng(1)
    fields = {n: rng.standard_normal((nz, 1, nx)).astype(T) for n in ("ex", "ey", "ez", "bx", "by", "bz")}
    xi = np.sin(np.pi * np.arange(nz) / nz) ** 2
    e, b = np.polyval(psi_e[::-1], xi), np.polyval(psi_b[::-1], xi)
    h = P.pic_create(make_cfg(nx=nx, nz=nz, precision=precision, targets=0, corr_mode=1, cap=8))
    try:
        P.pic_set_correction_stencil(h, psi_e, np.pad(psi_b, (0, 5 - len(psi_b))))
        P.pic_set_state(h, P.make_state(P.PIC_HOST, fields, None))
        P.pic_step(h, 1)
        outs = [np.zeros((nz, 1, nx), T) for _ in range(6)]
        P.pic_debug_gather_copies(h, P.PIC_HOST, outs)
        # Psi_B's spread amplifies the rounding of the solve's input; the parity bars hold ten of it
        for c, n in enumerate(("ex", "ey")):
            want = np.fft.ifft(np.fft.fft(fields[n].astype(np.float64), axis=0) * (e / b)[:, None, None], axis=0).real
            assert rel_l2(outs[c], want) <= TOL[precision] * max(1.0, b.max() / b.min() / 10), c
    finally:
        P.pic_destroy(h)
