"""The z-line solve of the exact rational multiplier against the FP64 oracle (which inverts Psi_B(D_z) as a
circulant), where its choices change: one to four factors, real and in conjugate pairs; lines too short for
the scan around the period, with its first steps and with all of them; ragged last chunks; lines per block
from eight down to one, with a partial last block."""
import numpy as np
import pytest

from tests._pic import P, rel_l2
from tests.test_gpu_parity import TOL, _random_pair

pytestmark = pytest.mark.gpu

FACTORS = [((1.0, 5.0),), ((1.0, -0.9), (1.0, 30.0)), ((1.0, 0.5, 0.8),), ((1.0, 5.0), (1.0, 0.5, 0.8)),
           ((1.0, 0.5, 0.8), (1.0, -0.6, 0.3)), ((1.0, -0.9), (1.0, 30.0), (1.0, 0.5, 0.8))]


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("factors", range(len(FACTORS)))
@pytest.mark.parametrize("nx,nz", [(3, 5), (6, 31), (610, 45), (305, 66), (301, 129), (5, 1023), (3, 4100), (2, 7000)])
def test_rational_lines(precision, factors, nx, nz):
    psi_b = np.ones(1)
    for f in FACTORS[factors]:
        psi_b = np.convolve(psi_b, f)
    xi = np.linspace(0.0, 1.0, 401)
    v = np.polyval(psi_b[::-1], xi)
    cond = v.max() / v.min()  # amplifies the rounding of the solve's input; the parity bars hold ten of it
    pair = _random_pair(2, precision, npart=0, nx=nx, nz=nz, corr_mode=1,
                        coeffs=(np.array([1.0, 0.1, 0, 0, 0]), np.pad(psi_b, (0, 5 - len(psi_b)))))
    try:
        expect = pair.o.gather_copies()
        P.pic_step(pair.h, 1)
        outs = [np.zeros(pair.o.shape, dtype=pair.T) for _ in range(6)]
        P.pic_debug_gather_copies(pair.h, P.PIC_HOST, outs)
        for c in range(2):
            assert rel_l2(outs[c], expect[c]) <= TOL[precision] * max(1.0, cond / 10), c
    finally:
        pair.close()
