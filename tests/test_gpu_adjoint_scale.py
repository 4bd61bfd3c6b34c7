"""The adjoint's coefficient gradient is linear in the upstream gradient dw over the range that the adjoint fields
allow: the products of a field and an adjoint value leave FP32's range before either factor does, and are formed and
summed in FP64."""
import numpy as np
import pytest

from tests._pic import P, make_cfg

pytestmark = pytest.mark.gpu


# fields of 1e-14 and particles of weight 1e-12: the adjoint of the fields is about 1e-14 dw, the copies' adjoint 1e-26
# dw and its products with the fields 1e-40 dw. At dw = 2^-20 these lie below FP32's smallest number, the factors
# six powers of ten above the smallest normal one
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dexp", [-20, 40, 80])
def test_gradient_is_linear_in_dw(precision, dexp):
    nx, nz = 24, 64
    T = np.float32 if precision == 0 else np.float64
    cfg = make_cfg(nx=nx, nz=nz, dt=0.5, precision=precision, ppc=4, init_beam=1, u_th=0.0, gamma=3.0)
    cfg.omega_p_dz = 3e-6
    rng = np.random.default_rng(3)
    fields = {n: (1e-14 * rng.standard_normal((nz, 1, nx))).astype(T) for n in ("ex", "ey", "ez", "bx", "by", "bz")}
    h = P.pic_create(cfg)
    try:
        P.pic_set_correction_stencil(h, *P.pic_compute_correction_coeffs(0, 0.5))
        s = P.make_state(P.PIC_HOST, fields, None)
        s.np = -1  # the beam of pic_create stays
        P.pic_set_state(h, s)
        P.pic_adjoint_forward(h, 2, 2)
        a = np.concatenate(P.pic_adjoint_backward(h, 1.0))
        b = np.concatenate(P.pic_adjoint_backward(h, float(np.ldexp(1.0, dexp))))
    finally:
        P.pic_destroy(h)
    assert np.isfinite(a).all() and np.abs(a).min() > 0
    # FP32: the recomputed steps add the currents in another order
    assert np.abs(np.ldexp(b, -dexp) - a).max() <= (1e-3 if precision == 0 else 1e-9) * np.abs(a).max(), (a, b)
