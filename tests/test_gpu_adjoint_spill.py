"""The adjoint of a run whose bins overflow (the tape takes the waiting particles from the spill list) against
the same run with room in its bins, and the particles it leaves behind."""
import numpy as np
import pytest

from tests.test_gpu_adjoint import _beam_pair, _gpu_grad
from tests import test_gpu_adjoint as A
from tests._pic import P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("every", [1, 3, 8])
def test_gradient_with_spilled_particles(monkeypatch, precision, every):
    torch = pytest.importorskip("torch")
    out = []
    make = A.make_cfg
    for cap in (8, 64):  # 8 per cell and species at the start, then clumps
        monkeypatch.setattr(A, "make_cfg", lambda **kw: make(cap=cap, **kw))
        pair, _, _ = _beam_pair(ppc=8, u_th=0.3, precision=precision)
        try:
            n = P.pic_num_particles(pair.h)
            res = _gpu_grad(pair.h, pair.cfg, 8, every, torch.float64 if precision else torch.float32)
            if cap == 8 and precision == 1:  # FP32 bins hold at least 16
                assert P.pic_bin_stats(pair.h)[1] > 0
            assert P.pic_num_particles(pair.h) == n
            out.append(np.concatenate([[res[0]], res[1], res[2], *[g.reshape(-1) for g in res[3]]]))
        finally:
            pair.close()
    a, b = out
    # the same sums in another order, through 8 steps
    assert np.abs(a - b).max() <= (1e-11 if precision else 1e-3) * np.abs(b).max()
    assert abs(a[0] - b[0]) <= (1e-11 if precision else 1e-4) * abs(b[0])
