"""A viscosity law so large that the relaxation rates vanish (theta^n beyond the range of
the storage's arithmetic, or its square): the step streams, as the oracle's does, and
stays finite.  Bounds: those of the other parity tests (FP64 1e-12, FP32 2e-5)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1109_6672_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [60.0, 100.0, 700.0])
@pytest.mark.parametrize("precision,bound", [(lbm.LBM_P_FP64, 1e-12), (lbm.LBM_P_FP32, 2e-5)])
def test_vanishing_rates(precision, bound, n):
    p = inputs.base_params(37, 9, tau_f=0.35, tau_h=0.5, b=5.0, energy_model=inputs.E_INTERNAL,
                           mu_law=1, mu_n=n, correction=0)
    rho, ux, uy, T = inputs.uniform_fields(37, 9, seed=3, u_amp=0.02, T_amp=0.03, rho_amp=0.02)
    f = (rho, ux, uy, 2.5 * T)  # 2.5^60 = 8e23, 2.5^100 = 6e39, 2.5^700 = 4e278
    want = orc.Oracle(p).init(*f).step(6).pops()
    assert np.isfinite(want).all()
    g = lbm.Lbm(dict(p, precision=precision)).init(*f).step(6)
    assert np.abs(g.pops() - want).max() <= bound * np.abs(want).max()
    g.close()
