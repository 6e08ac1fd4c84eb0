"""Grids with more rows than a launch has blocks along y (65535) at the default height:
FP32 to 2e-5 and 16-bit storage to 8 quanta of the largest deviation from the rest
state, as the other parity tests."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1109_6672_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def test_tall_grid():
    size = (3, 400001)
    p = inputs.base_params(*size, tau_f=0.35, tau_h=0.5)
    f = inputs.uniform_fields(*size, seed=3, u_amp=0.02, T_amp=0.03, rho_amp=0.02)
    want = orc.Oracle(p).init(*f).step(2).pops()
    rest = orc.Oracle(dict(p, nx=1, ny=1)).init(1.0, 0.0, 0.0, p["T0"]).pops()
    for precision, bound in ((lbm.LBM_P_FP32, 2e-5 * np.abs(want).max()),
                             (lbm.LBM_P_FP32_BF16, 8 * 2.0 ** -8 * np.abs(want - rest).max())):
        g = lbm.Lbm(dict(p, precision=precision))
        for rows in (0, 1):
            g.set_launch(0, rows).init(*f).step(2)
            assert np.abs(g.pops() - want).max() <= bound, (precision, rows)
        g.close()
