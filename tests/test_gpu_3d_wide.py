"""A D3Q19 grid with more tiles along y than a launch has blocks there (65535): FP32 to
2e-5 of the oracle, as the other parity tests."""
import numpy as np
import pytest

from oracle import oracle3d as o3
from paper_1109_6672_gb300 import inputs, lbm
from paper_1109_6672_gb300.lbm3d import Lbm3d

pytestmark = pytest.mark.gpu


def test_wide_grid_3d():
    size = (2, 262150, 1)
    p = inputs.base_params3d(*size, tau_f=0.35, tau_h=0.5)
    f = inputs.uniform_fields3d(*size, seed=5, u_amp=0.02, T_amp=0.03, rho_amp=0.02)
    want = o3.Oracle3d(p).init(*f).step(2).pops()
    g = Lbm3d(dict(p, precision=lbm.LBM_P_FP32)).init(*f).step(2)
    assert np.abs(g.pops() - want).max() <= 2e-5 * np.abs(want).max()
    g.close()
