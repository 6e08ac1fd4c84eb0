"""FP64 tiles on grids one or two columns wide with tall requested tiles, periodic and
between walls of non-equilibrium extrapolation, against the oracle (the FP64 parity
bound of the other kernels, 1e-12)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1109_6672_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

SIDES = {"periodic": dict(),
         "nee": dict(bc=[0, 0, 1, 2], T_wall=[1.0, 1.0, 1.04, 1.0], wall_nee=12)}


@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("size", [(1, 32), (1, 64), (2, 33), (2, 64)],
                         ids=lambda s: f"{s[0]}x{s[1]}")
def test_tall_tiles_on_narrow_grids(size, sides):
    p = inputs.base_params(*size, tau_f=0.35, tau_h=0.5, **SIDES[sides])
    f = inputs.uniform_fields(*size, seed=3, u_amp=0.02, T_amp=0.03, rho_amp=0.02)
    want = orc.Oracle(p).init(*f).step(12).pops()
    for rows in (32, 64):
        g = lbm.Lbm(p).set_launch(0, rows).init(*f).step(12)
        assert np.abs(g.pops() - want).max() <= 1e-12 * np.abs(want).max(), rows
        g.close()
