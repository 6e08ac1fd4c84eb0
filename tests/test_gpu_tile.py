"""FP64 tile kernel: sizes at the edges of its tiles (one node, one row or
column, exact tiles, one node over, grids narrower than a warp) against the
oracle, over the side rules it writes itself, and bit-equality of the tile
heights.  The bound is the FP64 parity bound of the other kernels (1e-12)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1109_6672_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

P, ISO, ADI, INL, OUT = 0, 1, 2, 3, 4
SIDES = {
    "periodic": dict(bc=[P, P, P, P]),
    "walls": dict(bc=[ISO, ADI, ADI, ISO], T_wall=[1.04, 1.0, 1.0, 0.97],
                  u_wall=[[0, 0.03], [0, -0.02], [0.04, 0], [0.05, 0]]),
    "nee": dict(bc=[ISO, ADI, ADI, ISO], T_wall=[1.04, 1.0, 1.0, 0.97], wall_nee=13,
                u_wall=[[0, 0.03], [0, -0.02], [0.04, 0], [0.05, 0]]),
    "nee_mrt_x": dict(bc=[ADI, ISO, P, P], T_wall=[1.0, 1.05, 1.0, 1.0], wall_nee=3, collision=1,
                      s_q=1.4, mu_law=2, mu_S=0.2),
    "cavity": dict(bc=[ISO, ISO, ADI, ADI], T_wall=[1.1, 0.9, 1.0, 1.0], energy_model=1, g=1e-3,
                   b=5.0),
    "open": dict(bc=[INL, OUT, P, P], correction=0, in_rho=1.0, in_drho=0.01, in_du=0.007,
                 in_dT=0.006, in_omega=0.09, u_wall=[[0.01, 0.002], [0, 0], [0, 0], [0, 0]]),
}
SIZES = [(3, 3), (4, 33), (5, 97), (8, 12), (9, 13), (31, 3), (33, 32), (65, 9), (200, 3)]


@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("size", SIZES, ids=lambda s: f"{s[0]}x{s[1]}")
def test_tile_parity(sides, size):
    p = inputs.base_params(*size, tau_f=0.35, tau_h=0.5, **SIDES[sides])
    f = inputs.uniform_fields(*size, seed=3, u_amp=0.02, T_amp=0.03, rho_amp=0.02)
    want = orc.Oracle(p).init(*f).step(12).pops()
    got = None
    for rows in (0, 1, 3, 50):
        g = lbm.Lbm(p).set_launch(0, rows).init(*f).step(12)
        pops = g.pops()
        g.close()
        assert np.abs(pops - want).max() <= 1e-12 * np.abs(want).max(), rows
        if got is not None:
            np.testing.assert_array_equal(pops, got)
        got = pops


@pytest.mark.parametrize("size", [(1, 1), (1, 7), (6, 1), (2, 2)], ids=lambda s: f"{s[0]}x{s[1]}")
def test_tile_one_node_axes(size):
    p = inputs.base_params(*size, tau_f=0.35, tau_h=0.5)
    f = inputs.uniform_fields(*size, seed=3, u_amp=0.02, T_amp=0.03, rho_amp=0.02)
    want = orc.Oracle(p).init(*f).step(12).pops()
    g = lbm.Lbm(p).init(*f).step(12)
    assert np.abs(g.pops() - want).max() <= 1e-12 * np.abs(want).max()
    g.close()
