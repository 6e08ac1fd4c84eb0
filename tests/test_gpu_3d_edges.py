"""D3Q19 step at the edges of its tiles and z ranges (one node along an axis, one
over a tile, grids narrower than a warp), over every kind of side: populations that
leave through periodic sides, walls, and edges where both meet, in FP64 (both tile
shapes) and FP32 (each launch shape) against the oracle.  Bounds: 1e-12 in FP64 and
2e-5 in FP32, those of the other three-dimensional parity tests."""
import numpy as np
import pytest

from oracle import oracle3d as o3
from paper_1109_6672_gb300 import inputs, lbm
from paper_1109_6672_gb300.lbm3d import Lbm3d

pytestmark = pytest.mark.gpu

P, ISO, ADI = 0, 1, 2
UX = [[0.0, 0.02, -0.01], [0.0, -0.015, 0.02]]
UY = [[0.01, 0.0, 0.02], [-0.02, 0.0, 0.01]]
UZ = [[0.02, 0.01, 0.0], [-0.01, 0.02, 0.0]]
SIDES = {
    "periodic": dict(),
    "x": dict(bc_x=[ISO, ADI], T_wall_x=[1.03, 1.0], u_wall_x=UX),
    "y": dict(bc_y=[ADI, ISO], T_wall_y=[1.0, 0.98], u_wall_y=UY),
    "xz": dict(bc_x=[ISO, ISO], T_wall_x=[1.03, 0.97], bc_z=[ADI, ADI], u_wall_z=UZ,
               energy_model=inputs.E_INTERNAL, g=1e-3, b=5.0),
    "xyz": dict(bc_x=[ADI, ISO], T_wall_x=[1.0, 1.02], u_wall_x=UX, bc_y=[ISO, ADI],
                T_wall_y=[0.98, 1.0], u_wall_y=UY, bc_z=[ISO, ISO], T_wall_z=[1.01, 0.99],
                u_wall_z=UZ),
}
SIZES = [(2, 2, 2), (3, 17, 5), (16, 16, 4), (17, 4, 33), (32, 5, 3), (33, 9, 2), (65, 3, 7)]


@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("size", SIZES, ids=lambda s: "x".join(map(str, s)))
def test_edges_3d(size, sides):
    p = inputs.base_params3d(*size, tau_f=0.35, tau_h=0.5, **SIDES[sides])
    f = inputs.uniform_fields3d(*size, seed=5, u_amp=0.02, T_amp=0.03, rho_amp=0.02)
    want = o3.Oracle3d(p).init(*f).step(12).pops()
    runs = [(lbm.LBM_P_FP64, s, 1e-12) for s in ((0, 0), (8, 0))] + [
        (lbm.LBM_P_FP32, s, 2e-5) for s in ((0, 0), (8, 0), (16, 0), (8, 1))]
    for precision, shape, bound in runs:
        g = Lbm3d(dict(p, precision=precision)).set_launch(*shape).init(*f).step(12)
        assert np.abs(g.pops() - want).max() <= bound * np.abs(want).max(), (precision, shape)
        g.close()


@pytest.mark.parametrize("size", [(1, 1, 1), (1, 5, 3), (6, 1, 2), (3, 4, 1)],
                         ids=lambda s: "x".join(map(str, s)))
def test_one_node_axes_3d(size):
    p = inputs.base_params3d(*size, tau_f=0.35, tau_h=0.5)
    f = inputs.uniform_fields3d(*size, seed=5, u_amp=0.02, T_amp=0.03, rho_amp=0.02)
    want = o3.Oracle3d(p).init(*f).step(12).pops()
    for precision, bound in ((lbm.LBM_P_FP64, 1e-12), (lbm.LBM_P_FP32, 2e-5)):
        g = Lbm3d(dict(p, precision=precision)).init(*f).step(12)
        assert np.abs(g.pops() - want).max() <= bound * np.abs(want).max(), precision
        g.close()
