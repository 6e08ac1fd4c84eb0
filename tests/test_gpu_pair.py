"""Step over column pairs (FP32 and 16-bit storage) at the edges of its blocks: odd
widths (the last pair holds one node), one to three nodes along an axis, one column
more or less than a block's 128, block heights beyond the grid, over every rule of its
sides and alone or in a batch.  FP32 to 2e-5 of the FP64 oracle, as the other FP32
parity tests; 16-bit storage to 8 quanta of the largest deviation from the rest state, as
there; a batch to 1e-5 of the single grids."""
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
    "x_mrt": dict(bc=[ADI, ISO, P, P], T_wall=[1.0, 1.05, 1.0, 1.0], collision=1, s_q=1.4),
    "y_nee": dict(bc=[P, P, ISO, ADI], T_wall=[1.0, 1.0, 1.03, 1.0], wall_nee=12),
    "cavity": dict(bc=[ISO, ISO, ADI, ADI], T_wall=[1.1, 0.9, 1.0, 1.0], energy_model=1, g=1e-3,
                   b=5.0),
    "open": dict(bc=[INL, OUT, P, P], correction=0, in_rho=1.0, in_drho=0.01, in_du=0.007,
                 in_dT=0.006, in_omega=0.09, u_wall=[[0.01, 0.002], [0, 0], [0, 0], [0, 0]]),
}
SIZES = [(3, 3), (4, 17), (5, 3), (127, 4), (128, 7), (129, 3), (130, 26), (257, 5)]
STEPS = 12


def _case(size, sides, precision):
    p = inputs.base_params(*size, tau_f=0.35, tau_h=0.5, precision=precision, **SIDES[sides])
    return p, inputs.uniform_fields(*size, seed=3, u_amp=0.02, T_amp=0.03, rho_amp=0.02)


def _oracle(p, f):
    return orc.Oracle(dict(p, precision=lbm.LBM_P_FP64)).init(*f).step(STEPS).pops()


@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("size", SIZES, ids=lambda s: f"{s[0]}x{s[1]}")
def test_pair_parity_fp32(sides, size):
    p, f = _case(size, sides, lbm.LBM_P_FP32)
    want, got = _oracle(p, f), None
    for rows in (0, 1, 5, 64):
        g = lbm.Lbm(p).set_launch(1, rows).init(*f).step(STEPS)
        pops = g.pops()
        g.close()
        assert np.abs(pops - want).max() <= 2e-5 * np.abs(want).max(), rows
        if got is not None:
            np.testing.assert_array_equal(pops, got)
        got = pops


@pytest.mark.parametrize("precision,quantum", [(lbm.LBM_P_FP32_FP16, 2.0 ** -11),
                                               (lbm.LBM_P_FP32_BF16, 2.0 ** -8)])
@pytest.mark.parametrize("size", SIZES, ids=lambda s: f"{s[0]}x{s[1]}")
def test_pair_parity_16bit(size, precision, quantum):
    for sides in ("periodic", "walls", "cavity"):
        p, f = _case(size, sides, precision)
        want = _oracle(p, f)
        g = lbm.Lbm(p).init(*f).step(STEPS)
        err = np.abs(g.pops() - want).max()
        g.close()
        rest = orc.Oracle(dict(p, nx=1, ny=1, bc=[P] * 4, precision=lbm.LBM_P_FP64)).init(
            1.0, 0.0, 0.0, p["T0"]).pops()
        assert err <= 8 * quantum * np.abs(want - rest).max(), sides


@pytest.mark.parametrize("size", [(1, 1), (1, 7), (6, 1), (2, 2)], ids=lambda s: f"{s[0]}x{s[1]}")
def test_pair_one_node_axes(size):
    p, f = _case(size, "periodic", lbm.LBM_P_FP32)
    want = _oracle(p, f)
    g = lbm.Lbm(p).init(*f).step(STEPS)
    assert np.abs(g.pops() - want).max() <= 2e-5 * np.abs(want).max()
    g.close()


def test_pair_batch_matches_single():
    cases = [_case(size, sides, lbm.LBM_P_FP32)
             for size, sides in zip(SIZES, ["periodic", "walls", "x_mrt", "cavity"] * 2)]
    for rows, dynamic in ((0, 1), (1, 0), (5, 1)):
        b = lbm.Batch(lbm.LBM_P_FP32, len(cases), 1 << 28)
        b.set_schedule(rows, dynamic)
        slots = [b.add(p, f, STEPS) for p, f in cases]
        b.run(STEPS)
        for (p, f), s in zip(cases, slots):
            g = lbm.Lbm(p).init(*f).step(STEPS)
            want = g.pops()
            assert np.abs(b.pops(s) - want).max() <= 1e-5 * np.abs(want).max(), (rows, p["nx"])
            g.close()
        b.close()
