"""A batch that grows between two runs of the same length and physics mode: every grid
as in a batch that held them all from the start (the same kernels and schedule: bit for
bit), with a work list that outgrows its first allocation of 1024 items."""
import numpy as np
import pytest

from paper_1109_6672_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [lbm.LBM_P_FP64, lbm.LBM_P_FP32])
def test_batch_grows_between_equal_runs(precision):
    cases = [inputs.cavity(n=n, Ra=1e4, dT_over_T0=0.2, precision=precision, seed=n)
             for n in (40, 300, 257, 300)]
    b = lbm.Batch(precision, 4, 1 << 28)
    b.set_schedule(1, 1)
    slots = [b.add(*cases[0], 40)]
    b.run(20)
    slots += [b.add(p, f, 20) for p, f in cases[1:]]
    b.run(20)
    for (p, f), s, n in zip(cases, slots, (40, 20, 20, 20)):
        one = lbm.Batch(precision, 1, 1 << 28)
        one.set_schedule(1, 1)
        t = one.add(p, f, n)
        one.run(20)
        one.run(20)
        np.testing.assert_array_equal(b.pops(s), one.pops(t))
        one.close()
    b.close()
