"""The records of a solve that blows up inside one call of many steps.

The status of a step's record tells whether a site was flagged in that step or
before; the kernels that take many steps in one launch may not let later steps
into it.  Unlimited LBGK on states far from equilibrium loses positivity after a
few steps; every record of one call equals that of the same steps launch by
launch, and the first flagged record is the first with flagged sites.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import inputs, lbm

from test_gpu_parity import rand_state

pytestmark = pytest.mark.gpu

STEPS = 30


def records(f, **cfg):
    g = lbm.Lattice(stats_history=STEPS, **cfg)
    g.set_populations(f)
    g.step(STEPS)
    with pytest.raises(lbm.LBMError) as e:  # the sticky status, cleared here
        g.synchronize()
    assert e.value.status == lbm.ERR_NONFINITE
    return [(h["step"], h["n_bad"], h["status"]) for h in g.stats_history(STEPS)]


@pytest.mark.parametrize("lattice,precision,limiters", [
    (lbm.D2Q9, lbm.FP32, 0), (lbm.D2Q9, lbm.FP32, lbm.LIM_EHRENFEST), (lbm.D2Q9, lbm.FP64, 0), (lbm.D2Q9, lbm.FP16, 0),
    (lbm.D1Q3, lbm.FP32, 0), (lbm.D1Q3, lbm.FP64, lbm.LIM_EHRENFEST)])
def test_status_of_each_record_is_its_own(lattice, precision, limiters):
    if lattice == lbm.D2Q9:
        nx, ny, other, beta = 80, 60, lbm.KERNEL_TILED, 0.99999
        f = rand_state(9, ny, nx, 5, eps=0.7)
    else:
        nx, ny, other, beta = 700, 1, lbm.KERNEL_TUBE, 1 - 1e-9
        f = np.array([2 / 3, 1 / 6, 1 / 6])[:, None, None] * inputs.shock_tube(nx, 1.0, 0.2)[0][None, None, :]
    cfg = dict(lattice=lattice, nx=nx, ny=ny, boundary=lbm.BC_WALLS, precision=precision, beta=beta, u_lid=0.1,
               limiters=limiters, delta_ehrenfest=1e3, k_max=1)
    want = records(f, kernel=other, **cfg)
    first = next(i for i, (_, bad, _) in enumerate(want) if bad)
    assert first > 1
    assert [s for _, _, s in want] == [0] * first + [lbm.ERR_NONFINITE] * (STEPS - first)
    for _ in range(5):
        assert records(f, **cfg) == want
