"""Steps with candidates among steps without, in one resident launch.

Where a step has no Ehrenfests' candidates the resident kernel's blocks go on
without the tail, which may lag by several steps; where one has, they wait for
it.  Each step's candidates, chosen sites and record have to be its own: one
call of many steps against the same steps launch by launch, on states in which
candidates come and go.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import inputs, lbm

from test_gpu_parity import rand_state

pytestmark = pytest.mark.gpu

COUNTS = ("step", "n_pos", "n_med", "n_ehr", "n_cand", "n_bad", "status")


def one_call_and_launches(kernel, f, steps, **cfg):
    a, b = lbm.Lattice(stats_history=steps, **cfg), lbm.Lattice(kernel=kernel, stats_history=steps, **cfg)
    for g in (a, b):
        g.set_populations(f)
    n = a.launch_count()
    a.step(steps)
    assert a.launch_count() == n + 1
    b.step(steps)
    np.testing.assert_array_equal(a.get_populations(), b.get_populations())
    np.testing.assert_array_equal(a.limited_sites(), b.limited_sites())
    ha, hb = a.stats_history(steps), b.stats_history(steps)
    for x, y in zip(ha, hb):
        assert [x[k] for k in COUNTS] == [y[k] for k in COUNTS]
    some = np.array([x["n_cand"] > 0 for x in ha])
    assert np.count_nonzero(some[1:] != some[:-1]) >= 10  # they do come and go


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP64])
@pytest.mark.parametrize("nx,delta,k", [(800, 3e-3, 4), (800, 5e-3, 1), (3000, 4e-3, 2)])
def test_tube_candidates_come_and_go(nx, delta, k, precision):
    rho, _ = inputs.shock_tube(nx)
    f = np.array([2 / 3, 1 / 6, 1 / 6])[:, None, None] * rho[None, None, :]
    one_call_and_launches(lbm.KERNEL_TUBE, f, 400, lattice=lbm.D1Q3, nx=nx, ny=1, boundary=lbm.BC_WALLS,
                          precision=precision, beta=1 - 1e-9, limiters=lbm.LIM_EHRENFEST, delta_ehrenfest=delta, k_max=k)


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.BF16, lbm.FP64])
@pytest.mark.parametrize("nx,ny,heavy,delta,beta", [(64, 48, 2, 1e-3, 0.999), (96, 40, 1, 5e-4, 0.9999)])
def test_cavity_candidates_come_and_go(nx, ny, heavy, delta, beta, precision):
    one_call_and_launches(lbm.KERNEL_TILED, rand_state(9, ny, nx, 5, eps=0.0, heavy=heavy), 300, lattice=lbm.D2Q9,
                          nx=nx, ny=ny, boundary=lbm.BC_WALLS, precision=precision, beta=beta,
                          limiters=lbm.LIM_EHRENFEST, delta_ehrenfest=delta, k_max=3)
