"""CUDA-graph replay of a lone lattice (lbm_set_graph).

Lattices that are stepped launch by launch: above the resident kernel's size,
entropic f*, an ensemble-dependent limiter, an explicit kernel.  Runs of steps
replayed from a graph, with plain steps before, between and after (from either
buffer), give the populations, chosen sites and records of plain steps.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import lbm

from test_gpu_parity import rand_state

pytestmark = pytest.mark.gpu

EHR_MED = lbm.LIM_EHRENFEST | lbm.LIM_MEDIAN
CASES = {
    "fused": dict(nx=600, ny=500, precision=lbm.FP32, limiters=EHR_MED),
    "fused16": dict(nx=500, ny=600, precision=lbm.BF16, limiters=lbm.LIM_EHRENFEST),
    "entropic": dict(nx=64, ny=48, precision=lbm.FP32, limiters=EHR_MED, equilibrium=lbm.EQ_ENTROPIC),
    "threshold": dict(nx=64, ny=48, precision=lbm.FP32, limiters=lbm.LIM_EHRENFEST | lbm.LIM_THRESHOLD),
    "entthresh": dict(nx=70, ny=40, precision=lbm.FP32, limiters=lbm.LIM_ENTTHRESH),
    "tiled64": dict(nx=40, ny=70, precision=lbm.FP64, limiters=EHR_MED, kernel=lbm.KERNEL_TILED),
    "tube": dict(nx=(1 << 20) + 5, ny=1, precision=lbm.FP32, limiters=lbm.LIM_EHRENFEST, lattice=lbm.D1Q3),
}


@pytest.mark.parametrize("name", CASES)
def test_replayed_steps_are_plain_steps(name):
    cfg = dict(dict(lattice=lbm.D2Q9, boundary=lbm.BC_WALLS, beta=0.97, delta_median=1e-4, delta_ehrenfest=1e-3, k_max=9,
                    stats_history=32), **CASES[name])
    if cfg["lattice"] == lbm.D2Q9:
        cfg["u_lid"] = 0.1
    f = rand_state(9 if cfg["lattice"] == lbm.D2Q9 else 3, cfg["ny"], cfg["nx"], 41, eps=0.03, heavy=3)
    a, b = lbm.Lattice(**cfg), lbm.Lattice(**cfg)
    a.set_graph(4)
    for g in (a, b):
        g.set_populations(f)
    for n in (1, 11, 2, 8, 5):
        a.step(n)
        b.step(n)
        np.testing.assert_array_equal(a.get_populations(), b.get_populations())
        np.testing.assert_array_equal(a.limited_sites(), b.limited_sites())
    assert a.launch_count() == b.launch_count()
    for x, y in zip(a.stats_history(27), b.stats_history(27)):
        assert {k: x[k] for k in x if k.startswith("n_") or k in ("step", "status")} == \
            {k: y[k] for k in y if k.startswith("n_") or k in ("step", "status")}
        for k in ("mass", "sum_dS", "dS_lbgk", "dS_lim"):
            assert abs(x[k] - y[k]) <= 1e-12 * abs(y[k]) + 1e-300, k
    a.set_graph(0)
    a.step(3)
    b.step(3)
    np.testing.assert_array_equal(a.get_populations(), b.get_populations())
