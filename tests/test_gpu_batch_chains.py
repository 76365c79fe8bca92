"""Batches whose fused lattices fall into several chains of launches.

A limiter class with 2^20 sites or more has its own chain and kernel; the other
classes share the general one, and tubes and channel-like lattices run beside
them.  Every lattice evolves bit for bit as it does alone, on either side of
that line, with and without graph replay, and after members leave.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

P, E, M = lbm.LIM_POSITIVITY, lbm.LIM_EHRENFEST, lbm.LIM_MEDIAN


def _cfg(nx, ny, lim, boundary=lbm.BC_WALLS, lattice=lbm.D2Q9):
    return dict(lattice=lattice, nx=nx, ny=ny, boundary=boundary, precision=lbm.FP32, beta=0.97, u_lid=0.08,
                limiters=lim, delta_median=1e-5, delta_ehrenfest=1e-4, k_max=max(1, nx * ny // 5000))


# the class sizes: exactly 2^20 sites (own chain), one row less (general chain)
MIXES = {
    "line": [(1024, 1024, E), (1024, 1023, M | E), (100, 75, P)],
    "all_classes": [(1030, 1021, M), (1024, 1024, P | E), (700, 800, E), (900, 700, 0), (1100, 960, P | M | E)],
    "mixed": [(1024, 1024, M), (64, 300, P | E), (90, 40, P | M | E), (3000, 1, P | M | E)],
}


@pytest.mark.parametrize("graph", [0, 4])
@pytest.mark.parametrize("mix", sorted(MIXES))
def test_chains_match_lone_runs(mix, graph):
    cfgs = []
    for nx, ny, lim in MIXES[mix]:
        if ny == 1:
            cfgs.append(_cfg(nx, ny, lim, lattice=lbm.D1Q3))
        else:
            cfgs.append(_cfg(nx, ny, lim, lbm.BC_PERIODIC if ny == 40 else lbm.BC_WALLS))

    def ic(i):
        c = cfgs[i]
        if c["lattice"] == lbm.D1Q3:
            rho, ux = inputs.shock_tube(c["nx"])
            return rho, ux, None
        return inputs.random_moments(i, c["nx"], c["ny"], umax=0.06)

    steps = 11
    alone = []
    for i, c in enumerate(cfgs):
        g = lbm.Lattice(**c)
        g.init(*ic(i))
        g.step(steps)
        mid = g.get_populations(), g.stats()
        g.step(2)
        alone.append((mid, g.get_populations()))
    b = lbm.Batch()
    slots = [b.add(**c) for c in cfgs]
    for i, s in enumerate(slots):
        b.init(s, *ic(i))
    if graph:
        b.set_graph(graph)
    b.step(3)
    b.step(steps - 3)
    b.synchronize()
    for s, (mid, _) in zip(slots, alone):
        np.testing.assert_array_equal(b.get_populations(s), mid[0])
        bs = b.stats(s)
        assert all(bs[k] == mid[1][k] for k in ("step", "n_pos", "n_med", "n_ehr", "n_cand", "n_bad"))
    b.remove(slots[0])  # the chains are laid out anew
    b.step(2)
    b.synchronize()
    for s, (_, end) in list(zip(slots, alone))[1:]:
        np.testing.assert_array_equal(b.get_populations(s), end)
