"""The key queue of the dense-candidate preselection at its fullest.

With k above the number of candidates every one of them is queued for its FP64
key, so each block's queue fills in every round of the grid tail and is drained
a block's worth at a time; with k a third of them it fills every few rounds.
No candidate may be lost or keyed twice: the count of valid candidates and the
chosen sites are the oracle's.
"""
import numpy as np
import pytest

import oracle
from paper_0704_0043_gb300 import lbm

from test_gpu_parity import pair, rand_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("part", [1.0, 0.33])
def test_queue_fills_in_every_round(part):
    n = 1024
    k = int(part * n * n)
    g, oc = pair(lattice=lbm.D2Q9, nx=n, ny=n, boundary=lbm.BC_WALLS, beta=0.99, u_lid=0.05, precision=lbm.FP32,
                 limiters=lbm.LIM_EHRENFEST, delta_ehrenfest=1e-3, k_max=k)
    g.set_populations(rand_state(9, n, n, 1301, eps=0.2))
    f = g.get_populations()
    g.step(1)
    r = oracle.step(oc, f)
    st = g.stats(check=False)
    assert st["n_cand"] == r.stats["n_cand"] > n * n // 2
    assert st["n_ehr"] == min(k, r.stats["n_cand"])
    np.testing.assert_array_equal(g.limited_sites(), np.sort(r.selected))
