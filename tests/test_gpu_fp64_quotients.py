"""The FP64 step's shared-reciprocal quotients (csrc/lattice.cuh).

A quotient is taken from a reciprocal and settled by its exact residual; where an
operand lies outside 2^-500 .. 2^499 (or the quotient is a power of two with a
residual), the site is evaluated again with IEEE divisions.  Both ways give the bits of the plain
division, so FP64 populations and dS must equal the oracle's at every scale:
the step is homogeneous of degree one, and scaling a state by a power of two
moves its quotients from the fast path (scale 1, 2^200) to the general one
(2^-480, 2^490), and through the border (2^-245: dS terms near 2^-500).
"""
import numpy as np
import pytest

import oracle
from paper_0704_0043_gb300 import lbm

from test_gpu_parity import pair, rand_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [0, 200, -245, -480, 490])
@pytest.mark.parametrize("q,ny,nx", [(9, 13, 37), (3, 1, 301)])
def test_fp64_step_equals_oracle_at_every_scale(q, ny, nx, exponent):
    scale = 2.0 ** exponent
    g, oc = pair(lattice=lbm.D2Q9 if q == 9 else lbm.D1Q3, nx=nx, ny=ny, boundary=lbm.BC_WALLS, beta=0.97,
                 u_lid=0.1 if q == 9 else 0.0, rho_wall=scale, precision=lbm.FP64,
                 limiters=lbm.LIM_POSITIVITY | lbm.LIM_EHRENFEST | lbm.LIM_MEDIAN, delta_median=1e-4 * scale,
                 delta_ehrenfest=2e-3 * scale, k_max=5)
    f = rand_state(q, ny, nx, 77) * scale
    # a patch at rest (dS terms exactly zero) and one whose velocity is a power of two
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4) if q == 9 else np.array([2 / 3, 1 / 6, 1 / 6])
    f[:, :, 2:9] = (w * scale)[:, None, None]
    f[1, :, 12:18] = f[1, :, 12:18].mean()
    # and one at rest up to an ulp or two: quotients next to rounding boundaries
    f[:, :, 20:30] = np.nextafter(f[:, :, 2:3], [[[0.0]], [[np.inf]], [[0.0]]] * (q // 3))
    g.set_populations(f)
    for _ in range(3):
        r = oracle.step(oc, f)
        g.step(1)
        got = g.get_populations()
        assert np.array_equal(got, r.f.reshape(got.shape))
        f = r.f
    np.testing.assert_array_equal(g.limited_sites(), np.sort(r.selected))
