"""The FP32 levels of dS_0's radix descent: exact integer sums per bin.

With the filter acting alone, sum (1 - phi^2) dS over the limited sites equals
delta_0 (1 - (2 beta - 1)^2) sum dS; phi is an FP32 square root, so each term
errs by about 1e-7 dS, which is 1e-5 of a right side of 1 % of sum dS (bound
1e-4).  Sizes: less than one block, remainders of a warp's 32 values and of a
block's round, more than one round of all blocks; amplitudes from crowded bins
to dS spread over many binades, down to rounding level.  Two runs agree exactly.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


@pytest.mark.parametrize("nx,ny", [(16, 9), (33, 31), (129, 127), (1301, 977)])
@pytest.mark.parametrize("eps", [0.15, 1e-2, 1e-4])
def test_filter_alone_meets_the_threshold_equation(nx, ny, eps):
    runs = []
    for _ in range(2):
        g = lbm.Lattice(lattice=lbm.D2Q9, nx=nx, ny=ny, boundary=lbm.BC_PERIODIC, beta=0.95, limiters=lbm.LIM_ENTTHRESH,
                        entthresh_delta0=0.1, precision=lbm.FP32)
        f = inputs.random_populations(7, 9, ny, nx, W9, eps)
        # amplitudes falling along y: dS over many binades
        w = W9[:, None, None]
        f = w + (f - w) * (2.0 ** -(np.arange(ny) % 12))[None, :, None]
        g.set_populations(f)
        g.step(1)
        st = g.stats()
        np.testing.assert_allclose(st["dS_lim"], 0.1 * (1 - 0.9 * 0.9) * st["sum_dS"], rtol=1e-4)
        runs.append((g.get_populations(), st))
    np.testing.assert_array_equal(runs[0][0], runs[1][0])
    assert runs[0][1] == runs[1][1]
