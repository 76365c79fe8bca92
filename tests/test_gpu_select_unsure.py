"""Ehrenfests' selection where the FP32 dS does not stand for the FP64 key.

The fused kernel keys up to 32 candidates of a work item and leaves the rest to
the tail, which spares those that their FP32 dS rules out.  Near a zero of some
f*_k, at thresholds near the rounding noise of dS, and with entropic f* the FP32
dS may be off by more than the margin of that rule.  The chosen sites and the
count are those of the tiled kernel, which keys every candidate where it
finds it; candidates above and below what the tail holds in shared memory.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import inputs, lbm

from test_gpu_parity import W9, rand_state
from test_select_premise import CX, CY, feq, flow_of_least

pytestmark = pytest.mark.gpu

SHAPES = [(300, 200, 0.15), (50, 36, 0.4)]


def same_choice(f, nx, ny, steps=1, **cfg):
    a, b = (lbm.Lattice(lattice=lbm.D2Q9, nx=nx, ny=ny, boundary=lbm.BC_WALLS, precision=lbm.FP32,
                        limiters=lbm.LIM_EHRENFEST, kernel=k, **cfg) for k in (lbm.KERNEL_FUSED, lbm.KERNEL_TILED))
    for g in (a, b):
        g.set_populations(f)
        g.step(steps)
    sa, sb = a.stats(check=False), b.stats(check=False)
    assert sa["n_cand"] == sb["n_cand"] > cfg["k_max"]
    np.testing.assert_array_equal(a.limited_sites(), b.limited_sites())


@pytest.mark.parametrize("nx,ny,part", SHAPES)
def test_some_feq_near_zero(nx, ny, part):
    r = np.random.default_rng(1)
    least = 10.0 ** r.uniform(-6.9, -6.2, (ny, nx))
    arrives = feq(*flow_of_least(least))
    ghost = np.array([-2, 0, 1, 0, 1, 0, 0, 0, 0])[:, None, None]  # leaves the moments alone
    arrives += np.sqrt(least * r.uniform(0.048, 0.052, least.shape)) * ghost
    f = np.stack([np.roll(arrives[k], (-CY[k], -CX[k]), (0, 1)) for k in range(9)])  # before free flight
    same_choice(f, nx, ny, beta=0.99, delta_ehrenfest=1e-3, k_max=int(part * nx * ny))


@pytest.mark.parametrize("nx,ny,part", SHAPES)
@pytest.mark.parametrize("delta", [0.0, 1e-18])
def test_threshold_near_the_noise_of_ds(nx, ny, part, delta):
    x, y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny)
    ux, uy = 0.1 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y), -0.1 * np.cos(2 * np.pi * x) * np.sin(2 * np.pi * y)
    arrives = feq(1 + 0.01 * np.cos(2 * np.pi * x), ux, uy)
    f = np.stack([np.roll(arrives[k], (-CY[k], -CX[k]), (0, 1)) for k in range(9)])
    same_choice(f, nx, ny, beta=0.99, delta_ehrenfest=delta, k_max=int(part * nx * ny))


@pytest.mark.parametrize("nx,ny,part", SHAPES)
def test_entropic_populations_around_zero(nx, ny, part):
    """f' = 0 up to FP32 rounding in one population of every second site: the key is
    finite or +inf, whichever the FP32 value."""
    r = np.random.default_rng(2)
    f = rand_state(9, ny, nx, 3, eps=0.1)
    a = 2 * 0.99 - 1
    rho = f.sum(0)
    u = [(np.array(c)[:, None, None] * f).sum(0) / rho for c in (CX, CY)]
    s = [np.sqrt(1 + 3 * v * v) for v in u]
    ax = [{0: 2 - q, 1: (2 - q) * (2 * v + q) / (1 - v), -1: (2 - q) * (1 - v) / (2 * v + q)} for v, q in zip(u, s)]
    fs = np.stack([rho * W9[k] * ax[0][CX[k]] * ax[1][CY[k]] for k in range(9)])
    n = f - fs
    ghost = np.array([-2, 1, 0, 1, 0, 0, 0, 0, 0])[:, None, None]
    t = fs[3] / a - n[3]  # n_3 + t = f*_3 / a: f'_3 = f*_3 - a n_3 = 0
    arrives = f + np.where(r.random((ny, nx)) < 0.5, t, 0.0) * ghost
    g = np.stack([np.roll(arrives[k], (-CY[k], -CX[k]), (0, 1)) for k in range(9)])
    same_choice(g, nx, ny, beta=0.99, delta_ehrenfest=1e-3, k_max=int(part * nx * ny), equilibrium=lbm.EQ_ENTROPIC)
