"""FP32 tubes around the edges of the tube kernel's chunks of 128 sites.

A chunk on which nothing acts is finished at once; the chunks with the tube's
ends, with limited sites or with candidates take another way for those sites.
Both, alone and batched (groups of 8 chunks), give the populations and counts
of the tiled kernel bit for bit.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

E, EM, PEM = lbm.LIM_EHRENFEST, lbm.LIM_EHRENFEST | lbm.LIM_MEDIAN, 7
COUNTS = ("n_pos", "n_med", "n_ehr", "n_cand", "n_bad")


def _cfg(nx, lim, boundary, **kw):
    return dict(lattice=lbm.D1Q3, nx=nx, ny=1, boundary=boundary, precision=lbm.FP32, beta=0.999, limiters=lim,
                delta_median=1e-5, delta_ehrenfest=1e-6, k_max=9, **kw)


def _ic(nx):
    rho, ux = inputs.shock_tube(nx)
    rng = np.random.default_rng(nx)
    at = rng.integers(0, nx, 12)
    at[:4] = [0, nx - 1, nx // 2, (nx // 128) * 128 % nx]
    rho = np.array(rho, dtype=np.float64)
    rho[at] *= 1.0 + 0.02 * rng.standard_normal(12)
    return rho, ux, None


# V = 4 from 19457 sites; multiples of 128 and one site about them
@pytest.mark.parametrize("nx", [19583, 19584, 19585, 20481])
@pytest.mark.parametrize("boundary", [lbm.BC_WALLS, lbm.BC_PERIODIC])
@pytest.mark.parametrize("lim", [0, E, EM, PEM])
def test_lone_chunks_match_tiled(nx, boundary, lim):
    a = lbm.Lattice(**_cfg(nx, lim, boundary, kernel=lbm.KERNEL_TUBE))
    b = lbm.Lattice(**_cfg(nx, lim, boundary, kernel=lbm.KERNEL_TILED))
    for g in (a, b):
        g.init(*_ic(nx))
        g.step(25)
    np.testing.assert_array_equal(a.get_populations(), b.get_populations())
    sa, sb = a.stats(), b.stats()
    assert all(sa[k] == sb[k] for k in COUNTS)
    assert abs(sa["mass"] - sb["mass"]) <= 1e-9 * sb["mass"]


@pytest.mark.parametrize("lim", [0, E, PEM])
def test_batched_chunks_match_tiled(lim):
    sizes = [3, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025, 1152, 1153, 2048, 2049]
    batch = lbm.Batch()
    slots = []
    for nx in sizes:
        slots.append(batch.add(**_cfg(nx, lim, lbm.BC_WALLS)))
        batch.init(slots[-1], *_ic(nx))
    batch.step(25)
    batch.synchronize()
    for nx, s in zip(sizes, slots):
        g = lbm.Lattice(**_cfg(nx, lim, lbm.BC_WALLS, kernel=lbm.KERNEL_TILED))
        g.init(*_ic(nx))
        g.step(25)
        np.testing.assert_array_equal(batch.get_populations(s), g.get_populations(), err_msg=f"nx {nx}")
        sa, sb = batch.stats(s), g.stats()
        assert all(sa[k] == sb[k] for k in COUNTS), nx
