"""The field kernels on lattices from one column to one row.

A site's row is its index times a reciprocal of nx: every site of widths of one,
of powers of two and their neighbours, and of lattices taller than a grid's y
dimension goes to its own place (init, set, get, moments).
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import lbm

from test_gpu_fields import W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 70001), (2, 66000), (3, 40000), (7, 9), (8, 1000), (31, 33), (33, 31),
                                   (255, 3), (257, 5), (4099, 2), (70001, 1)])
def test_every_site_has_its_place(nx, ny, precision):
    g = lbm.Lattice(lattice=lbm.D2Q9, nx=nx, ny=ny, boundary=lbm.BC_PERIODIC, precision=precision)
    w = W[9][:, None, None]
    f = w * (1 + 0.1 * np.random.default_rng(nx).uniform(-1, 1, (9, ny, nx)))
    want = f if precision == lbm.FP64 else (f - w).astype(np.float32).astype(np.float64) + w
    g.set_populations(f)
    np.testing.assert_array_equal(g.get_populations(), want)
    rho, ux, uy = (want.sum(0), (want[1] - want[3] + want[5] - want[6] - want[7] + want[8]) / want.sum(0),
                   (want[2] - want[4] + want[5] + want[6] - want[7] - want[8]) / want.sum(0))
    for a, b in zip(g.moments(), (rho, ux, uy)):
        np.testing.assert_allclose(a.reshape(ny, nx), b, rtol=0, atol=1e-14)
    g.init(rho, ux, uy)
    usq = ux * ux + uy * uy
    c = [0 * ux, ux, uy, -ux, -uy, ux + uy, uy - ux, -ux - uy, ux - uy]
    fs = np.stack([rho * v * (1 + 3 * e + 4.5 * e * e - 1.5 * usq) for v, e in zip(W[9], c)])
    np.testing.assert_allclose(g.get_populations(), fs, rtol=0, atol=1e-14 if precision == lbm.FP64 else 1e-8)
