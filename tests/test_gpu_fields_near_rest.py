"""Moments of a fluid very near rest (csrc/site.cuh, FP32 storage).

Deviations of 1e-8 to 1e-11 of rho_ref end below the last place of the FP64
populations' sums.  Each is rounded once, to 2^(e - 58) with 2^e <= rho_ref, so
rho u is off by at most six half units (D1Q3: two), rho by nine (three), and
the quotients and the final values round to FP64.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import lbm

from test_gpu_fields import W, lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [1e-8, 1e-10, 1e-11])
@pytest.mark.parametrize("rho_ref", [1.0, 2.7])
@pytest.mark.parametrize("q,nx,ny", [(9, 130, 9), (3, 999, 1)])
def test_moments_very_near_rest(q, nx, ny, rho_ref, eps):
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("no extended precision on this host")
    g = lattice(q, nx, ny, lbm.FP32, rho_ref)
    rw = (rho_ref * W[q])[:, None, None]
    f = rw + eps * np.random.default_rng(4).uniform(-1, 1, (q, ny, nx))
    dev = (f - rw).astype(np.float32)  # what is stored: the difference is exact, then rounded
    g.set_populations(f)
    x = dev.astype(np.longdouble)
    cx = {9: [0, 1, 0, -1, 0, 1, -1, -1, 1], 3: [0, -1, 1]}[q]
    cy = {9: [0, 0, 1, 0, -1, 1, 1, -1, -1], 3: [0, 0, 0]}[q]
    rho = x.sum(0) + rw.astype(np.longdouble).sum()
    out = g.moments()
    half = 2.0 ** (np.floor(np.log2(rho_ref)) - 59)
    assert (np.abs(out[0] - rho) <= q * half + 2.0 ** -53 * rho).all()
    for c, got in zip((cx, cy), out[1:]):
        if not any(c):
            continue
        u = sum(a * v for a, v in zip(c, x)) / rho
        # the sum's rounding and three of the quotient
        assert (np.abs(got - u) <= sum(map(abs, c)) * half / rho + 2.0 ** -51 * np.abs(u)).all()
