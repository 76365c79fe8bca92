"""The field kernels' integer conversions and fixed-point moments (csrc/fields.cu).

set / get: the stored deviation is float(f - rho_ref W) (then the 16-bit
rounding), read back as double(g) + rho_ref W, each operation rounded once: bit
for bit, for values from zero and subnormals to far above rho_ref.  moments of
FP32 / 16-bit storage: within one rounding of the sums of the stored values in
extended precision (rho and rho u: half an ulp of FP64 plus 2^-58 per population;
u: two more roundings), ordinary deviations and those at or above rho_ref (the
FP64 formula, nine roundings) alike.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import lbm

pytestmark = pytest.mark.gpu

W = {9: np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4), 3: np.array([2 / 3, 1 / 6, 1 / 6])}


def lattice(q, nx, ny, precision, rho_ref):
    return lbm.Lattice(lattice=lbm.D2Q9 if q == 9 else lbm.D1Q3, nx=nx, ny=ny, boundary=lbm.BC_WALLS,
                       precision=precision, rho_ref=rho_ref)


def state(q, ny, nx, rho_ref, eps, seed):
    rng = np.random.default_rng(seed)
    return rho_ref * W[q][:, None, None] * (1 + eps * rng.uniform(-1, 1, (q, ny, nx)))


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32, lbm.FP16])
@pytest.mark.parametrize("q,nx,ny", [(9, 257, 3), (9, 7, 300), (3, 1001, 1)])
def test_set_get_round_as_written(q, nx, ny, precision):
    rho_ref = 2.7
    g = lattice(q, nx, ny, precision, rho_ref)
    f = state(q, ny, nx, rho_ref, 0.3, 1)
    rw = rho_ref * W[q]
    flat = f.reshape(q, -1)
    flat[:, 0] = rw                                              # deviations of exactly zero
    flat[:, 1] = rw * (1 + 2.0 ** -50)                           # one or two ulps
    flat[:, 2] = 0.0
    flat[:, 3] = -rw
    flat[:, 4] = 1e30 if precision == lbm.FP64 else 3000.0       # far above rho_ref
    flat[:, 5] = rw + 2.0 ** -25 * (1 + 2.0 ** -24)              # near a tie of the FP32 rounding
    g.set_populations(f)
    want = f
    if precision != lbm.FP64:
        dev = (f - rw[:, None, None]).astype(np.float32)
        if precision == lbm.FP16:
            dev = dev.astype(np.float16).astype(np.float32)
        want = dev.astype(np.float64) + rw[:, None, None]
    np.testing.assert_array_equal(g.get_populations().reshape(f.shape), want)


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.BF16])
@pytest.mark.parametrize("rho_ref,eps", [(1.0, 0.2), (2.7, 1e-4), (1e-3, 0.2), (300.0, 0.2), (1.0, 6.0)])
@pytest.mark.parametrize("q,nx,ny", [(9, 130, 9), (3, 999, 1)])
def test_moments_of_the_stored_values(q, nx, ny, rho_ref, eps, precision):
    g = lattice(q, nx, ny, precision, rho_ref)
    f = np.abs(state(q, ny, nx, rho_ref, eps, 2))
    g.set_populations(f)
    rw = rho_ref * W[q]
    stored = g.get_populations().reshape(q, ny, nx)
    dev = (stored - rw[:, None, None]).astype(np.float32)        # the stored deviation, exactly
    x = dev.astype(np.longdouble) + rw.astype(np.longdouble)[:, None, None]
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("no extended precision on this host")
    cx = {9: [0, 1, 0, -1, 0, 1, -1, -1, 1], 3: [0, -1, 1]}[q]
    cy = {9: [0, 0, 1, 0, -1, 1, 1, -1, -1], 3: [0, 0, 0]}[q]
    rho = x.sum(0)
    ux = sum(c * v for c, v in zip(cx, x)) / rho
    uy = sum(c * v for c, v in zip(cy, x)) / rho
    out = g.moments(check=False)
    # the FP64 formula of the fallback rounds every population and nine sums
    tol = 2.0 ** -52 * (1 if eps < 1 else 10)
    assert np.abs((out[0] - rho) / rho).max() <= tol
    # rho u is off by at most ten half-ulps of the largest population, u by two roundings more
    scale = np.abs(x).max(0) / rho
    assert (np.abs(out[1] - ux) <= tol * (6 * scale + 2 * np.abs(ux))).all()
    if q == 9:
        assert (np.abs(out[2] - uy) <= tol * (6 * scale + 2 * np.abs(uy))).all()
