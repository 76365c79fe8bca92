"""Where the FP32 dS of a candidate stands for its FP64 key (csrc/select.cuh).

The one-block tail leaves a candidate without its FP64 key when its FP32 dS says
that it cannot be among the k largest, which supposes the two within 1/64 of
one another.  The tail supposes it only for polynomial f*, delta of at least
rho_ref / 16384, every f*_k of at least rho_ref / 256 and rho of at most 2 rho_ref.

A numpy model of the FP32 evaluation (the kernels' operations and order on the
deviations; fused multiply-adds as products rounded apart, so the model rounds
more often) against FP64 from the same stored values, on random states up to
these limits: well within 1/64.  Outside them it is not: both kinds of state for
which the tail evaluates every key break the 1/64.
"""
import numpy as np
import pytest

W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
F = np.float32


def feq(rho, ux, uy):
    usq = ux * ux + uy * uy
    c = [0 * ux, ux, uy, -ux, -uy, ux + uy, uy - ux, -ux - uy, ux - uy]
    return np.stack([rho * w * (1 + 3 * e + 4.5 * e * e - 1.5 * usq) for w, e in zip(W9, c)])


def flow_of_least(least):
    """rho and u at which f*_4 has the given value near zero and the others are above 0.005."""
    return np.ones_like(least), np.full_like(least, 0.5), (3 - np.sqrt(9 - 12 * (0.625 - 9 * least))) / 6


def key64(g):
    f = g.astype(np.float64) + W9[:, None]
    rho = f.sum(0)
    ux = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8]) / rho
    uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / rho
    fs = feq(rho, ux, uy)
    return ((f - fs) ** 2 / fs).sum(0), fs, rho


def ds32(g):
    drho = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8]
    rho = F(1) + drho
    inv = F(1) / rho
    ux = (((g[1] - g[3]) + (g[5] - g[6])) + (g[8] - g[7])) * inv
    uy = (((g[2] - g[4]) + (g[5] + g[6])) - (g[7] + g[8])) * inv
    m = F(-1.5) * (ux * ux + uy * uy)
    gs = [None] * 9
    for w, b, c, k, o in ((F(1 / 9), F(1 / 3), ux, 1, 3), (F(1 / 9), F(1 / 3), uy, 2, 4),
                          (F(1 / 36), F(1 / 12), ux + uy, 5, 7), (F(1 / 36), F(1 / 12), uy - ux, 6, 8)):
        e = F(4.5) * c * c + m
        a, odd = w * (rho * e + drho), b * rho * c
        gs[k], gs[o] = a + odd, a - odd
    gs[0] = drho - (((gs[1] + gs[2]) + (gs[3] + gs[4])) + ((gs[5] + gs[6]) + (gs[7] + gs[8])))
    n = [g[k] - gs[k] for k in range(9)]
    rm = ((n[0] + n[1]) + (n[2] + n[3])) + ((n[4] + n[5]) + (n[6] + n[7])) + n[8]
    hx = F(0.5) * (((n[1] - n[3]) + (n[5] - n[6])) + (n[8] - n[7]))
    hy = F(0.5) * (((n[2] - n[4]) + (n[5] + n[6])) - (n[7] + n[8]))
    n[0], n[1], n[3], n[2], n[4] = n[0] - rm, n[1] - hx, n[3] + hx, n[2] - hy, n[4] + hy
    return sum(n[k] * n[k] / (F(W9[k]) + gs[k]) for k in range(9))


def states(seed, n, umax, noise):
    """rho in (0.05, 2), u up to umax, deviations from f* of the given size (FP32, as stored)."""
    r = np.random.default_rng(seed)
    rho, speed, at = r.uniform(0.05, 2, n), umax * np.sqrt(r.uniform(0, 1, n)), r.uniform(0, 2 * np.pi, n)
    f = feq(rho, speed * np.cos(at), speed * np.sin(at))
    f += noise(r, n) * r.uniform(-1, 1, (9, n)) * W9[:, None]
    return (f - W9[:, None]).astype(F)


@pytest.mark.parametrize("seed", range(4))
def test_fp32_value_stands_for_the_key_within_the_limits(seed):
    g = states(seed, 400000, 0.6, lambda r, n: 10.0 ** r.uniform(-3, 0, n))
    key, fs, rho = key64(g)
    on = (fs.min(0) >= 1 / 256) & (rho <= 2) & (key >= 1 / 16384) & np.isfinite(key)
    assert np.count_nonzero(on) > 50000
    assert np.count_nonzero(on & (key < 1e-3)) > 3000 and np.count_nonzero(on & (fs.min(0) < 1 / 128)) > 1000
    assert np.abs(ds32(g)[on] / key[on] - 1).max() < 1 / 256


def test_it_does_not_outside_them():
    g = states(9, 400000, 0.2, lambda r, n: np.full(n, 1e-7))  # near equilibrium: dS of rounding noise
    key, fs, rho = key64(g)
    on = fs.min(0) >= 1 / 256
    assert np.abs(ds32(g)[on] / key[on] - 1).max() > 1 / 64
    # f*_4 near zero; n = s (e_2 + e_4 - 2 e_0) leaves the moments alone
    least = 10.0 ** np.random.default_rng(3).uniform(-6.5, -4, 200000)
    f = feq(*flow_of_least(least))
    f += np.sqrt(0.05 * least) * np.array([-2, 0, 1, 0, 1, 0, 0, 0, 0])[:, None]
    g = (f - W9[:, None]).astype(F)
    key, fs, rho = key64(g)
    on = fs.min(0) > 2e-7
    assert np.count_nonzero(on) > 100000
    assert np.abs(ds32(g)[on] / key[on] - 1).max() > 1 / 64
