"""The resident kernel: many steps of a small lattice in one launch.

With the default kernel choice a small lattice takes its steps in the resident
kernel; an explicit choice (fused, tiled, tube) takes them launch by launch.
Both run the same per-site operations, so the populations and the Ehrenfests'
sites are the same bit for bit, the counts equal, and the sums equal to the
rounding of their other grouping.  Shapes with one tile, ragged tiles, several
tiles a block; every boundary; candidates from none to most sites (more than
the tail keys alone, more than it holds in shared memory); calls split anyhow.
"""
import numpy as np
import pytest

from paper_0704_0043_gb300 import inputs, lbm

from test_gpu_parity import rand_state

pytestmark = pytest.mark.gpu

ALL = lbm.LIM_POSITIVITY | lbm.LIM_EHRENFEST | lbm.LIM_MEDIAN


def both(kernel, f, steps, **cfg):
    """The same steps resident (in calls of different lengths) and launch by launch."""
    a, b = lbm.Lattice(stats_history=3, **cfg), lbm.Lattice(kernel=kernel, stats_history=3, **cfg)
    for g in (a, b):
        g.set_populations(f)
    n = a.launch_count()
    a.step(1)
    a.step(steps - 1)
    assert a.launch_count() == n + (1 if steps == 1 else 2)  # one launch a call
    for _ in range(steps):
        b.step(1)
    np.testing.assert_array_equal(a.get_populations(), b.get_populations())
    np.testing.assert_array_equal(a.limited_sites(), b.limited_sites())
    tol = 1e-12 if cfg["precision"] == lbm.FP64 else 1e-6
    for x, y in zip(a.stats_history(3), b.stats_history(3)):
        for key in ("step", "n_pos", "n_med", "n_ehr", "n_cand", "n_bad", "status"):
            assert x[key] == y[key], (key, x, y)
        for key in ("mass", "sum_dS", "dS_lbgk", "dS_lim"):
            assert abs(x[key] - y[key]) <= tol * abs(y[key]) + 1e-300, (key, x[key], y[key])
    return a, b


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP64, lbm.BF16, lbm.FP16])
@pytest.mark.parametrize("nx,ny", [(5, 5), (32, 8), (33, 17), (257, 130), (700, 300)])
@pytest.mark.parametrize("boundary", [lbm.BC_WALLS, lbm.BC_PERIODIC, lbm.BC_CHANNEL, lbm.BC_NODE_WALLS,
                                      lbm.BC_DIFFUSIVE])
def test_d2q9_resident_equals_launches(boundary, nx, ny, precision):
    if nx * ny > 100000 and boundary in (lbm.BC_PERIODIC, lbm.BC_DIFFUSIVE):
        pytest.skip("one large shape per wall kind is enough")
    a, _ = both(lbm.KERNEL_TILED, rand_state(9, ny, nx, 7 + nx, eps=0.05, heavy=3), 6, lattice=lbm.D2Q9, nx=nx, ny=ny,
                boundary=boundary, precision=precision, beta=0.97, u_lid=0.1, limiters=ALL, delta_median=1e-4,
                delta_ehrenfest=2e-3, k_max=7)
    assert a.stats(check=False)["n_med"] > 0 or nx * ny < 200


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP64])
@pytest.mark.parametrize("nx,boundary", [(3, lbm.BC_WALLS), (128, lbm.BC_PERIODIC), (129, lbm.BC_WALLS),
                                         (5003, lbm.BC_PERIODIC), (200001, lbm.BC_WALLS)])
def test_d1q3_resident_equals_launches(nx, boundary, precision):
    rho, _ = inputs.shock_tube(nx)
    w = np.array([2 / 3, 1 / 6, 1 / 6])
    f = w[:, None, None] * rho[None, None, :] * (1 + 0.01 * np.random.default_rng(nx).uniform(-1, 1, (3, 1, nx)))
    both(lbm.KERNEL_TUBE, f, 9, lattice=lbm.D1Q3, nx=nx, ny=1, boundary=boundary, precision=precision, beta=0.999,
         limiters=ALL, delta_median=1e-5, delta_ehrenfest=1e-4, k_max=4)


@pytest.mark.parametrize("k_max", [0, 1, 20, 700, 100000])
@pytest.mark.parametrize("eps,heavy", [(0.0, 5), (0.0, 40), (0.02, 300), (0.15, 300)])
@pytest.mark.parametrize("kernel", [lbm.KERNEL_FUSED, lbm.KERNEL_TILED])
def test_candidates_from_a_few_to_most_sites(kernel, eps, heavy, k_max):
    """A few candidates (keyed by the tail), dozens (by every block), thousands
    (more than the tail's shared memory holds)."""
    nx, ny = 300, 200
    _, b = both(kernel, rand_state(9, ny, nx, 3, eps=eps, heavy=heavy), 3, lattice=lbm.D2Q9, nx=nx, ny=ny,
                boundary=lbm.BC_WALLS, precision=lbm.FP32, beta=0.99, u_lid=0.05,
                limiters=lbm.LIM_EHRENFEST | lbm.LIM_MEDIAN, delta_median=1e-3, delta_ehrenfest=1e-3, k_max=k_max)
    assert b.stats(check=False)["n_cand"] > 0


def test_timed_steps_among_resident_ones():
    """Steps sampled by lbm_timing are launched on their own; the others stay resident."""
    cfg = dict(lattice=lbm.D2Q9, nx=90, ny=70, boundary=lbm.BC_WALLS, precision=lbm.FP32, beta=0.97, u_lid=0.1,
               limiters=ALL, delta_median=1e-4, delta_ehrenfest=1e-3, k_max=5)
    a, b = lbm.Lattice(**cfg), lbm.Lattice(**cfg)
    for g in (a, b):
        g.init(*inputs.cavity_rest(90, 70))
    a.timing(True, every=4)
    a.step(13)
    assert a.timing_read()[2] == 4
    b.step(13)
    np.testing.assert_array_equal(a.get_populations(), b.get_populations())


@pytest.mark.parametrize("limiters", [0, lbm.LIM_POSITIVITY, lbm.LIM_MEDIAN, lbm.LIM_POSITIVITY | lbm.LIM_MEDIAN])
@pytest.mark.parametrize("nx,ny", [(5, 32), (32, 33), (100, 100), (128, 128), (250, 50), (17, 300)])
@pytest.mark.parametrize("boundary", [lbm.BC_WALLS, lbm.BC_PERIODIC, lbm.BC_CHANNEL, lbm.BC_NODE_WALLS,
                                      lbm.BC_DIFFUSIVE])
def test_cluster_equals_launches(boundary, nx, ny, limiters):
    """The smallest lattices without Ehrenfests' steps run as one cluster: bands of
    two rows and more, ragged bands, several sites a thread, medians at the bands'
    edges (every row is out of equilibrium) and several to a thread."""
    both(lbm.KERNEL_TILED, rand_state(9, ny, nx, 11 + nx, eps=0.05, heavy=2), 7, lattice=lbm.D2Q9, nx=nx, ny=ny,
         boundary=boundary, precision=lbm.FP32, beta=0.97, u_lid=0.1, limiters=limiters, delta_median=1e-4, k_max=0)


def test_cluster_records_the_control_point():
    """Probe samples of the cluster are the moments after each step."""
    nx, ny = 50, 40
    g = lbm.Lattice(lattice=lbm.D2Q9, nx=nx, ny=ny, boundary=lbm.BC_DIFFUSIVE, precision=lbm.FP32, beta=0.95, u_lid=0.1,
                    limiters=lbm.LIM_MEDIAN, delta_median=1e-4)
    g.init(*inputs.cavity_rest(nx, ny))
    g.probe(33 * nx + 3, 8)
    want = []
    for n in (1, 3, 2):
        g.step(n)
        want.append(tuple(a[33, 3] for a in g.moments()))
    got = g.probe_read(8)
    np.testing.assert_array_equal(got[[0, 3, 5]], np.array(want))
