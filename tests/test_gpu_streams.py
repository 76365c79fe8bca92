"""Small lattices on several streams.

A lattice by itself takes its steps in one launch that fills the GPU.  With live
lattices on other streams the launch is held to its share of the SMs, one round
of tiles, or the steps are launched one by one, so that the streams overlap as
they would without it.  The populations are the same whichever way, also from
threads, and the lattice has the GPU to itself again when the others are gone.
"""
import threading

import numpy as np
import pytest
import torch

from paper_0704_0043_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

STEPS = 12


def cavity(n, stream, precision=lbm.FP32):
    g = lbm.Lattice(stream=stream, lattice=lbm.D2Q9, nx=n, ny=n, boundary=lbm.BC_WALLS, precision=precision, beta=0.97,
                    u_lid=0.1, limiters=lbm.LIM_EHRENFEST | lbm.LIM_MEDIAN, delta_median=1e-4, delta_ehrenfest=1e-3,
                    k_max=5)
    g.init(*inputs.cavity_rest(n, n))
    return g


def launches(g, n):
    before = g.launch_count()
    g.step(n)
    return g.launch_count() - before


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP64])
def test_launches_follow_the_streams_in_use(precision):
    streams = [torch.cuda.Stream() for _ in range(4)]
    large, small = cavity(300, 0, precision), cavity(40, 0, precision)
    assert launches(large, 3) == 1 and launches(small, 3) == 1
    same = cavity(50, 0, precision)  # the same stream: they take turns anyway
    assert launches(large, 3) == 1
    others = [cavity(30, s.cuda_stream, precision) for s in streams]
    assert launches(large, 3) == 6  # more tiles than its share of the SMs
    assert launches(small, 3) == 1 and launches(others[0], 3) == 1
    del others, same
    assert launches(large, 3) == 1
    large.synchronize()


@pytest.mark.parametrize("threads", [False, True])
def test_populations_on_several_streams(threads):
    sizes = [40, 100, 300, 300, 150]
    want = []
    for n in sizes:
        g = cavity(n, 0)
        g.step(STEPS)
        want.append(g.get_populations())
        del g
    streams = [torch.cuda.Stream() for _ in sizes]
    gs = [cavity(n, s.cuda_stream) for n, s in zip(sizes, streams)]

    def run(g):
        for _ in range(STEPS // 4):
            g.step(4)

    if threads:
        ts = [threading.Thread(target=run, args=(g,)) for g in gs]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    else:
        for _ in range(STEPS // 4):
            for g in gs:
                g.step(4)
    for g, f in zip(gs, want):
        np.testing.assert_array_equal(g.get_populations(), f)


def test_a_long_kernel_elsewhere_does_not_hold_the_steps():
    """One block busy on another stream: the steps go on beside it, as launches of their own would."""
    large = cavity(480, 0)
    large.step(3)
    large.synchronize()
    s, done = torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(s):
        torch.cuda._sleep(int(3e9))  # a second or two
        done.record(s)
    assert launches(large, 20) == 1
    large.synchronize()
    assert not done.query()
    torch.cuda.synchronize()
