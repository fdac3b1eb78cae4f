"""Simulations on several streams of one device. Launches of many steps hold the
SMs of their whole grid, so they are taken while the grids of all streams fit side
by side; beyond, steps are launched one by one and the streams' kernels overlap.
The results are the same bits either way."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def make(width, height, i, stream=None, **kw):
    from paper_2303_02210_gb300.lbm import Simulation
    return Simulation(wl.base_params(width=width, height=height, front_row=60.0, growth_mode="bulk", growth_rate=1e-3,
                                     wall_mode="advance", wall_min_gap=30.0, seed=3, sim_id=i), stream=stream, **kw)


def launches(sim, n):
    """Kernels launched by one call of n steps."""
    before = sim.stats()["launches"]
    sim.step(n)
    return sim.stats()["launches"] - before


def check(sims, width, height):
    for i, s in enumerate(sims):
        r = make(width, height, i, update_kernel="plain")
        r.step(s.stats()["step"])
        assert np.array_equal(r.pops(), s.pops())
        assert np.array_equal(r.mask(), s.mask())
        assert r.stats()["div_total"] == s.stats()["div_total"]
        r.close()


def test_small_grids_run_side_by_side():
    import torch
    sims = [make(128, 256, i, torch.cuda.Stream()) for i in range(8)]
    for _ in range(5):
        for s in sims:
            s.step(40)
    assert all(launches(s, 9) == 1 for s in sims)
    check(sims, 128, 256)
    for s in sims:
        s.close()


def test_grids_that_do_not_fit_step_by_step():
    import torch
    sims = [make(2048, 640, i, torch.cuda.Stream()) for i in range(3)]
    for _ in range(5):
        for s in sims:
            s.step(10)
    assert all(launches(s, 9) == 18 for s in sims)
    check(sims, 2048, 640)
    # one left, and one more on its stream (the two take turns): many steps a launch again
    for s in sims[1:]:
        s.close()
    assert launches(sims[0], 9) == 1
    t = make(2048, 640, 7, sims[0].stream)
    assert launches(sims[0], 9) == launches(t, 9) == 1
    sims[0].close()
    t.close()


def test_a_batch_shares_the_device():
    import torch
    from paper_2303_02210_gb300.lbm import Batch
    with torch.cuda.stream(torch.cuda.Stream()):
        members = [make(256, 256, i) for i in range(4)]
        batch = Batch(members)
    s = make(128, 256, 0, torch.cuda.Stream())
    for _ in range(4):
        batch.step(12)
        s.step(12)
    assert launches(s, 9) == 18
    check([s], 128, 256)
    check(members, 256, 256)
    batch.close()
    assert launches(s, 9) == 1
    s.close()
    for m in members:
        m.close()
