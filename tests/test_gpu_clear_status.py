"""``lbm_clear_status`` between the steps of a healthy, growing run changes
nothing but the sticky bits: the divisions already selected for the coming step
are applied, those of the latest step stay listed, and the run goes on bit for
bit as one that was not cleared, in every form of the update."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

FORMS = [
    # lattice, precision, update kernel, steps per call (1: the step-by-step launches)
    ("d2q9", "fp32", "plain", 1),
    ("d2q9", "fp32", "tma", 1),
    ("d2q9", "fp32", "tma_sel", 1),
    ("d2q9", "fp32", "tma_st", 1),
    ("d2q9", "fp32", "auto", 7),
    ("d2q9", "fp64", "auto", 3),
    ("d2q9", "bf16", "auto", 5),
    ("d2q7", "fp32", "plain", 1),
    ("d2q7", "fp32", "tma", 1),
    ("d2q7", "fp32", "auto", 7),
    ("d2q7", "fp64", "auto", 3),
]


def params(lattice="d2q9", width=640, **kw):
    # (density growth close to its saturation: steps that starve, so that a sticky bit is set and cleared)
    return wl.base_params(width=width, height=160, front_row=60.0, growth_mode="density", rho0=1.02,
                          growth_rate=2e-3, wall_mode="advance", wall_min_gap=40.0, lattice=lattice, seed=5, **kw)


def same(a, b, status=True):
    sa, sb = a.stats(), b.stats()
    for k in sa:
        if k not in ("launches", "update_kernel", "clip_mass") and (status or k != "status"):
            assert sa[k] == sb[k], (k, sa[k], sb[k])
    for x, y in zip(a.last_events(), b.last_events()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.mask(), b.mask())
    assert np.array_equal(a.heights(), b.heights())


@pytest.mark.parametrize("lattice,precision,kernel,n", FORMS)
def test_clear_between_steps(lattice, precision, kernel, n):
    from paper_2303_02210_gb300.lbm import Simulation
    p = params(lattice)
    a = Simulation(p, precision=precision, update_kernel=kernel)
    b = Simulation(p, precision=precision, update_kernel=kernel)
    for i in range(4):
        a.step(n)
        b.step(n)
        assert a.stats()["events_last"] > 0
        b.lbm_clear_status()
        assert b.stats()["status"] == 0
        same(a, b, status=False)
    # the next step's divisions add their mass
    a.step(1)
    b.step(1)
    same(a, b, status=False)
    counts = b.last_events()[2]
    assert counts.sum() == b.stats()["events_last"] > 0
    a.close()
    b.close()


@pytest.mark.parametrize("precision,kernel", [("fp32", "auto"), ("fp32", "plain"), ("fp64", "auto")])
def test_clear_between_batch_steps(precision, kernel):
    from paper_2303_02210_gb300.lbm import Batch, Simulation
    ps = [params(width=w, sim_id=w) for w in (96, 200, 640)]
    a = [Simulation(p, precision=precision, update_kernel=kernel) for p in ps]
    b = [Simulation(p, precision=precision, update_kernel=kernel) for p in ps]
    ba, bb = Batch(a), Batch(b)
    for _ in range(3):
        ba.step(5)
        bb.step(5)
        for s in b:
            s.lbm_clear_status()
        for x, y in zip(a, b):
            same(x, y, status=False)
    ba.close()
    bb.close()
