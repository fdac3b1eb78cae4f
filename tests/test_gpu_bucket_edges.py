"""Divisions per CTA of the staged updates around the number its bucket lists
(128: the rest of the selection is then scanned instead), repeats among them:
bit for bit against the plain-load update."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,kernel", [("d2q9", "auto"), ("d2q9", "tma"), ("d2q9", "tma1"), ("d2q9", "tma_st"),
                                            ("d2q7", "auto"), ("d2q7", "tma")])
@pytest.mark.parametrize("per_cta", [110, 128, 250])
def test_buckets_full_and_over(lattice, kernel, per_cta):
    from paper_2303_02210_gb300.lbm import Simulation
    # 31 tiles of 128 x 2 nodes (16 of 128 x 4) dealt over 10 (5) CTAs
    ctas = 5 if kernel == "tma1" else 10
    p = wl.base_params(width=128, height=160, front_row=60.0, growth_mode="bulk", wall_mode="fixed",
                       growth_rate=per_cta * ctas * 0.1 / (128 * 60), lattice=lattice, seed=11)
    a = Simulation(p, update_kernel="plain")
    b = Simulation(p, update_kernel=kernel)
    a.step(8)
    b.step(8)
    assert a.stats()["events_last"] >= 0.9 * per_cta * ctas
    assert np.array_equal(a.pops(), b.pops())
    for x, y in zip(a.last_events(), b.last_events()):
        assert np.array_equal(x, y)
    a.close()
    b.close()


@pytest.mark.parametrize("lattice,kernel", [("d2q9", "auto"), ("d2q9", "tma"), ("d2q9", "tma1"), ("d2q9", "tma_st"),
                                            ("d2q7", "auto"), ("d2q7", "tma")])
@pytest.mark.parametrize("precision", ["fp32", "fp16"])
def test_over_in_tiles_at_the_front_alone(lattice, kernel, precision):
    from paper_2303_02210_gb300.lbm import Simulation
    if precision == "fp16" and (lattice == "d2q7" or kernel == "tma_st"):
        pytest.skip("no such form")
    # 122 tiles of 128 x 2 nodes over 28 CTAs, about ten of them at the front
    # with 200 divisions each: a CTA over its bucket has tiles without any
    p = wl.base_params(width=256, height=220, front_row=120.0, growth_mode="edge", edge_depth=8, wall_mode="fixed",
                       growth_rate=2000 * 0.1 / (256 * 120), lattice=lattice, seed=13)
    a = Simulation(p, precision=precision, update_kernel="plain")
    b = Simulation(p, precision=precision, update_kernel=kernel)
    a.step(8)
    b.step(8)
    assert a.stats()["events_last"] >= 1900
    assert np.array_equal(a.pops(), b.pops())
    for x, y in zip(a.last_events(), b.last_events()):
        assert np.array_equal(x, y)
    a.close()
    b.close()
