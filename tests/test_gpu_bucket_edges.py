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
