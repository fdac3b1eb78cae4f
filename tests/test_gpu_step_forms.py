"""Which launches a call of lbm_step takes: two for every step, or up to 64 steps
in one, by the initial window and the call's steps. The results of calls on both
sides of the line are those of the plain-load launches, bit for bit."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,precision,width,rows,growth,fewest", [
    ("d2q9", "fp32", 128, 53, 1e-4, 1), ("d2q9", "bf16", 1024, 150, 1e-4, 1), ("d2q7", "fp32", 512, 300, 1e-4, 1),
    ("d2q9", "fp32", 2048, 100, 1e-4, 2), ("d2q7", "fp32", 2048, 100, 1e-4, 1), ("d2q9", "fp32", 1024, 400, 1e-4, 2),
    ("d2q7", "fp32", 2048, 1000, 1e-4, 2), ("d2q9", "fp32", 2048, 1000, 1e-4, 4), ("d2q9", "fp16", 2048, 700, 1e-4, 8),
    ("d2q9", "fp16", 4096, 634, 1e-4, 0),
    ("d2q9", "fp16", 1024, 400, 1e-3, 1), ("d2q9", "bf16", 2048, 700, 1e-3, 2), ("d2q7", "fp32", 2048, 1000, 1e-3, 1),
    ("d2q9", "fp16", 4096, 634, 1e-3, 2), ("d2q9", "fp32", 4096, 900, 1e-3, 0)])
def test_fewest_steps_of_one_launch(lattice, precision, width, rows, growth, fewest):
    from paper_2303_02210_gb300.lbm import Simulation
    p = wl.base_params(width=width, height=rows + 60, front_row=float(rows), growth_mode="edge", growth_rate=growth,
                       wall_mode="fixed", lattice=lattice, seed=3)
    s = Simulation(p, precision=precision)
    done = 0
    for n in sorted({1, max(1, fewest - 1), max(1, fewest), 9}):
        before = s.stats()["launches"]
        s.step(n)
        done += n
        assert s.stats()["launches"] - before == (1 if fewest and n >= fewest else 2 * n), n
    r = Simulation(p, precision=precision, update_kernel="plain")
    r.step(done)
    assert np.array_equal(r.pops(), s.pops())
    assert r.stats()["div_total"] == s.stats()["div_total"]
    r.close()
    s.close()
