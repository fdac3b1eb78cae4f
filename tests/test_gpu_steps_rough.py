"""Many steps in one launch on fronts that one planner CTA could scan whole but
that span many rows: their sums are exchanged then, and back to whole scans once
the front is smoother. Bit for bit against the step-by-step launches."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,precision,width,growth", [("d2q9", "fp32", 129, "edge"), ("d2q9", "fp32", 500, "bulk"),
                                                            ("d2q9", "fp16", 333, "density"), ("d2q7", "fp32", 405, "edge")])
@pytest.mark.parametrize("amp", [60.0, 70.0, 120.0])
def test_rough_fronts(lattice, precision, width, growth, amp):
    from paper_2303_02210_gb300.lbm import Simulation
    p = wl.base_params(width=width, height=400, front_row=150.0, growth_mode=growth, growth_rate=1e-3,
                       front_kind="sinusoidal", front_amp=amp, front_kmax=5, wall_mode="advance", wall_min_gap=60.0,
                       lattice=lattice, seed=17)
    a = Simulation(p, precision=precision, update_kernel="plain")
    b = Simulation(p, precision=precision)
    st = a.stats()
    assert (st["H_top"] - st["hmin"] > 96) == (amp > 65)
    for n in (3, 40):
        a.step(n)
        b.step(n)
        sa, sb = a.stats(), b.stats()
        for k in sa:
            if k not in ("launches", "update_kernel", "clip_mass"):
                assert sa[k] == sb[k], (k, sa[k], sb[k])
        assert np.array_equal(a.pops(), b.pops())
        assert np.array_equal(a.mask(), b.mask())
        assert np.array_equal(a.heights(), b.heights())
        for x, y in zip(a.last_events(), b.last_events()):
            assert np.array_equal(x, y)
    a.close()
    b.close()
