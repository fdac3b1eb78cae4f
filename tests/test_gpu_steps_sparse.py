"""Many steps in one launch with fewer than one division a step, on fronts just
wider than one planner CTA scans (512 columns): the coming step draws many
candidates (few are accepted) by more planner CTAs than have words of the front
to scan, and then needs no division at all, so that nothing but the CTAs' counts
holds the commit back. Bit for bit against the step-by-step launches."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,precision,width", [("d2q9", "fp32", 513), ("d2q9", "fp32", 700), ("d2q9", "bf16", 520),
                                                     ("d2q7", "fp32", 544)])
def test_no_division_after_many_candidates(lattice, precision, width):
    from paper_2303_02210_gb300.lbm import STATUS_TIMEOUT, Simulation
    p = wl.base_params(width=width, height=160, front_row=60.0, growth_mode="edge", edge_depth=2, wall_mode="fixed",
                       growth_rate=0.5 * 0.1 / (60.0 * width), front_kind="sinusoidal", front_amp=55.0, front_kmax=3,
                       lattice=lattice, seed=7)
    a = Simulation(p, precision=precision, update_kernel="plain")
    b = Simulation(p, precision=precision)
    steps = []
    for _ in range(200):
        a.step(1)
        st = a.stats()
        steps.append((st["ns_last"], st["cand_last"]))
    b.step(200)
    sb = b.stats()
    assert not sb["status"] & STATUS_TIMEOUT
    assert sb["launches"] == 4  # 64 + 64 + 64 + 8 steps
    # the state this test is for: a division, its first pass sized by the
    # candidates of the division before (more than 16 for each CTA that scans
    # the front), then a step without one
    scan = -(-(-(-width // 32)) // 4)
    ratio, hit = 0.0, 0
    for (n, c), (m, _) in zip(steps, steps[1:]):
        hit += n == 1 and m == 0 and 1.15 * ratio + 64 > 16 * scan
        ratio = c if n == 1 else ratio
    assert hit
    for k in ("ns_total", "div_total", "cand_last", "mass_fix", "S1", "S2", "H_top", "hmin", "y_hi", "carry", "status"):
        assert st[k] == sb[k], (k, st[k], sb[k])
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.mask(), b.mask())
    for x, y in zip(a.last_events(), b.last_events()):
        assert np.array_equal(x, y)
    a.close()
    b.close()
