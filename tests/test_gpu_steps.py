"""Many steps in one launch (the automatic form of lbm_step for small and
middle-sized active windows) against the step-by-step launches of the
plain-load kernel: everything the library reports, bit for bit, for every growth
mode, storage type and lattice that takes it, at the edges of its rules (fronts
scanned whole by each planner CTA up to 512 columns, exchanged beyond; one and
many planner CTAs; candidates short of n_s; launches of 64 steps), mixed with
step-by-step launches of the same simulation, and with its waits running out."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [
    # lattice, precision, width, growth, wall, rate
    ("d2q9", "fp32", 1, "bulk", "fixed", 1e-2),
    ("d2q9", "fp32", 40, "bulk", "advance", 3e-2),
    ("d2q9", "fp32", 128, "none", "fixed", 0.0),
    ("d2q9", "fp32", 512, "edge", "advance", 1e-3),
    ("d2q9", "fp32", 515, "edge", "fixed", 1e-3),
    ("d2q9", "fp32", 1024, "density", "advance", 1e-3),
    ("d2q9", "fp32", 1056, "band", "advance", 2e-5),
    ("d2q9", "fp32", 4096, "bulk", "advance", 3e-3),
    ("d2q9", "fp16", 777, "density", "advance", 1e-3),
    ("d2q9", "fp16", 2100, "bulk", "advance", 1e-3),
    ("d2q9", "bf16", 130, "edge", "fixed", 1e-3),
    ("d2q7", "fp32", 129, "bulk", "advance", 1e-3),
    ("d2q7", "fp32", 3000, "edge", "advance", 1e-3),
]


def params(lattice, width, growth, wall, rate, **kw):
    return wl.base_params(width=width, height=160, front_row=60.0, growth_mode=growth, wall_mode=wall,
                          wall_min_gap=30.0, growth_rate=rate, lattice=lattice, seed=3, **kw)


def same(a, b):
    sa, sb = a.stats(), b.stats()
    # (launches and the kernel differ by design; the clip mass is a float sum in any order)
    for k in sa:
        if k not in ("launches", "update_kernel", "clip_mass"):
            assert sa[k] == sb[k], (k, sa[k], sb[k])
    assert abs(sa["clip_mass"] - sb["clip_mass"]) <= 1e-6 * max(1.0, abs(sa["clip_mass"]))
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.mask(), b.mask())
    assert np.array_equal(a.heights(), b.heights())
    for x, y in zip(a.last_events(), b.last_events()):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("lattice,precision,width,growth,wall,rate", CASES)
def test_many_steps_per_launch_bit_exact(lattice, precision, width, growth, wall, rate):
    from paper_2303_02210_gb300.lbm import Simulation
    p = params(lattice, width, growth, wall, rate)
    a = Simulation(p, precision=precision, update_kernel="plain")
    b = Simulation(p, precision=precision)
    for n in (1, 2, 66):
        a.step(n)
        b.step(n)
        same(a, b)
    # (66 steps: a launch of 64 and one of 2)
    assert b.stats()["launches"] == 4
    a.close()
    b.close()


def test_starved_and_rough_fronts():
    """Far fewer accepted candidates than drawn (density growth near its
    saturation: many rounds), and a front rougher than the 32 rows of one scan."""
    from paper_2303_02210_gb300.lbm import Simulation
    for kw in (dict(growth="density", rho0=1.02, rate=2e-3), dict(growth="edge", rate=1e-3)):
        g = kw.pop("growth")
        r = kw.pop("rate")
        p = params("d2q9", 640, g, "fixed", r, front_kind="sinusoidal", front_amp=50.0, front_kmax=4, **kw)
        a = Simulation(p, update_kernel="plain")
        b = Simulation(p)
        a.step(40)
        b.step(40)
        same(a, b)


def test_mixed_with_step_by_step_launches():
    """Kernel timing steps one update and one planner at a time, a batch steps
    its members by the batched launches: before and after the fused form."""
    from paper_2303_02210_gb300.lbm import Batch, Simulation
    p = params("d2q9", 700, "bulk", "advance", 2e-3)
    a = Simulation(p, update_kernel="plain")
    b = Simulation(p)
    for n in (5, 3, 8):
        b.step(n)
        b.lbm_timing_enable(4)
        b.step(n)
        b.lbm_timing_read()
        batch = Batch([b])
        batch.step(n)
        batch.close()
        a.step(3 * n)
        same(a, b)
    f = a.pops()
    a.set_pops(f)
    b.set_pops(f)
    a.step(7)
    b.step(7)
    same(a, b)


@pytest.mark.parametrize("lattice", ["d2q9", "d2q7"])
@pytest.mark.parametrize("withhold", [1, 2])
def test_waits_run_out_and_the_handle_recovers(lattice, withhold):
    """A staged copy withheld, or an arrival of the step's barrier: every CTA
    leaves, the step count is where the host expects it, and after recovery the
    handle steps as a fresh one does from the same state."""
    from paper_2303_02210_gb300.lbm import STATUS_TIMEOUT, Simulation
    p = params(lattice, 600, "none", "fixed", 0.0)
    a = Simulation(p, update_kernel="plain")
    b = Simulation(p)
    b.lbm_debug_waits(200_000, withhold)
    b.step(5)
    st = b.stats()
    assert st["status"] & STATUS_TIMEOUT and st["step"] == 5
    b.lbm_debug_waits(0, 0)
    b.lbm_clear_status()
    a.step(5)
    f = a.pops()
    a.set_pops(f)
    b.set_pops(f)
    a.step(20)
    b.step(20)
    assert b.stats()["status"] == 0
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.mask(), b.mask())
    assert np.array_equal(a.heights(), b.heights())


def test_two_streams_at_once():
    """Two simulations on streams of their own, their launches overlapping."""
    import torch
    from paper_2303_02210_gb300.lbm import Simulation
    p = [params("d2q9", w, "bulk", "advance", 1e-3) for w in (300, 2048)]
    ref = [Simulation(q, update_kernel="plain") for q in p]
    sims = [Simulation(q, stream=torch.cuda.Stream()) for q in p]
    for _ in range(4):
        for s in sims:
            s.step(50)
    for r, s in zip(ref, sims):
        r.step(200)
        same(r, s)
