"""Batches with few tiles, in the paper's regime (noise that drives populations
negative at nearly every node), against the same members stepped alone by the
plain-load kernel, bit for bit: D2Q9, whose staged batched update deals smaller
chunks of tiles then, and D2Q7; widths at the edges of a tile and of a warp's 64
columns, odd ones, both negative fixes, advancing walls."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def member(i, width, lattice="d2q7", **kw):
    p = wl.paper_params(width=width, height=260, growth_mode="bulk", wall_mode="advance", front_row=60.0,
                        front_amp=0.5, negfix_mode="rescale" if i % 2 else "literal", lattice=lattice,
                        sim_id=i, seed=11 + i)
    p.update(kw)
    return p


def check(ps, steps):
    from paper_2303_02210_gb300.lbm import Batch, Simulation
    ref = [Simulation(p, update_kernel="plain") for p in ps]
    sims = [Simulation(p) for p in ps]
    batch = Batch(sims)
    for n in steps:
        batch.step(n)
        for r, s in zip(ref, sims):
            r.step(n)
            assert np.array_equal(r.pops(), s.pops())
            assert np.array_equal(r.mask(), s.mask())
            sr, ss = r.stats(), s.stats()
            for k in ("mass_fix", "quiescent_fix", "S1", "S2", "ns_total", "div_total", "y_r", "y_hi", "step", "status"):
                assert sr[k] == ss[k], k
    batch.close()


@pytest.mark.parametrize("lattice", ["d2q9", "d2q7"])
@pytest.mark.parametrize("widths", [(1, 64, 65, 128), (129, 512, 63, 300, 256, 31), (2047,) * 3, (64, 128, 256, 512) * 16])
def test_small_batches_bit_exact(lattice, widths):
    check([member(i, w, lattice, sigma=0.0 if i == 2 else 0.01) for i, w in enumerate(widths)], (1, 20))
