"""Quotients by a shared divisor (the negative fix's rescaling, u = j / rho, Eq. 4's
mean) are IEEE division's, bit for bit: FP64 runs equal the oracle's where nearly
every node is rescaled, at divisors and numerators over many magnitudes, clipped
zeros among them; FP32 forms (staged, plain, fused) equal one another there."""
import numpy as np
import pytest

from paper_2303_02210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", ["d2q9", "d2q7"])
@pytest.mark.parametrize("negfix", ["literal", "rescale"])
@pytest.mark.parametrize("scale", [1.0, 1e-9, 1e12])
def test_rescaled_nodes(lattice, negfix, scale):
    from oracle.oracle import OracleSim
    from paper_2303_02210_gb300.lbm import Simulation
    # every density-valued parameter scaled together: the divisors' magnitudes
    # move out of the method's range at the extremes (the plain division then)
    p = wl.paper_params(width=90, height=70, front_row=30.0, lattice=lattice, negfix_mode=negfix, sigma=0.02 * scale,
                        rho_init=0.1 * scale, rho_c=0.05 * scale, rho_cell=0.01 * scale, rho0=0.15 * scale,
                        growth_rate=0.0, growth_mode="none", wall_mode="fixed", seed=9)
    o = OracleSim(p)
    g = Simulation(p, precision="fp64")
    o.step(12)
    g.step(12)
    assert np.array_equal(g.pops(), o.pops())
    a = Simulation(p, update_kernel="plain")
    a.step(12)
    for k in ("tma", "auto"):
        b = Simulation(p, update_kernel=k)
        b.step(12)
        assert np.array_equal(a.pops(), b.pops()), k
