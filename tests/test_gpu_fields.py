"""lbm_fields against Eq. 1 in IEEE doubles, bit for bit, from the populations the
library itself returns: rho the sum in index order, u = j / rho with one
correctly rounded division. The inputs reach both forms of the kernel (exact
integer sums; plain FP64 for ranges of 2^22 and more, negative zeros and
denormals), odd widths, and rows above the window."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HALF_SQRT3 = 0.8660254037844386


def eq1(f, q):
    r = f[0]
    for i in range(1, q):
        r = r + f[i]
    if q == 9:
        jx = ((((f[1] - f[3]) + f[5]) - f[6]) - f[7]) + f[8]
        jy = ((((f[2] - f[4]) + f[5]) + f[6]) - f[7]) - f[8]
    else:
        jx = ((((f[1] - f[4]) + 0.5 * f[2]) - 0.5 * f[3]) - 0.5 * f[5]) + 0.5 * f[6]
        jy = (((f[2] + f[3]) - f[5]) - f[6]) * HALF_SQRT3
    z = r == 0
    s = np.where(z, 1.0, r)
    return r, np.where(z, 0.0, jx / s), np.where(z, 0.0, jy / s)


@pytest.mark.parametrize("lattice,precision,width", [("d2q9", "fp32", 129), ("d2q9", "fp32", 64), ("d2q9", "fp16", 77),
                                                     ("d2q9", "bf16", 96), ("d2q9", "fp64", 33), ("d2q7", "fp32", 131),
                                                     ("d2q7", "fp64", 40)])
def test_fields_bit_exact(lattice, precision, width):
    from paper_2303_02210_gb300 import workloads as wl
    from paper_2303_02210_gb300.lbm import Simulation
    q = 7 if lattice == "d2q7" else 9
    p = wl.base_params(width=width, height=96, front_row=40.0, growth_rate=1e-3, lattice=lattice, seed=5)
    sim = Simulation(p, precision=precision)

    def check():
        f = sim.pops()
        for got, want in zip(sim.fields(), eq1(f, q)):
            assert np.array_equal(got.view(np.int64), np.ascontiguousarray(want).view(np.int64))

    check()
    sim.step(25)
    check()
    # populations over all ratios from 1 to 2^40 of their largest, some zero
    rng = np.random.default_rng(3)
    f = rng.uniform(0.5, 1.0, (q, 96, width)) * 2.0 ** -rng.integers(0, 41, (q, 96, width))
    near = rng.uniform(0.5, 1.0, (q, 96, width)) * 2.0 ** -rng.integers(0, 23, (q, 96, width))
    f = np.where(rng.random((96, width)) < 0.7, near, f)
    f[rng.random(f.shape) < 0.2] = 0.0
    f[:, 80:] = 0.0  # no mass: above the window
    f[0, 81, :] = -0.0
    f[1, 10, ::3] = 1e-41  # denormal in FP32
    f[2, 11, ::5] = -0.0
    f[:, 12, ::2] *= 2.0 ** 30
    if precision in ("fp16", "bf16"):
        f = np.minimum(f, 1.0)
    sim.set_pops(f)
    check()
    sim.close()
