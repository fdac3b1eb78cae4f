"""The device memory of one simulation beyond its two copies of the populations
and its mask stays small: a small lattice is not charged for structures sized by
the largest launch grid."""
import pytest

from paper_2303_02210_gb300 import lbm
from paper_2303_02210_gb300 import workloads as wl


@pytest.mark.parametrize("precision,elem", [("fp32", 4), ("fp64", 8), ("fp16", 2)])
@pytest.mark.parametrize("width,height,most", [(1, 3, 1 << 18), (128, 256, 1 << 19), (1024, 1024, 3 << 20)])
def test_bookkeeping_is_small(precision, elem, width, height, most):
    p = wl.base_params(width=width, height=height, growth_rate=1e-4, front_row=2.0)
    populations = 2 * 9 * ((width + 2 * 4 + 31) // 32 * 32) * height * elem
    assert lbm.lbm_footprint(p, precision) - populations <= most


def test_staged_buckets_only_where_a_form_is_staged():
    p = wl.base_params(width=4096, height=2048, growth_rate=0.0, growth_mode="none", front_row=9.0)
    q = dict(p, y_periodic=1, wall_mode="fixed", front_kind="full")
    assert lbm.lbm_footprint(q) < lbm.lbm_footprint(p)
    assert lbm.lbm_footprint(p) - lbm.lbm_footprint(q) <= (2 << 20) + (1 << 14)
