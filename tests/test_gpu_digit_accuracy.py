"""FP64 translations as digit products against the FP64 kernels of the same
plan geometry, at the rounding of FP64 itself."""
import numpy as np
import pytest

import workloads as W
from oracle import direct

pytestmark = pytest.mark.gpu

MEDIA = {"imp": W.Medium(W.IMPEDANCE, (60.0,), alpha=30.0), "two": W.WORKLOADS[3].medium, "low": W.Medium(W.IMPEDANCE, (1.0,), alpha=1.0)}
# Largest rounding error of one level's list in FP64 arithmetic, measured against extended precision for
# k h = 0.01 .. 25, p = 9 .. 45, strengths of one size and of a million sizes: 4e-15 of the field.  Products that keep the digit orders
# 0 .. 6 are at 1.5e-15 there, orders 0 .. 5 alone at 3e-14.  Three levels, both sides:
TOL = 8e-15
FAR_FREE, FAR_REACT = 2, 4


def _torch():
    return pytest.importorskip("torch")


@pytest.mark.parametrize("medium,levels,part", [("imp", 4, FAR_FREE), ("imp", 5, FAR_FREE), ("two", 5, FAR_FREE),
                                                ("two", 4, FAR_REACT), ("low", 4, FAR_FREE)])
def test_digit_products_round_no_worse_than_fp64(medium, levels, part):
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 2000
    med = MEDIA[medium]
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=levels)
    g = np.random.default_rng(levels)
    size = 10.0 ** (-6.0 * g.random((8, 8)))[np.minimum((xy[:, 0] * 8).astype(int), 7),
                                             np.minimum(((xy[:, 1] - 0.02) * 8).astype(int), 7)]
    q = torch.from_numpy(W.strengths(1, n, 1, salt=levels) * size).cuda()
    with Plan(xy, med, tol=1e-6, levels=levels, dense_m2l=True) as plan:
        got = plan.apply(q, parts=part).cpu().numpy()
        launches = plan.info["launches_last_apply"]
        p = plan.info["p"]
    # a width whose digits pass the plan's 16 GB keeps the FP64 kernels
    digit_bytes = sum((2 if l < levels else 1) * 4 ** l * ((2 * (2 * p[l] + 1) + 15) // 16) * 192 for l in range(2, levels + 1))
    with Plan(xy, med, tol=1e-6, levels=levels, dense_m2l=True, max_rhs=int(16.5e9 / digit_bytes)) as plan:
        want = plan.apply(q, parts=part).cpu().numpy()
        assert plan.info["launches_last_apply"] < launches          # no slicing launches
    assert direct.rel_l2(got, want) < TOL, direct.rel_l2(got, want)
