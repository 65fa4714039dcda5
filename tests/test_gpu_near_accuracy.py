"""The stored near field of FP64 plans: two points next to one another have a large entry, which must not cost
the entries of all other pairs their digits."""
import numpy as np
import pytest

import workloads as W
from oracle import direct

pytestmark = pytest.mark.gpu

MED = W.Medium(W.IMPEDANCE, (400.0,), alpha=10.0)
# A leaf's sum has an error of at most 2.8e-16 (55- and 54-bit digits, against extended precision); two of them,
# and entries up to 4 where that has up to 1:
TOL = 2e-15


def _torch():
    return pytest.importorskip("torch")


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("gap", [1e-300, 1e-30, 1e-11])
def test_almost_coincident_points_leave_the_other_sums_alone(adaptive, gap):
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 1500
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=17)
    xy[0] = xy[1] = (0.0, 0.6)
    xy[2] = (1.0, 0.02)                      # the same root square and tree for both clouds
    q = W.strengths(1, n, 1, salt=17)
    q[:, :2] = 0.0
    got = []
    for dx in (gap, 1e-3):
        xy[1, 0] = dx
        with Plan(xy, MED, tol=1e-6, p=6, leaf_size=32, adaptive=adaptive) as plan:
            got.append(plan.apply(torch.from_numpy(q).cuda(), parts=1).cpu().numpy()[:, 2:])
    assert direct.rel_l2(got[0], got[1]) < TOL, direct.rel_l2(got[0], got[1])


@pytest.mark.parametrize("adaptive", [False, True])
def test_almost_coincident_points_see_one_another(adaptive):
    """Two targets 1e-300 apart: (i / 4) H0 of that distance times the other's strength, on top of the common rest."""
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 300
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=18)
    xy[0], xy[1], xy[2] = (0.0, 0.6), (1e-300, 0.6), (1.0, 0.02)
    q = W.strengths(1, n, 1, salt=18)
    with Plan(xy, MED, tol=1e-6, p=6, leaf_size=32, adaptive=adaptive) as plan:
        y = plan.apply(torch.from_numpy(q).cuda(), parts=1).cpu().numpy()[0]
    x = MED.k[0] * 1e-300
    g = 0.25j * (1.0 + 2j / np.pi * (np.log(x / 2.0) + np.euler_gamma))
    assert abs((y[0] - g * q[0, 1]) - (y[1] - g * q[0, 0])) < 1e-12 * abs(g)
