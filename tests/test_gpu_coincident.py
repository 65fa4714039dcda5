"""Coincident points: their entries of the stored near field are infinite and have no digits."""
import numpy as np
import pytest

import workloads as W
from oracle import direct

pytestmark = pytest.mark.gpu

MED = W.Medium(W.IMPEDANCE, (20.0,), alpha=10.0)


def _torch():
    return pytest.importorskip("torch")


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("same", [2, 5, 40])
def test_coincident_points_keep_the_stored_near_field(adaptive, same):
    """`same` points at one place: their own targets are not finite (the sources there are infinitely strong), all
    others are, and the stored blocks still serve the near field of the plan."""
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n, nrhs = 600, 2
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=9)
    xy[1:same] = xy[0]
    q = W.strengths(1, n, nrhs, salt=4)
    alone = q.copy()
    alone[:, :same] = 0.0
    alone[:, 0] = q[:, :same].sum(axis=1)                # one source of the summed strength
    want = direct.direct_apply(MED, xy[same - 1:], np.concatenate([alone[:, :1], alone[:, same:]], axis=1))[:, 1:]
    wadj = direct.direct_apply(MED, xy[same - 1:], np.concatenate([alone[:, :1], alone[:, same:]], axis=1).conj()).conj()[:, 1:]
    with Plan(xy, MED, tol=1e-10, leaf_size=16, max_rhs=nrhs, adaptive=adaptive) as plan:
        for run, ref in ((plan.apply, want), (plan.adjoint, wadj)):
            y = run(torch.from_numpy(q).cuda()).cpu().numpy()
            assert not np.isfinite(y[:, :same]).any()
            assert direct.rel_l2(y[:, same:], ref) < 1e-8, direct.rel_l2(y[:, same:], ref)
        near = plan.apply(torch.from_numpy(q).cuda(), parts=1).cpu().numpy()
        assert not np.isfinite(near[:, :same]).any() and np.isfinite(near[:, same:]).all()
        plan.apply(torch.from_numpy(q).cuda())
        if not adaptive:
            # stored blocks: 16 bytes a pair on top of the strengths', fields' and points' bytes
            moved = plan.info["bytes_last_apply"]["p2p"]
            assert moved > 64.0 * nrhs * n + 16.0 * n


@pytest.mark.parametrize("adaptive", [False, True])
def test_infinite_values_are_those_of_the_kernel(adaptive):
    """An entry is (inf, 1 / 4): each product's sign and its NaN where a part of the strength is zero."""
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    xy = W.points_in_box(1, 300, ((0.0, 1.0), (0.02, 1.02)), salt=12)
    xy[1] = xy[0]
    q = np.zeros((3, 300), dtype=complex)
    q[:, 0] = (-1.0, 1.0 + 1.0j, 0.0)
    q[:, 1] = (2.0j, -1.0 - 3.0j, 0.0)
    with Plan(xy, MED, tol=1e-6, leaf_size=16, max_rhs=3, adaptive=adaptive) as plan:
        y = plan.apply(torch.from_numpy(q).cuda(), parts=1).cpu().numpy()[:, :2]
        w = plan.adjoint(torch.from_numpy(q).cuda()).cpu().numpy()[:, :2]
    inf, nan = np.inf, np.nan
    re = np.array([[nan, -inf], [-inf, inf], [nan, nan]])         # target 0 sees the strength of 1, and the other way round
    im = np.array([[inf, nan], [-inf, inf], [nan, nan]])
    assert np.array_equal(y.real, re, equal_nan=True) and np.array_equal(y.imag, im, equal_nan=True)
    assert np.array_equal(w.real, re, equal_nan=True) and np.array_equal(w.imag, im, equal_nan=True)
