"""Fused passes at the sizes where their tiles and splits have edges: position
gradients and few-right-hand-side mixed applies of leaves with one point, more
than a warp, more than a CTA and none at all; the leaves' L2P at every width; stored blocks next to coincident
points; restarted GMRES at its smallest bases."""
import numpy as np
import pytest

import workloads as W
from oracle import direct

pytestmark = pytest.mark.gpu

# impedance, and two layers (whose lowest leaves also sum their reaction directly)
MEDIA = {"imp": W.WORKLOADS[1].medium, "two": W.WORKLOADS[3].medium}
GRAD_TOL = 1e-8      # a plan of tol 1e-10, as the parity tests bound the same comparison
MIXED_TOL = 1e-5     # a mixed plan of tol 1e-6, as the parity tests


def _torch():
    return pytest.importorskip("torch")


def _clustered(n, crowd, salt):
    """n points in the unit square, `crowd` of them in one sixteenth-wide corner of it."""
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=salt)
    xy[:crowd, 0] = 0.53 + 0.15 * xy[:crowd, 0]
    xy[:crowd, 1] = 0.03 + 0.15 * (xy[:crowd, 1] - 0.02)
    return xy


@pytest.mark.parametrize("medium,n,crowd,levels,nrhs", [
    ("imp", 40, 0, 2, 1), ("imp", 330, 300, 2, 1), ("two", 330, 131, 2, 2), ("two", 300, 33, 3, 1), ("imp", 300, 17, 4, 5)])
def test_gradient_leaf_edges(medium, n, crowd, levels, nrhs):
    _torch()
    from paper_1703_09136_gb300 import Plan
    med, xy = MEDIA[medium], _clustered(n, crowd, levels)
    q, g = W.strengths(1, n, nrhs, salt=1), W.strengths(1, n, nrhs, salt=2)
    want = direct.position_grad(med, xy, q, g)
    with Plan(xy, med, tol=1e-10, levels=levels, max_rhs=nrhs) as plan:
        got = plan.grad(q, g)
        assert np.array_equal(got, plan.grad(q, g))
    assert np.linalg.norm(got - want) < GRAD_TOL * np.linalg.norm(want)


@pytest.mark.parametrize("medium,n,crowd,levels,nrhs", [
    ("imp", 40, 0, 2, 1), ("imp", 330, 300, 2, 4), ("two", 330, 257, 2, 3), ("two", 300, 33, 3, 2), ("imp", 300, 17, 4, 1)])
def test_few_rhs_leaf_edges(medium, n, crowd, levels, nrhs):
    torch = _torch()
    from paper_1703_09136_gb300 import MIXED, Plan
    med, xy = MEDIA[medium], _clustered(n, crowd, levels)
    q = W.strengths(1, n, nrhs, salt=1).astype(np.complex64)
    want = direct.direct_apply(med, xy, q.astype(complex))
    adj = direct.direct_apply(med, xy, q.astype(complex).conj()).conj()      # G is complex symmetric
    with Plan(xy, med, tol=1e-6, levels=levels, max_rhs=nrhs, precision=MIXED) as plan:
        dev = plan.apply(torch.from_numpy(q).cuda()).cpu().numpy()
        assert direct.rel_l2(dev, want) < MIXED_TOL, direct.rel_l2(dev, want)
        host = plan.apply(q)                                                 # buffers in host memory
        assert np.array_equal(np.asarray(host), dev)
        back = plan.adjoint(torch.from_numpy(q).cuda()).cpu().numpy()
        assert direct.rel_l2(back, adj) < MIXED_TOL, direct.rel_l2(back, adj)


@pytest.mark.parametrize("p,nrhs", [(7, 5), (13, 33), (15, 64), (17, 65), (23, 33), (25, 5), (31, 64)])
def test_leaf_l2p_in_the_downward_pass(p, nrhs):
    """Leaf widths of every staging size (up to 128 columns in the pass, more beside it), ragged right-hand
    sides, leaves of zero to a dozen points; against the FP64 plan of the same orders."""
    torch = _torch()
    from paper_1703_09136_gb300 import MIXED, Plan
    n, med = 4001, MEDIA["two"]
    xy = _clustered(n, 0, p)
    q = W.strengths(1, n, nrhs, salt=p)
    with Plan(xy, med, tol=1e-6, p=p, levels=5, max_rhs=nrhs) as plan:
        want = plan.apply(torch.from_numpy(q).cuda()).cpu().numpy()
    with Plan(xy, med, tol=1e-6, p=p, levels=5, max_rhs=nrhs, precision=MIXED, small_rhs=-1) as plan:
        columns = 2 * (2 * plan.info["p"][-1] + 1)
        assert plan.info["leaf_l2p_fused"] == (columns <= 128)      # one column block
        got = plan.apply(torch.from_numpy(q.astype(np.complex64)).cuda()).cpu().numpy()
    assert direct.rel_l2(got, want) < MIXED_TOL, direct.rel_l2(got, want)


def test_coincident_points_spoil_their_own_targets_only():
    """Two points at one place: their mutual entry is infinite, so the stored
    blocks cannot be cut into digits and the plan keeps the evaluating kernel."""
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    xy = _clustered(300, 40, 9)
    xy[1] = xy[0]
    q = W.strengths(1, 300, 2, salt=4)
    q[:, 0] = 0.0                                # the others see one source at that place
    want = direct.direct_apply(MEDIA["imp"], xy[1:], q[:, 1:])
    with Plan(xy, MEDIA["imp"], tol=1e-10, levels=3, max_rhs=2) as plan:
        y = plan.apply(torch.from_numpy(q).cuda()).cpu().numpy()
    assert not np.isfinite(y[:, :2]).all()
    assert direct.rel_l2(y[:, 2:], want[:, 1:]) < GRAD_TOL


@pytest.mark.parametrize("n,restart", [(1, 1), (3, 1), (60, 2), (200, 7), (200, 400)])
def test_gmres_basis_edges(n, restart):
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=n)
    b = torch.from_numpy(W.strengths(1, n, 1, salt=6)[0]).cuda()
    sigma = 4.0 * n                              # dominates the operator: every restart length converges
    with Plan(xy, MEDIA["imp"], tol=1e-10, levels=2, max_rhs=1) as plan:
        x, it, rr = plan.solve(b, sigma=sigma, tol=1e-9, restart=restart, maxit=200)
        res = b - sigma * x - plan.apply(x.reshape(1, -1))[0]
        assert rr <= 1e-9 and float(res.norm()) <= 2e-9 * float(b.norm())
        x2, it2, rr2 = plan.solve(b, sigma=sigma, x0=x, tol=1e-8, restart=restart, maxit=200)
        assert it2 == 0 and torch.equal(x2, x)   # already there
