"""FP64 plans whose cloud leaves boxes of a diagonal level empty: the locals of
such boxes are never written, so nothing of them (allocator contents, the
plan's own check, earlier calls of another width) may reach a result."""
import numpy as np
import pytest

import workloads as W
from oracle import direct

pytestmark = pytest.mark.gpu

TOL = 1e-10      # diagonal against dense translations: 1e-12 a level (the plan's check), several levels


def _torch():
    return pytest.importorskip("torch")


def _strip(n):
    """A strip four times as wide as high, 16 wavelengths high: the upper half of its root square is empty."""
    return W.Medium(W.IMPEDANCE, (100.0,), alpha=50.0), W.points_in_box(1, n, ((0.0, 4.0), (0.05, 1.05)), salt=21)


def test_other_calls_do_not_reach_empty_boxes_of_diagonal_levels():
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 3000
    med, xy = _strip(n)
    q = torch.from_numpy(W.strengths(1, n, 2, salt=21)).cuda()
    g = torch.from_numpy(W.strengths(1, n, 1, salt=22)).cuda()
    q1 = q[:1].contiguous()
    bad = q.clone()
    bad[1, 5] = complex("nan")
    with Plan(xy, med, tol=1e-6, max_rhs=2, dense_m2l=True) as dense:
        want, wgrad = dense.apply(q1).cpu().numpy(), dense.grad(q1, g).cpu().numpy()
    with Plan(xy, med, tol=1e-6, max_rhs=2) as plan:
        info = plan.info
        assert info["diag_levels"] & ((1 << info["levels"]) - 1), info["diag_levels"]     # one above the leaves
        first, fgrad = plan.apply(q1).cpu().numpy(), plan.grad(q1, g).cpu().numpy()
        assert direct.rel_l2(first, want) < TOL, direct.rel_l2(first, want)
        assert np.linalg.norm(fgrad - wgrad) < TOL * np.linalg.norm(wgrad)
        for other in (q * 1e12, q * 1e200, bad):
            plan.apply(other)
            assert np.array_equal(plan.apply(q1).cpu().numpy(), first)
            plan.apply(other)
            assert np.array_equal(plan.adjoint(q1.conj().resolve_conj().contiguous()).conj().cpu().numpy(), first)
            plan.apply(other)
            assert np.array_equal(plan.grad(q1, g).cpu().numpy(), fgrad)


@pytest.mark.parametrize("scale", [-100, 300])
def test_first_call_does_not_see_what_planning_left(scale):
    """A power of two on the strengths multiplies every result exactly, on a fresh plan's first call too."""
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 3000
    med, xy = _strip(n)
    q = W.strengths(1, n, 1, salt=23)
    with Plan(xy, med, tol=1e-6) as plan:
        one = plan.apply(torch.from_numpy(q).cuda()).cpu().numpy()
    with Plan(xy, med, tol=1e-6) as plan:
        got = plan.apply(torch.from_numpy(q * 2.0 ** scale).cuda()).cpu().numpy()
    assert np.array_equal(got, one * 2.0 ** scale)
