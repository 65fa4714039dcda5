"""More right-hand sides than a grid dimension counts: kernels that have them there run
in several launches."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MED = W.Medium(W.IMPEDANCE, (20.0,), alpha=10.0)


def _torch():
    return pytest.importorskip("torch")


@pytest.mark.parametrize("adaptive,mixed", [(False, False), (True, False), (True, True)])
def test_more_right_hand_sides_than_a_grid_dimension(adaptive, mixed):
    torch = _torch()
    from paper_1703_09136_gb300 import FP64, MIXED, Plan
    n, nrhs = 40, 65537
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=5)
    g = np.random.default_rng(5)
    q = (g.standard_normal((nrhs, n)) + 1j * g.standard_normal((nrhs, n))).astype(np.complex64 if mixed else np.complex128)
    pick = [0, 1, 65534, 65535, 65536]
    with Plan(xy, MED, tol=1e-6, p=4, leaf_size=4, max_rhs=nrhs, dense_m2l=not adaptive, adaptive=adaptive,
              precision=MIXED if mixed else FP64) as plan:
        y = plan.apply(torch.from_numpy(q).cuda()).cpu().numpy()
        for r in pick:
            one = plan.apply(torch.from_numpy(q[r:r + 1]).cuda()).cpu().numpy()
            assert np.array_equal(y[r], one[0]), r


def test_gradients_of_more_right_hand_sides_than_a_grid_dimension():
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n, nrhs = 40, 65537
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=5)
    q, f = np.zeros((nrhs, n), dtype=complex), np.zeros((nrhs, n), dtype=complex)
    pick = [0, 1, 65534, 65535, 65536]
    q[pick], f[pick] = W.strengths(1, n, 5, salt=1), W.strengths(1, n, 5, salt=2)
    with Plan(xy, MED, tol=1e-6, p=4, leaf_size=4, max_rhs=nrhs, dense_m2l=True) as plan:
        got = plan.grad(torch.from_numpy(q).cuda(), torch.from_numpy(f).cuda()).cpu().numpy()
        want = plan.grad(torch.from_numpy(q[pick]).cuda(), torch.from_numpy(f[pick]).cuda()).cpu().numpy()
    assert np.linalg.norm(got - want) < 1e-13 * np.linalg.norm(want)     # the same 5 terms, sums in another order
