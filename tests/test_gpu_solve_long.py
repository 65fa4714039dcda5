"""GMRES on vectors longer than one cluster orthogonalises: several blocks a
Gram-Schmidt pass, their partial sums, short bases that restart, and the
boundary between the two kernels; both precisions."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _torch():
    return pytest.importorskip("torch")


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n,restart", [(4096, 5), (4097, 5), (4097, 40), (20011, 3), (20011, 60)])
def test_gmres_of_long_vectors(n, restart, mixed):
    torch = _torch()
    from paper_1703_09136_gb300 import FP64, MIXED, Plan
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.05, 1.05)), salt=n)
    dt = np.complex64 if mixed else np.complex128
    b = torch.from_numpy(W.strengths(1, n, 1, salt=n)[0].astype(dt)).cuda()
    sigma, tol = 0.01 * n * (1 + 0.5j), 1e-4 if mixed else 1e-9     # of the operator's size: several steps, every basis converges
    with Plan(xy, W.Medium(W.IMPEDANCE, (20.0,), alpha=10.0), tol=1e-8, precision=MIXED if mixed else FP64) as plan:
        x, it, rr = plan.solve(b, sigma=sigma, tol=tol, restart=restart, maxit=400)
        assert it >= 4                       # bases of several vectors, and more than one for the short ones
        res = (b - sigma * x - plan.apply(x.reshape(1, -1))[0]).to(torch.complex128)
        norm = float(b.to(torch.complex128).norm())
        assert rr <= tol and float(res.norm()) <= 2 * tol * norm, (it, rr, float(res.norm()) / norm)
        y, it2, rr2 = plan.solve(b, sigma=sigma, tol=tol, restart=restart, maxit=400)
        assert it2 == it and rr2 == rr and torch.equal(x, y)
