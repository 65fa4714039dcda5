"""FP64 applies of strengths at the ends of the exponent range: digit products and stored near field
keep every binade that FP64 arithmetic keeps."""
import numpy as np
import pytest

import workloads as W
from oracle import direct

pytestmark = pytest.mark.gpu

MEDIUM = W.Medium(W.IMPEDANCE, (60.0,), alpha=30.0)


def _torch():
    return pytest.importorskip("torch")


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("scale", [-1012, -900, 950])
def test_strengths_at_the_ends_of_the_exponent_range(adaptive, scale):
    """Normal results of strengths near both ends of the FP64 range.  Near -1012 the highest orders' coefficients
    are subnormal: 2^-1074 against 2^-1012, times 2^20 of the translations, leaves 1e-12."""
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 500
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=3)
    q = W.strengths(1, n, 1, salt=3)
    with Plan(xy, MEDIUM, tol=1e-6, leaf_size=16, adaptive=adaptive) as plan:
        for part in (1, 2, 4, 15):
            one = plan.apply(torch.from_numpy(q).cuda(), parts=part).cpu().numpy()
            got = plan.apply(torch.from_numpy(q * 2.0 ** scale).cuda(), parts=part).cpu().numpy()
            got = np.ldexp(got.view(np.float64), -scale).view(np.complex128)
            assert direct.rel_l2(got, one) < 1e-10, (part, direct.rel_l2(got, one))
