"""A plan's first apply inside a caller's own graph capture: the side streams of the concurrent
passes are made and joined there."""
import numpy as np
import pytest

import workloads as W
from oracle import direct

pytestmark = pytest.mark.gpu


def _torch():
    return pytest.importorskip("torch")


@pytest.mark.parametrize("adaptive,mixed", [(False, False), (True, False), (True, True)])
def test_first_apply_inside_a_callers_capture(adaptive, mixed):
    torch = _torch()
    from paper_1703_09136_gb300 import FP64, MIXED, Plan
    n = 2000
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.05, 1.05)), salt=31)
    q = torch.from_numpy(W.strengths(1, n, 1, salt=31).astype(np.complex64 if mixed else np.complex128)).cuda()
    kw = dict(tol=1e-6, precision=MIXED if mixed else FP64, adaptive=adaptive)
    med = W.Medium(W.IMPEDANCE, (30.0,), alpha=10.0)
    with Plan(xy, med, **kw) as plan:
        want = plan.apply(q).cpu().numpy()
    with Plan(xy, med, **kw) as plan:
        out = torch.zeros_like(q)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            plan.apply(q, out=out)
        for _ in range(3):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert direct.rel_l2(out.cpu().numpy(), want) < (1e-6 if mixed else 1e-15)
        del graph
