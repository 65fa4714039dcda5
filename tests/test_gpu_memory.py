"""Device memory that holds a plan but not the stores that only make it faster (digits and
operator slices, bases, FP32 blocks): the plan is made without them, and a call that runs out of memory can be made again."""
import numpy as np
import pytest

import workloads as W
from oracle import direct

pytestmark = pytest.mark.gpu

MED = W.Medium(W.IMPEDANCE, (20.0,), alpha=10.0)
MB = 1 << 20


def _torch():
    return pytest.importorskip("torch")


class _Filled:
    """All but `keep` bytes of the device's free memory, taken by the test."""

    def __init__(self, keep):
        self.keep = keep

    def __enter__(self):
        torch = _torch()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.blocks = []
        for size in (4096 * MB, 256 * MB, 16 * MB, 2 * MB):
            while torch.cuda.mem_get_info()[0] > self.keep + size:
                try:
                    self.blocks.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
                except torch.cuda.OutOfMemoryError:
                    break
        return self

    def __exit__(self, *exc):
        self.blocks.clear()
        _torch().cuda.empty_cache()


def _used(make):
    """A plan and the bytes it took."""
    torch = _torch()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    plan = make()
    return plan, before - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("max_rhs,share", [(512, 0.75), (24, 0.85), (2, 0.8)])
def test_plan_without_room_for_its_digits(adaptive, max_rhs, share):
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 20000
    xy = torch.from_numpy(W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=6)).cuda()
    q = torch.from_numpy(W.strengths(1, n, 1, salt=6)).cuda()
    make = lambda: Plan(xy, MED, tol=1e-6, max_rhs=max_rhs, adaptive=adaptive, dense_m2l=not adaptive)    # noqa: E731
    plan, used = _used(make)
    want = plan.apply(q).cpu().numpy()
    launches, buffers = plan.info["launches_last_apply"], plan.info["buffer_bytes"]
    plan.close()
    out = torch.empty_like(q)
    with _Filled(int(share * used)):
        with make() as tight:
            tight.apply(q, out=out)
            got = out.cpu().numpy()
            assert tight.info["buffer_bytes"] < buffers
            if max_rhs > 100:
                assert tight.info["launches_last_apply"] < launches        # no slicing launches
    assert direct.rel_l2(got, want) < 1e-12, direct.rel_l2(got, want)


def test_gradient_that_ran_out_of_memory_can_be_asked_again():
    torch = _torch()
    from paper_1703_09136_gb300 import MIXED, HfmmError, Plan
    n = 20000
    xy = torch.from_numpy(W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=6)).cuda()
    q, g = (torch.from_numpy(W.strengths(1, n, 1, salt=s).astype(np.complex64)).cuda() for s in (6, 7))
    with Plan(xy, MED, tol=1e-6, precision=MIXED) as plan:
        want = plan.grad(q, g).cpu().numpy()
    out = torch.empty((n, 2), dtype=torch.float64, device="cuda")
    with Plan(xy, MED, tol=1e-6, precision=MIXED) as plan:
        failed = 0
        for keep in (12 * MB, 40 * MB, 80 * MB, 120 * MB, 160 * MB, 200 * MB):
            with _Filled(keep):
                try:
                    plan.grad(q, g, out=out)
                    break
                except HfmmError as e:
                    assert "OOM" in str(e)
                    failed += 1
        assert failed > 0
        got = plan.grad(q, g).cpu().numpy()
    assert np.linalg.norm(got - want) < 1e-12 * np.linalg.norm(want)
