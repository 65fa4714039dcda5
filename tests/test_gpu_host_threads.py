"""Applies and plan creation from two host threads."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _torch():
    return pytest.importorskip("torch")


def _in_threads(bodies):
    errors = []

    def guard(f):
        try:
            f()
        except BaseException as e:      # noqa: BLE001  (handed to the main thread)
            errors.append(e)
    ts = [threading.Thread(target=guard, args=(f,)) for f in bodies]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("mixed", [False, True])
def test_applies_of_plans_with_different_orders_from_two_threads(mixed):
    """Each plan's launches ask for their own amount of shared memory; neither thread may lower the other's limit."""
    torch = _torch()
    from paper_1703_09136_gb300 import FP64, MIXED, Plan
    cases = []
    for k, n in ((4.0, 200), (300.0, 220)):
        xy = W.points_in_box(1, n, ((0.0, 1.0), (0.05, 1.05)), salt=n)
        plan = Plan(xy, W.Medium(W.IMPEDANCE, (k,), alpha=1.0), tol=1e-6, levels=2, precision=MIXED if mixed else FP64)
        q = torch.from_numpy(W.strengths(1, n, 1, salt=n).astype(np.complex64 if mixed else np.complex128)).cuda()
        cases.append((plan, q, plan.apply(q).cpu().numpy()))

    def body(plan, q, want):
        def run():
            stream = torch.cuda.Stream()
            out = torch.empty_like(q)
            for _ in range(1500):
                plan.apply(q, out=out, stream=stream)
            stream.synchronize()
            assert np.array_equal(out.cpu().numpy(), want)
        return run
    torch.cuda.synchronize()
    _in_threads([body(*c) for c in cases])
    for plan, _, _ in cases:
        plan.close()


def test_plans_of_different_orders_from_two_threads():
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    xy = W.points_in_box(1, 200, ((0.0, 1.0), (0.05, 1.05)), salt=8)
    q = torch.from_numpy(W.strengths(1, 200, 1, salt=8)).cuda()
    med = W.Medium(W.IMPEDANCE, (20.0,), alpha=10.0)
    want = {}
    for p in (4, 60):
        with Plan(xy, med, p=p, levels=2) as plan:
            want[p] = plan.apply(q).cpu().numpy()
    torch.cuda.synchronize()

    def body(p):
        def run():
            stream = torch.cuda.Stream()
            for _ in range(12):
                with Plan(xy, med, p=p, levels=2, stream=stream) as plan:
                    out = torch.empty_like(q)
                    plan.apply(q, out=out, stream=stream)
                    stream.synchronize()
                    assert np.array_equal(out.cpu().numpy(), want[p])
        return run
    _in_threads([body(4), body(60)])
