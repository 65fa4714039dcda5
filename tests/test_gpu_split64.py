"""FP64 translations as exact-slice tensor-core products (split64.cu) where
tiles, chunks and exponents have their edges: trees of one to six levels (target
rows narrower than a tile, partly empty, wider than 16 columns of one parity),
orders below, at and above a 32-coefficient chunk, ragged right-hand sides,
strengths far from one, and non-finite strengths."""
import numpy as np
import pytest

import workloads as W
from oracle import direct, fmm

pytestmark = pytest.mark.gpu

MEDIA = {"imp": W.WORKLOADS[1].medium, "imp-hi": W.Medium(W.IMPEDANCE, (90.0,), alpha=30.0),
         "two": W.WORKLOADS[3].medium, "three": W.WORKLOADS[4].medium}
TOL = 1e-11      # FP64 bound of the parity tests: FP64 against the CPU FMM at equal order


def _torch():
    return pytest.importorskip("torch")


def _case(medium, n, salt):
    xy = W.points_in_box(1, n, ((0.0, 1.0), (0.02, 1.02)), salt=salt)
    return MEDIA[medium], xy


@pytest.mark.parametrize("medium,n,levels,nrhs", [
    ("imp", 300, 2, 1), ("imp", 700, 3, 2), ("two", 900, 4, 3), ("three", 1200, 5, 1), ("three", 900, 6, 9),
    ("imp-hi", 500, 2, 2), ("imp-hi", 900, 3, 1)])
def test_split_translations_match_cpu_fmm(medium, n, levels, nrhs):
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    med, xy = _case(medium, n, levels)
    q = W.strengths(1, n, nrhs, salt=levels)
    ref = fmm.CpuFmm(xy, med, tol=1e-6, L=levels).apply(q)
    with Plan(xy, med, tol=1e-6, levels=levels, max_rhs=nrhs, dense_m2l=True) as plan:
        y = plan.apply(torch.from_numpy(q).cuda()).cpu().numpy()
        assert direct.rel_l2(y, ref) < TOL, direct.rel_l2(y, ref)
        # one right-hand side of a wider plan, and strengths near the ends of the range
        for scale in (1e-200, 1e200):
            ys = plan.apply(torch.from_numpy(q[:1] * scale).cuda()).cpu().numpy() / scale
            assert direct.rel_l2(ys, ref[:1]) < TOL, (scale, direct.rel_l2(ys, ref[:1]))


def test_split_translations_wide_rows():
    """Seven levels: rows of 64 boxes of one parity, so tiles of 16 columns, and
    the reaction lists as a launch of their own; against the direct sum
    of 300 sources at 500 points."""
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 40000
    med, xy = _case("two", n, 7)
    g = np.random.default_rng(5)
    q = np.zeros((2, n), dtype=complex)
    src = g.choice(n, 300, replace=False)
    q[:, src] = g.standard_normal((2, 300)) + 1j * g.standard_normal((2, 300))
    idx = np.union1d(src, g.choice(n, 200, replace=False))       # every other strength is zero
    ref = direct.direct_apply(med, xy[idx], q[:, idx])
    with Plan(xy, med, tol=1e-10, levels=7, max_rhs=2) as plan:
        y = plan.apply(torch.from_numpy(q).cuda()).cpu().numpy()
    assert direct.rel_l2(y[:, idx], ref) < 1e-9


def test_split_translations_zero_and_nonfinite():
    torch = _torch()
    from paper_1703_09136_gb300 import Plan
    n = 800
    med, xy = _case("imp", n, 11)
    q = W.strengths(1, n, 3, salt=3)
    q[1] = 0.0
    q[2, 17] = np.nan
    with Plan(xy, med, tol=1e-6, levels=3, max_rhs=3) as plan:
        y = plan.apply(torch.from_numpy(q).cuda()).cpu().numpy()
        y0 = plan.apply(torch.from_numpy(q[:1]).cuda()).cpu().numpy()
    assert np.array_equal(y[0], y0[0])           # neighbours do not change a right-hand side
    assert np.all(y[1] == 0.0)
    assert np.all(np.isnan(y[2].real) & np.isnan(y[2].imag))
