"""Combination sum from the sparse grid's surpluses (many points) against the oracle's sum over grids: dimensions 1 to 6,
a minimum level above one, points outside the box (the boundary cell's piece continued), chunks of increments, and a
state that is not finite (left to the sum over grids, point by point).

Tolerance 1e-12 of the largest |value|: sums over the increments (at most a few hundred here) of terms no larger than
the state, and grid coefficients with an absolute sum below 2,000: 2^-53 * 2,000 = 2.2e-13 a term of random sign."""
import numpy as np
import pytest

import oracle
from paper_2509_22156_gb300 import binding as B
from paper_2509_22156_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_22156_gb300 import build
    build.build()
    B.load()
    torch.cuda.set_device(0)


def kernels_of(P, u, pts, out):
    P.profile_enable(True)
    P.combine(u, pts, out)
    k = P.profile_read().kernels[2]
    P.profile_enable(False)
    return k


# (the last entry: whether the surpluses are the fewer operations)
@pytest.mark.parametrize("d,n,L0,n_pts,by_surpluses", [(1, 9, 1, 300000, False), (2, 8, 1, 200000, True),
                                                       (2, 9, 4, 51600, False), (3, 6, 1, 65537, True),
                                                       (3, 7, 2, 65537, True), (4, 5, 1, 30000, True),
                                                       (6, 4, 1, 4097, True)])
def test_combination_matches_oracle(d, n, L0, n_pts, by_surpluses):
    lo, hi = [-1.0] * d, [2.0] * d
    P = B.Problem(d, n, L0, W.OP_HEAT, lo, hi)
    O = oracle.Problem(d, n, L0, W.OP_HEAT, lo, hi)
    u = W.random_vector(31 + d, P.n_total)
    pts = W.random_vector(77 + d, n_pts * d, -1.2, 2.2).reshape(n_pts, d)
    pts[0] = lo
    pts[1] = hi
    pts[2] = 0.5
    out = torch.empty(n_pts, dtype=torch.float64, device="cuda")
    ud, pd = torch.from_numpy(u).cuda(), torch.from_numpy(pts).cuda()
    assert (kernels_of(P, ud, pd, out) > 2) == by_surpluses
    some = np.unique(np.concatenate([np.arange(64), np.arange(0, n_pts, max(1, n_pts // 2000))]))
    ref = O.combine(u, np.ascontiguousarray(pts[some]))
    got = out.cpu().numpy()[some]
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    small = torch.empty(16, dtype=torch.float64, device="cuda")
    assert kernels_of(P, ud, pd[:16].contiguous(), small) <= 2  # few points: the sum over grids
    assert np.abs(small.cpu().numpy() - out.cpu().numpy()[:16]).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_values_that_are_not_finite_stay_local(bad):
    P = B.Problem(3, 6, 1, W.OP_HEAT)
    u = W.random_vector(5, P.n_total)
    u[P.offsets[4] + 3] = bad
    pts = W.random_vector(6, 65537 * 3, 0.0, 1.0).reshape(-1, 3)
    ud, pd = torch.from_numpy(u).cuda(), torch.from_numpy(pts).cuda()
    out = torch.empty(len(pts), dtype=torch.float64, device="cuda")
    P.combine(ud, pd, out)
    few = torch.empty(600, dtype=torch.float64, device="cuda")
    P.combine(ud, pd[:600].contiguous(), few)  # the sum over grids
    a, b = out.cpu().numpy()[:600], few.cpu().numpy()
    assert np.isfinite(b).any() and not np.isfinite(out.cpu().numpy()).all()
    np.testing.assert_array_equal(np.isnan(a), np.isnan(b))
    np.testing.assert_allclose(a[np.isfinite(b)], b[np.isfinite(b)], rtol=1e-13, atol=1e-13)
