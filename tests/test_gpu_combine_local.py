"""Combination sum at points: the error at a point is relative to the values near it, for few points (the sum over
grids) and for many (groups of grids added first), on states whose values span many orders of magnitude.

Tolerance: on its way into the sum a value is rounded at most 5 d + 2 times as a member of its grid or group (weights,
products, the member's line), then in a sum of G grids and, grid by grid, 2^d corners: (5 d + 2 + G + 2^d) 2^-53 of
sum_l |c_l| I_l[|u_l|](x).  The reference is the sum over grids in extended precision, at the same place in the cells."""
import itertools
import math

import numpy as np
import pytest

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


def by_grids(P, lo, hi, u, pts):
    """(sum, sum of magnitudes) in extended precision."""
    X = np.longdouble
    h = (hi - lo) / (1 << int(P.levels[0][0]))
    xr = (pts - lo) / (h * (1 << int(P.levels[0][0])))  # in FP64, as the kernels place the points
    total, size = np.zeros(len(pts), X), np.zeros(len(pts), X)
    for g in range(P.G):
        lev = [int(l) for l in P.levels[g]]
        v = np.pad(u[P.offsets[g]:P.offsets[g + 1]].reshape([(1 << l) - 1 for l in lev]), 1).astype(X)
        cells, ts = [], []
        for i, l in enumerate(lev):
            s = xr[:, i].astype(X) * (1 << l)
            k = np.clip(np.floor(s).astype(int), 0, (1 << l) - 1)
            cells.append(k)
            ts.append(s - k)
        w = lev_weight(P, g)
        for corner in itertools.product((0, 1), repeat=P.d):
            c = np.ones(len(pts), X)
            for i in range(P.d):
                c = c * (ts[i] if corner[i] else 1 - ts[i])
            x = v[tuple(k + b for k, b in zip(cells, corner))]
            total += w * c * x
            size += np.abs(w * c * x)
    return total, size


def lev_weight(P, g):
    k = int(P.levels[0].sum()) - int(P.levels[g].sum())
    return (-1) ** k * math.comb(P.d - 1, k)


@pytest.mark.parametrize("d,n,L0,kind", [(2, 8, 1, "density"), (2, 9, 1, "density"), (3, 6, 1, "spike"), (3, 7, 2, "spike"),
                                         (4, 5, 1, "density"), (4, 5, 1, "spike"), (5, 4, 1, "rough"), (6, 4, 1, "spike")])
def test_errors_are_relative_to_the_values_near_a_point(d, n, L0, kind):
    lo, hi = (-6.0, 6.0) if kind == "density" else (0.0, 1.0)
    P = B.Problem(d, n, L0, B.PIT_OP_OU if kind == "density" else B.PIT_OP_HEAT, [lo] * d, [hi] * d)
    u = W.random_vector(41, P.n_total)
    if kind == "density":  # values from 1 down to 1e-60
        s = torch.empty(P.n_total, dtype=torch.float64, device="cuda")
        P.sample_initial(1, np.array([1.0] * d + [0.5] * d), s)
        u = s.cpu().numpy()
    elif kind == "spike":  # one node of every grid far above the others
        for g in range(P.G):
            u[P.offsets[g] + (P.offsets[g + 1] - P.offsets[g]) // 3] = 1e18
    n_pts = 200000 if d == 2 else 65537
    pts = W.random_vector(43, n_pts * d, lo, hi).reshape(n_pts, d)
    pts[:64] = lo + (hi - lo) * (1.3 * (pts[:64] - lo) / (hi - lo) - 0.15)  # some outside the box
    pts[64:80] = lo + (hi - lo) * np.round((pts[64:80] - lo) / (hi - lo) * 16) / 16  # some on nodes
    ud, pd = torch.from_numpy(u).cuda(), torch.from_numpy(pts).cuda()
    many, few = torch.empty(n_pts, dtype=torch.float64, device="cuda"), torch.empty(24, dtype=torch.float64, device="cuda")
    P.combine(ud, pd, many)
    some = np.unique(np.concatenate([np.arange(200), np.arange(0, n_pts, 97)]))[:1200]
    ref, size = by_grids(P, lo, hi, u, pts[some])
    tol = (5 * d + 2 + P.G + 2 ** d) * 2.0 ** -53 * size
    assert (np.abs(many.cpu().numpy()[some] - ref) <= tol).all()
    for at in range(0, len(some) - 24, 240):
        P.combine(ud, pd[some[at:at + 24]].contiguous(), few)
        assert (np.abs(few.cpu().numpy() - ref[at:at + 24]) <= tol[at:at + 24]).all()
    assert kind == "rough" or size.max() > 1e10 * size.min()  # (there are points where the largest value would not do as a scale)
