"""FP64 drift operators on grids too large for one SM, a cluster per grid (narrow batches), against the oracle: the three
operators, mixed derivatives, two and three axes, forcing, several entries, and failures.

Tolerance 1e-10: both sides solve to 1e-13 or tighter, their difference is about kappa 1e-13 a step (kappa < 100 here)."""
import numpy as np
import pytest

import oracle
from paper_2509_22156_gb300 import binding as B
from paper_2509_22156_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

A2, H2 = np.array([[0.0, 1.0], [-1.0, -0.1]]), np.array([[0.3, 0.1], [0.1, 0.2]])
A3, H3 = np.array([[-1.0, 0.5, 0.0], [0.0, -0.5, 0.3], [0.2, 0.0, -1.0]]), np.diag([0.5, 0.4, 0.3]) + 0.05
RATES = (3e3, 1.1e4, 2.0, 1e-3)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_22156_gb300 import build
    build.build()
    B.load()
    torch.cuda.set_device(0)


def make(name):
    if name == "ou":
        a = (2, 12, 5, B.PIT_OP_OU, [-6.0] * 2, [6.0] * 2)
        return B.Problem(*a), oracle.Problem(*a), 1e-3
    if name == "cme":
        a = (2, 12, 5, B.PIT_OP_CME, [0.0] * 2, [399.0] * 2)
        return B.Problem(*a, cme=RATES, drift_scheme=1), oracle.Problem(*a, cme=RATES, central=True), 1.0
    if name == "lsde2":
        a = (2, 12, 5, B.PIT_OP_LSDE, [-10.0] * 2, [10.0] * 2)
        return (B.Problem(*a, drift=A2, diffusion=H2, drift_scheme=1),
                oracle.Problem(*a, drift=A2, diffusion=H2, central=True), 1e-3)
    a = (3, 11, 4, B.PIT_OP_LSDE, [-4.0] * 3, [4.0] * 3)  # 15 x 15 x 31 nodes: a reach of 496
    return B.Problem(*a, drift=A3, diffusion=H3), oracle.Problem(*a, drift=A3, diffusion=H3), 1e-3


def opts(**kw):
    return B.solve_opts(B.PIT_PREC_FP64, **{**dict(rtol=1e-13, maxit=20000), **kw})


@pytest.mark.parametrize("name", ["ou", "cme", "lsde2", "lsde3"])
def test_cluster_steps_match_oracle(name):
    P, O, dt = make(name)
    assert max(np.diff(P.offsets)) > 2600  # beyond one SM's shared memory in FP64
    u = np.abs(W.random_vector(3, P.n_total)) + 0.1
    out = torch.empty(P.n_total, dtype=torch.float64, device="cuda")
    st = P.sequential_solve(torch.from_numpy(u).cuda(), dt, 3, out, opts())
    assert st.n_failed == 0 and st.n_items == 3 * P.G
    ref = O.sequential(u, dt, 3, rtol=1e-15)
    got = out.cpu().numpy()
    for g in range(P.G):
        sl = slice(P.offsets[g], P.offsets[g + 1])
        assert np.linalg.norm(got[sl] - ref[sl]) < 1e-10 * np.linalg.norm(ref[sl]), g
    # a batch of two with forcing
    u2, f2 = np.abs(W.random_vector(4, 2 * P.n_total)), W.random_vector(5, 2 * P.n_total)
    o2 = torch.empty(2 * P.n_total, dtype=torch.float64, device="cuda")
    P.phi_batch(dt, torch.from_numpy(u2).cuda(), o2, opts(), f=torch.from_numpy(f2).cuda())
    ref = O.phi(dt, u2, f2, rtol=1e-15)
    assert np.linalg.norm(o2.cpu().numpy() - ref) < 1e-10 * np.linalg.norm(ref)


def test_cluster_reports_failures():
    P, O, dt = make("lsde2")
    u = np.abs(W.random_vector(3, P.n_total))
    ud, out = torch.from_numpy(u).cuda(), torch.empty(P.n_total, dtype=torch.float64, device="cuda")
    with pytest.raises(B.PitError) as e:
        P.phi_batch(0.1, ud, out, opts(rtol=1e-14, maxit=1))
    assert e.value.status == B.PIT_ERR_NOCONV
    v = u.copy()
    v[P.offsets[1] + 7] = np.nan
    with pytest.raises(B.PitError) as e:
        P.phi_batch(dt, torch.from_numpy(v).cuda(), out, opts())
    assert e.value.status == B.PIT_ERR_NONFINITE
    P.phi_batch(dt, ud, out, opts())
    assert np.linalg.norm(out.cpu().numpy() - O.phi(dt, u, rtol=1e-15)) < 1e-10 * np.linalg.norm(u)


def test_mgrit_with_clusters_matches_sequential():
    # sweeps (narrow, a caller's guess, additive forcing, stored steps) run in clusters, relaxations do not
    P, O, dt = make("cme")
    u = np.exp(-0.5 * ((np.arange(P.n_total) % 97) / 20.0) ** 2) + 0.1
    uT, seq = (torch.empty(P.n_total, dtype=torch.float64, device="cuda") for _ in range(2))
    ud = torch.from_numpy(u).cuda()
    fine = opts(rtol=1e-12)
    for fas in (False, True):
        o = B.mgrit_opts(0.0, 32 * dt, 32, 4, 2, tol=1e-9, maxit=40, fine=fine, crs=fine, fas=fas, init=1)
        P.mgrit_solve(ud, o, uT)
        P.sequential_solve(ud, dt, 32, seq, fine)
        assert torch.linalg.norm(uT - seq) < 1e-8 * torch.linalg.norm(seq)


def test_cluster_sizes_and_problems_take_turns():
    # batches of one and two states take clusters of different sizes, whose CTAs need different shared memory, and so do
    # problems of different size: every earlier choice still runs after a later one
    def probs():
        for n in (12, 13):
            a = (2, n, 5, B.PIT_OP_OU, [-6.0] * 2, [6.0] * 2)
            yield B.Problem(*a), oracle.Problem(*a)
    pairs = list(probs())
    ref = {}
    for k, nb in [(1, 2), (1, 1), (1, 2), (0, 1), (1, 1), (0, 2), (1, 2), (0, 3), (0, 1)]:
        P, O = pairs[k]
        u = np.abs(W.random_vector(5 + k, P.n_total)) + 0.1
        out = torch.empty(nb * P.n_total, dtype=torch.float64, device="cuda")
        P.phi_batch(1e-3, torch.from_numpy(np.tile(u, nb)).cuda(), out, opts(), n_batch=nb)
        if k not in ref:
            ref[k] = O.phi(1e-3, u, rtol=1e-15)
        got = out.cpu().numpy().reshape(nb, -1)
        assert np.linalg.norm(got - ref[k]) < 1e-10 * np.linalg.norm(ref[k]) * np.sqrt(nb)
