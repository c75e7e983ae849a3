"""Direct solves of the heat operator's refinements against the oracle: every line length a transform is built for
(3, 7, 15, 31 nodes), chunked lines beyond it, grids of one node, steps from mild to stiff, and the calls that keep
the Krylov solve (a chosen preconditioner, few iterations, huge steps, two long axes).

Tolerance: rtol = 1e-11 on every step's FP64 (pair) residual, and ||A^-1|| <= 1, so S steps differ from the exact
propagation by at most S * 1e-11 relative to the largest state; checked at 1e-9 for up to 20 steps.  The pair form's
residual floor is 2^-48 (1 + 4 sum dt / h^2) (its rtol is set above it)."""
import numpy as np
import pytest

import oracle
from paper_2509_22156_gb300 import binding as B
from paper_2509_22156_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (d, n, dt): longest axes of 7 .. 1023 nodes, second longest 1 .. 31
CASES = [(1, 3, 1e-3), (1, 5, 1e-3), (1, 6, 1e-3), (1, 10, 1e-5), (2, 2, 0.1), (2, 9, 1e-4), (2, 9, 0.5), (3, 8, 1e-3),
         (4, 6, 1e-2), (5, 5, 1e-3), (6, 4, 1e-2)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_22156_gb300 import build
    build.build()
    B.load()
    torch.cuda.set_device(0)


def per_grid(P, a, b):
    return max(np.linalg.norm(a[P.offsets[g]:P.offsets[g + 1]] - b[P.offsets[g]:P.offsets[g + 1]]) /
               max(np.linalg.norm(b[P.offsets[g]:P.offsets[g + 1]]), 1e-300) for g in range(P.G))


@pytest.mark.parametrize("prec", [B.PIT_PREC_MIXED, B.PIT_PREC_MIXED_PAIR])
@pytest.mark.parametrize("d,n,dt", CASES)
def test_direct_steps_match_oracle(d, n, dt, prec):
    P = B.Problem(d, n, 1, W.OP_HEAT)
    O = oracle.Problem(d, n, 1, W.OP_HEAT)
    ref = W.random_vector(7, P.n_total)  # rough: every mode of every axis
    u0 = torch.from_numpy(ref).cuda()
    uT = torch.empty_like(u0)
    steps = 3 if dt >= 0.1 else 20
    # (the largest dt / h^2 of the set bounds the pair form's floor)
    floor = 2.0 ** -46 * (1 + 4 * dt * 4.0 ** n)
    rtol = max(1e-11, 4 * floor) if prec == B.PIT_PREC_MIXED_PAIR else 1e-11
    st = P.sequential_solve(u0, dt, steps, uT, B.solve_opts(prec, rtol=rtol, maxit=20000, inner_rtol=1e-6, ir_maxit=40))
    assert st.n_failed == 0
    scale = 1.0
    for _ in range(steps):
        nxt = O.phi(dt, ref, rtol=1e-15)
        scale = max(scale, np.linalg.norm(ref) / np.linalg.norm(nxt))
        ref = nxt
    # relative to the last state, a residual of an earlier step counts as much larger as that state was
    assert per_grid(P, uT.cpu().numpy(), ref) < max(1e-9, steps * rtol * scale * 40)


def test_krylov_keeps_the_calls_the_direct_solve_does_not_take():
    # a solve that is left to CG: no preconditioner, two iterations, a huge step, two axes of 63 nodes
    P = B.Problem(2, 7, 1, W.OP_HEAT)
    O = oracle.Problem(2, 7, 1, W.OP_HEAT)
    u = W.random_vector(11, P.n_total)
    ud, out = torch.from_numpy(u).cuda(), torch.empty(P.n_total, dtype=torch.float64, device="cuda")
    its = {}
    for name, kw, dt in (("direct", {}, 1e-3), ("none", dict(precond=B.PIT_PRECOND_NONE), 1e-3), ("huge", {}, 2.0)):
        st = P.phi_batch(dt, ud, out, B.solve_opts(B.PIT_PREC_MIXED, rtol=1e-12, maxit=20000, inner_rtol=1e-5,
                                                   ir_maxit=40, **kw))
        assert per_grid(P, out.cpu().numpy(), O.phi(dt, u, rtol=1e-15)) < 1e-9
        its[name] = st.sum_iters / P.G
    assert its["direct"] <= 4 < its["none"] and its["huge"] > 4
    with pytest.raises(B.PitError) as e:
        P.phi_batch(1e-2, ud, out, B.solve_opts(B.PIT_PREC_MIXED, rtol=1e-12, maxit=2, inner_rtol=1e-5, ir_maxit=1))
    assert e.value.status == B.PIT_ERR_NOCONV
    Q = B.Problem(2, 11, 5, W.OP_HEAT)  # levels (5..7)^2: a grid of 63 x 63 nodes
    R = oracle.Problem(2, 11, 5, W.OP_HEAT)
    u = W.random_vector(12, Q.n_total)
    out = torch.empty(Q.n_total, dtype=torch.float64, device="cuda")
    st = Q.phi_batch(1e-3, torch.from_numpy(u).cuda(), out,
                     B.solve_opts(B.PIT_PREC_MIXED, rtol=1e-12, maxit=20000, inner_rtol=1e-5, ir_maxit=40))
    assert st.sum_iters / Q.G > 4
    assert per_grid(Q, out.cpu().numpy(), R.phi(1e-3, u, rtol=1e-15)) < 1e-9


@pytest.mark.parametrize("prec,forced", [(B.PIT_PREC_MIXED, False), (B.PIT_PREC_MIXED, True), (B.PIT_PREC_MIXED_PAIR, True)])
@pytest.mark.parametrize("d,n", [(1, 10), (2, 7), (2, 10)])
def test_chunked_lines_give_the_same_bits_every_time(d, n, prec, forced):
    # lines of 63 nodes and more are cut into chunks that exchange sums: every call has to see the same ones
    P = B.Problem(d, n, 1, W.OP_HEAT)
    u = torch.from_numpy(np.tile(W.random_vector(21, P.n_total), 24)).cuda()
    f = torch.from_numpy(np.tile(W.random_vector(22, P.n_total), 24)).cuda() if forced else None
    out = torch.empty_like(u)
    first = None
    for _ in range(20):
        P.phi_batch(1e-3, u, out, B.solve_opts(prec, rtol=1e-9, maxit=4000, inner_rtol=1e-5, ir_maxit=12), f=f, n_batch=24)
        first = out[:P.n_total].clone() if first is None else first
        assert bool((out.view(24, -1) == first).all())
