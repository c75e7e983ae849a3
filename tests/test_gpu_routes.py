"""Both sides of the rules that choose a kernel, against the oracle.

Direct solve or CG of the heat refinements: dt / h^2 of the finest axis just below and above the line, for calls of one
step, of several, with and without forcing.  Every step's residual is at most 1.25 rtol ||b|| and ||A^-1|| <= 1, so the
result is off by at most 1.25 rtol sum ||b_s||.

Bodies of the steps kernel: grids of one to all axes in launches that run one body for all of them and in launches where
each grid runs its own (the FP64 form; the variable-coefficient operator with few large grids), every operator and form.
Tolerance 1e-9 for the refinements and FP64 (one step solved to 1e-12 and 1e-13 against 1e-15, condition numbers below
100) and 1e-4 for the FP32 form at rtol 1e-6 (FP32 rounding of a solve of condition 100: 1e-5)."""
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


@pytest.mark.parametrize("prec", [B.PIT_PREC_MIXED, B.PIT_PREC_MIXED_PAIR])
@pytest.mark.parametrize("d,n", [(1, 7), (2, 6), (3, 5), (5, 4)])
@pytest.mark.parametrize("steps,forced,line", [(1, False, 1.5), (1, True, 1.5), (4, True, 0.5), (4, False, 5.0)])
def test_both_sides_of_the_direct_solve(d, n, prec, steps, forced, line):
    P = B.Problem(d, n, 1, W.OP_HEAT)
    O = oracle.Problem(d, n, 1, W.OP_HEAT)
    u = W.random_vector(51, P.n_total)
    F = W.random_vector(52, steps * P.n_total).reshape(steps, -1) if forced else None
    its = []
    for x in (0.9 * line, 1.1 * line):
        dt = x / 4.0 ** n
        ref, off = u, np.zeros(P.G)
        for s in range(steps):
            b = ref + dt * F[s] if forced else ref
            off += [np.linalg.norm(b[P.offsets[g]:P.offsets[g + 1]]) for g in range(P.G)]
            ref = O.phi(dt, ref, f=F[s] if forced else None, rtol=1e-15)
        out = torch.empty(P.n_total, dtype=torch.float64, device="cuda")
        o = B.solve_opts(prec, rtol=1e-11, maxit=4000, inner_rtol=1e-6, ir_maxit=12)
        f = torch.from_numpy(F.reshape(-1)).cuda() if forced else None
        ud = torch.from_numpy(u).cuda()
        st = P.sequential_solve_forced(ud, dt, steps, out, o, forcing=f) if forced else P.sequential_solve(ud, dt, steps, out, o)
        assert st.n_failed == 0
        got = out.cpu().numpy()
        for g in range(P.G):
            sl = slice(P.offsets[g], P.offsets[g + 1])
            assert np.linalg.norm(got[sl] - ref[sl]) <= 1.25e-11 * off[g], (x, g)
        its.append(st.sum_iters)
    if steps == 1 and d in (2, 3):  # (one axis: the line preconditioner of CG is a direct solve too)
        assert its[0] > its[1]  # CG iterations on the milder step, a direct solve a pass on the other


OPS = {"heat": (W.OP_HEAT, 0.0, 1.0, 1e-3), "varheat": (W.OP_VARHEAT, 0.0, 1.0, 1e-3), "ou": (B.PIT_OP_OU, -6.0, 6.0, 1e-2)}


@pytest.mark.parametrize("prec", [B.PIT_PREC_FP64, B.PIT_PREC_MIXED, B.PIT_PREC_FP32, B.PIT_PREC_MIXED_PAIR])
@pytest.mark.parametrize("op,d,n,nb", [("heat", 4, 4, 3), ("heat", 6, 3, 2), ("ou", 2, 5, 1), ("ou", 4, 4, 3), ("ou", 5, 3, 1),
                                       ("varheat", 2, 4, 1), ("varheat", 2, 8, 1), ("varheat", 2, 8, 12), ("varheat", 3, 5, 1),
                                       ("varheat", 4, 4, 2)])
def test_grids_of_every_number_of_axes(op, d, n, nb, prec):
    if op == "ou" and prec == B.PIT_PREC_MIXED_PAIR:
        pytest.skip("the pair form is for the symmetric operators")
    code, lo, hi, dt = OPS[op]
    P = B.Problem(d, n, 1, code, [lo] * d, [hi] * d)
    O = oracle.Problem(d, n, 1, code, [lo] * d, [hi] * d)
    u = np.abs(W.random_vector(61 + d, P.n_total)) + 0.1
    out = torch.empty(nb * P.n_total, dtype=torch.float64, device="cuda")
    rtol = {B.PIT_PREC_FP64: 1e-13, B.PIT_PREC_FP32: 1e-6}.get(prec, 1e-12)
    if prec == B.PIT_PREC_MIXED_PAIR:
        rtol = max(rtol, 2.0 ** -45 * (1 + 4 * dt * 4.0 ** n))  # above the form's floor
    precond = B.PIT_PRECOND_NONE if op == "heat" else 0  # (the steps kernel in every form)
    st = P.phi_batch(dt, torch.from_numpy(np.tile(u, nb)).cuda(), out,
                     B.solve_opts(prec, rtol=rtol, maxit=20000, inner_rtol=1e-5, ir_maxit=40, precond=precond), n_batch=nb)
    assert st.n_failed == 0
    ref, got = O.phi(dt, u, rtol=1e-15), out.cpu().numpy().reshape(nb, -1)
    for g in range(P.G):
        sl = slice(P.offsets[g], P.offsets[g + 1])
        for b in (0, nb - 1):
            assert np.linalg.norm(got[b, sl] - ref[sl]) < (1e-4 if prec == B.PIT_PREC_FP32 else 1e-9) * np.linalg.norm(ref[sl]), g
