"""Integer-state refinement of the heat operator (steps without forcing) against the oracle: long decays (the state is
rescaled on the way), states of any magnitude, both initial guesses, grids on chip and in global memory, inputs that are
not finite, and the tolerance at which the FP64 check takes over.

Tolerance: every step's residual is at most rtol ||b|| and the form's own error a quarter of that, ||A^-1|| <= 1: S
steps are within 1.25 S rtol of the exact propagation relative to the state that decays least, 1e-9 for the S used."""
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


def opts(rtol=1e-11, guess=B.PIT_GUESS_DEFAULT):
    return B.solve_opts(B.PIT_PREC_MIXED, rtol=rtol, maxit=4000, inner_rtol=1e-6, ir_maxit=12, guess=guess)


def solve(P, u, dt, steps, o):
    out = torch.empty(P.n_total, dtype=torch.float64, device="cuda")
    st = P.sequential_solve(torch.from_numpy(u).cuda(), dt, steps, out, o)
    return out.cpu().numpy(), st


def worst(P, a, b):
    return max(np.linalg.norm(a[P.offsets[g]:P.offsets[g + 1]] - b[P.offsets[g]:P.offsets[g + 1]]) /
               np.linalg.norm(b[P.offsets[g]:P.offsets[g + 1]]) for g in range(P.G))


@pytest.mark.parametrize("guess", [B.PIT_GUESS_PREVIOUS, B.PIT_GUESS_EXTRAPOLATE])
@pytest.mark.parametrize("d,n,dt,steps", [(1, 5, 0.2, 60), (2, 5, 0.05, 60), (3, 4, 1e-3, 33), (4, 4, 1e-3, 20),
                                          (6, 3, 1e-3, 20)])
def test_long_decay_matches_oracle(d, n, dt, steps, guess):
    P = B.Problem(d, n, 1, W.OP_HEAT)
    O = oracle.Problem(d, n, 1, W.OP_HEAT)
    u = O.initial(W.IC_SINES, W.random_sine_modes(d, 4, 2, seed=3)) + 0.3 * O.initial(W.IC_SINES, W.sine_modes(d, [(1.0, [1] * d)]))
    got, st = solve(P, u, dt, steps, opts(guess=guess))
    assert st.n_failed == 0
    ref = O.sequential(u, dt, steps, rtol=1e-15)
    # (the lowest mode decays least: later residuals are relative to it)
    assert worst(P, got, ref) < 1e-9


def test_states_of_any_magnitude_scale_exactly():
    # the state is held times a power of two taken from its norm: results scale bit by bit
    P = B.Problem(3, 5, 1, W.OP_HEAT)
    u = W.random_vector(9, P.n_total)
    a, _ = solve(P, u, 1e-3, 12, opts())
    for e in (-300, -40, 40, 300):
        b, _ = solve(P, np.ldexp(u, e), 1e-3, 12, opts())
        np.testing.assert_array_equal(b, np.ldexp(a, e))
    z, st = solve(P, np.zeros(P.n_total), 1e-3, 12, opts())
    assert st.n_failed == 0 and not z.any()


def test_rough_states_and_global_memory_grids():
    # a line of 16,383 nodes needs the global-state variant
    P = B.Problem(1, 14, 1, W.OP_HEAT)
    O = oracle.Problem(1, 14, 1, W.OP_HEAT)
    u = W.random_vector(4, P.n_total)
    dt = 1e-9  # dt / h^2 = 0.27
    got, st = solve(P, u, dt, 6, opts())
    assert st.n_failed == 0
    assert worst(P, got, O.sequential(u, dt, 6, rtol=1e-15)) < 1e-9


def test_tight_tolerances_and_bad_inputs():
    P = B.Problem(2, 6, 1, W.OP_HEAT)
    O = oracle.Problem(2, 6, 1, W.OP_HEAT)
    u = O.initial(W.IC_SINES, W.random_sine_modes(2, 4, 3, seed=5))
    got, st = solve(P, u, 1e-3, 10, opts(rtol=2e-14))  # below what the integer residual is used for
    assert st.n_failed == 0
    assert worst(P, got, O.sequential(u, 1e-3, 10, rtol=1e-15)) < 1e-11
    for bad in (np.nan, np.inf):
        v = u.copy()
        v[P.offsets[2] + 1] = bad
        out = torch.empty(P.n_total, dtype=torch.float64, device="cuda")
        with pytest.raises(B.PitError) as e:
            P.sequential_solve(torch.from_numpy(v).cuda(), 1e-3, 3, out, opts())
        assert e.value.status == B.PIT_ERR_NONFINITE
        got = out.cpu().numpy()  # the other grids are solved
        ref = O.sequential(u, 1e-3, 3, rtol=1e-15)
        for g in range(P.G):
            sl = slice(P.offsets[g], P.offsets[g + 1])
            if g != 2:
                assert np.linalg.norm(got[sl] - ref[sl]) < 1e-9 * np.linalg.norm(ref[sl])


# The axes with one node add 2 dt / h^2 each to the diagonal, more than the listed axes where those are short: steps on
# both sides of the points where that sum passes a power of two, boxes with extents of their own, a minimum level above 1.
@pytest.mark.parametrize("d,n,L0,hi,dts", [
    (3, 2, 1, None, [0.1, 0.12, 0.13, 0.16, 0.2, 0.26, 0.32]),
    (4, 4, 1, None, [0.05, 0.08, 0.085, 0.12, 0.13, 0.2]),
    (6, 3, 1, None, [0.04, 0.05, 0.054, 0.06, 0.08, 0.09, 0.11, 0.16, 0.25]),
    (2, 3, 1, [1.0, 0.1], [0.002, 0.0026, 0.004, 0.0045, 0.006]),
    (3, 6, 1, [0.2, 1.0, 0.5], [0.005, 0.01, 0.015, 0.02, 0.03, 0.04]),
    (2, 5, 2, [0.5, 1.0], [0.01, 0.05, 0.2])])
def test_one_node_axes_at_large_steps(d, n, L0, hi, dts):
    box = ([0.0] * d, hi or [1.0] * d)
    P = B.Problem(d, n, L0, W.OP_HEAT, *box)
    O = oracle.Problem(d, n, L0, W.OP_HEAT, *box)
    u = W.random_vector(13, P.n_total)
    for dt in dts:
        got, st = solve(P, u, dt, 1, opts())
        assert st.n_failed == 0, dt
        assert worst(P, got, O.phi(dt, u, rtol=1e-15)) < 1e-9, dt


def states(O, u, dt, steps):
    out = [u]
    for _ in range(steps):
        out.append(O.phi(dt, out[-1], rtol=1e-15))
    return out


# A step that shrinks the state many times over: the extrapolated guess is then about the state before, far larger than
# the state whose norm the integers are scaled by.  Each step's residual is at most 1.25 rtol ||x_{s-1}|| and
# ||A^-1|| <= 1, so the state is off by 1.25 rtol times the sum of the earlier states' norms.
@pytest.mark.parametrize("d,n,dt,steps,kind", [
    (4, 1, 1.0, 2, "random"), (4, 1, 1.0, 12, "random"), (6, 1, 0.9, 5, "random"), (1, 4, 0.05, 4, "highest"),
    (1, 4, 0.5, 6, "random"), (1, 4, 0.5, 8, "highest"), (1, 6, 0.02, 6, "spike"), (1, 8, 0.01, 8, "spike"),
    (2, 5, 0.3, 6, "random"), (3, 5, 0.05, 10, "spike"), (3, 4, 0.9, 6, "random"), (6, 3, 0.5, 6, "random")])
def test_steps_that_shrink_the_state_many_times_over(d, n, dt, steps, kind):
    P = B.Problem(d, n, 1, W.OP_HEAT)
    O = oracle.Problem(d, n, 1, W.OP_HEAT)
    u = W.random_vector(17, P.n_total)
    for g in range(P.G):
        sl = slice(P.offsets[g], P.offsets[g + 1])
        m = P.offsets[g + 1] - P.offsets[g]
        if kind == "highest":
            u[sl] = np.sin(np.pi * m * np.arange(1, m + 1) / (m + 1))
        elif kind == "spike":
            u[sl] = 0.0
            u[sl][m // 2] = 1.0
    ref = states(O, u, dt, steps)
    for guess in (B.PIT_GUESS_PREVIOUS, B.PIT_GUESS_EXTRAPOLATE):
        got, st = solve(P, u, dt, steps, opts(guess=guess))
        assert st.n_failed == 0
        for g in range(P.G):
            sl = slice(P.offsets[g], P.offsets[g + 1])
            off = np.linalg.norm(got[sl] - ref[-1][sl])
            assert off <= 1.25e-11 * sum(np.linalg.norm(r[sl]) for r in ref[:-1]), g


def test_states_near_the_end_of_the_double_range():
    # a squared norm of up to 1.8e308 is finite, as in the form with the FP64 check
    P = B.Problem(3, 5, 1, W.OP_HEAT)
    u = W.random_vector(9, P.n_total)
    most = max(float(np.sum(u[P.offsets[g]:P.offsets[g + 1]] ** 2)) for g in range(P.G))
    e = (1023 - int(np.ceil(np.log2(most)))) // 2  # the largest norm squared times 4^e is below 2^1023
    assert np.ldexp(most, 2 * e) > 1e304
    a, _ = solve(P, u, 1e-3, 12, opts())
    b, st = solve(P, np.ldexp(u, e), 1e-3, 12, opts())
    assert st.n_failed == 0
    np.testing.assert_array_equal(b, np.ldexp(a, e))
    with pytest.raises(B.PitError) as err:
        solve(P, np.ldexp(u, e + 3), 1e-3, 12, opts())
    assert err.value.status == B.PIT_ERR_NONFINITE


def test_states_whose_squares_leave_the_double_range():
    # norms from 2^-500 to 2^-750: the squared norm is subnormal or zero from about 2^-511 on
    P = B.Problem(3, 5, 1, W.OP_HEAT)
    u = W.random_vector(9, P.n_total)
    a, _ = solve(P, u, 1e-3, 12, opts())
    for e in (-500, -512, -520, -535, -545, -750):
        b, st = solve(P, np.ldexp(u, e), 1e-3, 12, opts())
        assert st.n_failed == 0
        np.testing.assert_array_equal(b, np.ldexp(a, e))


@pytest.mark.parametrize("prec", [B.PIT_PREC_MIXED, B.PIT_PREC_FP64])
def test_steps_of_length_zero_return_the_state(prec):
    P = B.Problem(3, 5, 1, W.OP_HEAT)
    u = W.random_vector(9, P.n_total) * 10.0 ** W.random_vector(10, P.n_total, -40, 0)
    for steps in (1, 5):
        got, st = solve(P, u, 0.0, steps, B.solve_opts(prec, rtol=1e-11, maxit=4000, inner_rtol=1e-6, ir_maxit=12))
        assert st.n_failed == 0
        np.testing.assert_array_equal(got, u)
