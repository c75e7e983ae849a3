"""Performance cases of the framework: the calls a user's program makes, over the range of problems it takes.

Every case goes through the public binding (``paper_2509_22156_gb300.binding.Problem``).  Kinds of call:

  mgrit      ``mgrit_solve``: the parallel-in-time solve of every component grid (a whole run of the method)
  seq        ``sequential_solve``: time-sequential backward-Euler stepping of every component grid
  phi        ``phi_batch``: one batched backward-Euler step of many states (the building block of a driver of one's own)
  combine    ``combine``: the combination sum at evaluation points (post-processing of every run)
  recombine  ``recombine``: projection of the combined solution onto every grid (between the intervals of a run)
  netgrad    ``net_loss_grad``: loss and gradient of the learned coarse propagator on one set of states

Problem sizes, operators and solver options are those of the measured workloads, the experiments of the paper that
the benchmark runs beside them, and of the tests.
"""
import itertools
import math
import random

import numpy as np
import torch

from paper_2509_22156_gb300 import binding as B

OPS = {"heat": B.PIT_OP_HEAT, "varheat": B.PIT_OP_VARHEAT, "ou": B.PIT_OP_OU, "lsde": B.PIT_OP_LSDE,
       "cme": B.PIT_OP_CME}
PRECS = {"fp64": B.PIT_PREC_FP64, "mixed": B.PIT_PREC_MIXED, "pair": B.PIT_PREC_MIXED_PAIR}
BOX = {"heat": (0.0, 1.0), "varheat": (0.0, 1.0), "ou": (-6.0, 6.0), "lsde": (-10.0, 10.0), "cme": (0.0, 399.0)}
VAMP = 0.5
LSDE_A = [[0.0, 1.0], [-1.0, -0.1]]   # linear oscillator, Sec. 4.4.1 of the paper
LSDE_H = [[0.0, 0.0], [0.0, 0.2]]
CME_RATES = (3e3, 1.1e4, 2.0, 1e-3)   # toggle switch, Sec. 4.3 (production, saturation, exponent, degradation)


# ---------------------------------------------------------------------------------------------------------------
# cases
def listed():
    return [
        # the smallest whole solve: the paper's algorithm as printed (FAS, FCF) in FP64 on 273 nodes, where launches
        # and the latency of a step count
        dict(name="mgrit_heat2d_n5", kind="mgrit", op="heat", d=2, n=5, L0=1, form="plain", nsteps=64, m=4, levels=2,
             dt=0.1 / 64),
        # an ordinary whole solve: 109 grids, 1024 steps, refinement fine solves, FP32 coarse solves, lanes
        dict(name="mgrit_heat3d_n9", kind="mgrit", op="heat", d=3, n=9, L0=1, form="chosen", nsteps=1024, m=16,
             levels=2, dt=0.05 / 1024),
        # the largest whole solve: the benchmark's headline problem (4,921 grids, 11.9 M nodes, three levels) over half
        # of its time interval
        dict(name="mgrit_heat6d_n10", kind="mgrit", op="heat", d=6, n=10, L0=1, form="chosen", nsteps=256, m=16,
             levels=3, dt=0.02 / 512),
        # sequential stepping where the grids alone fill the GPU (one state, thousands of grids)
        dict(name="seq_heat6d_n9", kind="seq", op="heat", d=6, n=9, L0=1, prec="mixed", nsteps=128, dt=0.02 / 512),
        # sequential stepping of fewer grids than the GPU has SMs, symmetric operator with a coefficient table
        dict(name="seq_varheat3d_n8", kind="seq", op="varheat", d=3, n=8, L0=1, prec="mixed", nsteps=256,
             dt=0.1 / 2048),
        # sequential stepping of a drift operator (BiCGStab) in refinement
        dict(name="seq_ou4d_n7", kind="seq", op="ou", d=4, n=7, L0=1, prec="mixed", nsteps=512, dt=1.0 / 512),
        # the paper's oscillator at its own grid set: 7 grids of up to 32,385 nodes in FP64
        dict(name="seq_lsde2d_n14", kind="seq", op="lsde", d=2, n=14, L0=6, prec="fp64", nsteps=96, dt=1.0 / 3200),
        # the paper's toggle switch at its own grid set: 5 grids, 64,261 nodes, FP64
        dict(name="seq_cme2d_n13", kind="seq", op="cme", d=2, n=13, L0=6, prec="fp64", nsteps=256, dt=1.0),
        # one batched step with forcing, refinement on FP32 pairs
        dict(name="phi_heat3d_n9_b64", kind="phi", op="heat", d=3, n=9, L0=1, prec="pair", batch=64, forcing=True,
             dt=0.05 / 1024),
        # evaluation of the combined solution at the benchmark's number of points
        dict(name="combine_ou4d_n7", kind="combine", op="ou", d=4, n=7, L0=1, npts=65794),
        # recombination of the headline problem's state
        dict(name="recombine_heat6d_n10", kind="recombine", op="heat", d=6, n=10, L0=1),
        # loss and gradient of the learned coarse propagator over one state of every grid (a training batch)
        dict(name="netgrad_varheat3d_n8", kind="netgrad", op="varheat", d=3, n=8, L0=1, batch=1, dT=0.1 / 64),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["mgrit", "seq", "seq", "phi", "combine", "recombine", "netgrad"])
    if kind == "mgrit":
        which = rng.randrange(3)
        if which == 0:
            return dict(kind=kind, op="heat", d=2, n=rng.randint(4, 7), L0=1, form="plain", nsteps=4 * rng.randint(7, 31),
                        m=4, levels=2, dt=0.1 / 64)
        if which == 1:
            return dict(kind=kind, op="heat", d=3, n=rng.randint(6, 9), L0=1, form="chosen",
                        nsteps=16 * rng.randint(15, 63), m=16, levels=2, dt=0.05 / 1024)
        return dict(kind=kind, op="heat", d=rng.randint(4, 6), n=rng.randint(5, 9), L0=1, form="chosen", nsteps=256,
                    m=16, levels=3, dt=0.02 / 512)
    if kind == "seq":
        op = rng.choice(["heat", "varheat", "ou", "lsde", "cme"])
        if op == "heat":
            d = rng.randint(2, 6)
            return dict(kind=kind, op=op, d=d, n=rng.randint(5, 9), L0=1, prec=rng.choice(["mixed", "pair", "fp64"]),
                        nsteps=_log_int(rng, 17, 128), dt=0.02 / 512)
        if op == "varheat":
            return dict(kind=kind, op=op, d=rng.randint(2, 3), n=rng.randint(5, 8), L0=1,
                        prec=rng.choice(["mixed", "pair", "fp64"]), nsteps=_log_int(rng, 17, 512), dt=0.1 / 2048)
        if op == "ou":
            return dict(kind=kind, op=op, d=rng.randint(2, 4), n=rng.randint(5, 7), L0=1,
                        prec=rng.choice(["mixed", "fp64"]), nsteps=_log_int(rng, 17, 512), dt=1.0 / 512)
        if op == "lsde":
            return dict(kind=kind, op=op, d=2, n=rng.randint(11, 14), L0=rng.randint(5, 6), prec="fp64",
                        nsteps=_log_int(rng, 9, 96), dt=1.0 / 3200)
        return dict(kind=kind, op=op, d=2, n=rng.randint(11, 13), L0=rng.randint(5, 6), prec="fp64",
                    nsteps=_log_int(rng, 17, 256), dt=1.0)
    if kind == "phi":
        d = rng.randint(2, 4)
        return dict(kind=kind, op="heat", d=d, n=rng.randint(4, 9 if d < 4 else 7), L0=1,
                    prec=rng.choice(["mixed", "pair", "fp64"]), batch=_log_int(rng, 1, 64),
                    forcing=rng.random() < 0.5, dt=0.05 / 1024)
    if kind == "combine":
        d = rng.randint(2, 6)
        return dict(kind=kind, op=rng.choice(["ou", "heat"]), d=d, n=rng.randint(4, 9 if d < 5 else 8), L0=1,
                    npts=_log_int(rng, 33, 65794))
    if kind == "recombine":
        d = rng.randint(2, 6)
        return dict(kind=kind, op="heat", d=d, n=rng.randint(4, 10 if d < 6 else 9), L0=1)
    d = rng.randint(2, 4)
    return dict(kind=kind, op=rng.choice(["heat", "varheat"]), d=d, n=rng.randint(4, 8 if d < 4 else 6), L0=1,
                batch=rng.randint(1, 3), dT=0.1 / 64)


# ---------------------------------------------------------------------------------------------------------------
# inputs, from the seed alone
def _modes(d, seed, decay=0.0):
    """A dominant product of sines and seven smaller ones of frequencies 1..4 (parameters of sample_initial, kind 0);
    `decay`: every mode damped by the heat equation over that time."""
    r = random.Random(seed)
    p = [8.0]
    for k in range(8):
        f = [1] * d if k == 0 else [r.randint(1, 4) for _ in range(d)]
        a = 0.5 + r.random() if k == 0 else 0.1 * r.gauss(0.0, 1.0)
        p += [a * math.exp(-decay * math.pi ** 2 * sum(q * q for q in f))] + [float(q) for q in f]
    return np.array(p)


def _initial(case, seed):
    """(kind, parameters) of sample_initial for the case's operator."""
    r = random.Random(seed)
    d = case["d"]
    if case["op"] in ("heat", "varheat"):
        return 0, _modes(d, seed)
    if case["op"] == "ou":
        return 1, np.array([1.0 + 0.2 * r.uniform(-1, 1) for _ in range(d)] + [0.5 + 0.1 * r.random() for _ in range(d)])
    if case["op"] == "lsde":
        return 4, np.array([5.0 + r.uniform(-0.5, 0.5), 5.0 + r.uniform(-0.5, 0.5), 1 / 9, 0.0, 0.0, 1 / 9])
    return 4, np.array([133.0 + r.uniform(-5, 5), 133.0 + r.uniform(-5, 5), 133.0, 0.0, 0.0, 133.0])


def _points(case, seed):
    lo, hi = BOX[case["op"]]
    return lo + (hi - lo) * np.random.RandomState(seed % (1 << 31)).rand(case["npts"], case["d"])


def _weights(seed):
    """He-scaled normals, the last layer small: a network in training."""
    r = np.random.RandomState(seed % (1 << 31))
    out = []
    for k, (cin, cout) in enumerate([(3, 16), (17, 16), (17, 16), (17, 1)]):
        sd = 0.05 if k == 3 else math.sqrt(2.0 / (cin * 5 * 3))
        out += [sd * r.randn(cout * cin * 5), 0.01 * r.randn(cout)]
    return np.concatenate(out).astype(np.float32)


def _problem(case):
    lo, hi = BOX[case["op"]]
    d = case["d"]
    kw = {}
    if case["op"] == "lsde":
        kw = dict(drift=np.array(LSDE_A), diffusion=np.array(LSDE_H), drift_scheme=B.PIT_DRIFT_CENTRAL)
    elif case["op"] == "cme":
        kw = dict(cme=CME_RATES, drift_scheme=B.PIT_DRIFT_CENTRAL)
    return B.Problem(d, case["n"], case["L0"], OPS[case["op"]], [lo] * d, [hi] * d, vamp=VAMP, **kw)


def _solve_opts(prec):
    if prec == "fp64":
        return B.solve_opts(B.PIT_PREC_FP64, rtol=1e-12, maxit=20000)
    return B.solve_opts(PRECS[prec], rtol=1e-11, maxit=4000, inner_rtol=1e-6 if prec == "mixed" else 1e-5, ir_maxit=12)


def _mgrit_opts(case):
    t1 = case["nsteps"] * case["dt"]
    if case["form"] == "plain":  # the paper's algorithm: FAS, FCF relaxation, FP64 Krylov everywhere
        fine = B.solve_opts(B.PIT_PREC_FP64, rtol=1e-11, maxit=8000)
        return B.mgrit_opts(0.0, t1, case["nsteps"], case["m"], case["levels"], tol=1e-8, maxit=64, fine=fine,
                            crs=fine, fas=True)
    fine = B.solve_opts(B.PIT_PREC_MIXED, rtol=5e-12, maxit=4000, inner_rtol=1e-6, ir_maxit=12)
    if case["levels"] == 2:
        crs = B.solve_opts(B.PIT_PREC_FP32, rtol=1e-2, maxit=4000, inner_rtol=1e-5, ir_maxit=12)
        return B.mgrit_opts(0.0, t1, case["nsteps"], case["m"], 2, tol=1e-8, maxit=64, fine=fine, crs=crs,
                            relax=B.PIT_RELAX_F, init=1)
    crs = B.solve_opts(B.PIT_PREC_MIXED, rtol=1e-6, maxit=4000, inner_rtol=1e-6, ir_maxit=12)
    return B.mgrit_opts(0.0, t1, case["nsteps"], case["m"], 3, tol=4e-8, maxit=64, fine=fine, crs=crs,
                        relax=B.PIT_RELAX_F, lanes=1, init=2)


def prepare(case, seed):
    P = _problem(case)
    kind = case["kind"]
    nb = case.get("batch", 1)
    s = {"kind": kind, "P": P, "case": case}
    new = lambda k=1: torch.empty(k * P.n_total, dtype=torch.float64, device="cuda")  # noqa: E731
    u = new(nb)
    for b in range(nb):
        ik, prm = _initial(case, seed + 1000 * b)
        P.sample_initial(ik, prm, u[b * P.n_total:(b + 1) * P.n_total])
    s["u"] = u
    if kind == "mgrit":
        s["opts"], s["out"] = _mgrit_opts(case), new()
    elif kind == "seq":
        s["opts"], s["out"] = _solve_opts(case["prec"]), new()
    elif kind == "phi":
        s["opts"], s["out"], s["f"] = _solve_opts(case["prec"]), new(nb), None
        if case["forcing"]:
            s["f"] = new(nb)
            for b in range(nb):
                P.sample_initial(0, _modes(case["d"], seed + 7 + 1000 * b), s["f"][b * P.n_total:(b + 1) * P.n_total])
    elif kind == "combine":
        s["pts"] = torch.from_numpy(_points(case, seed)).cuda()
        s["out"] = torch.empty(case["npts"], dtype=torch.float64, device="cuda")
    elif kind == "recombine":
        s["out"] = new()
    else:
        y = new(nb)
        for b in range(nb):
            P.sample_initial(0, _modes(case["d"], seed + 1000 * b, case["dT"]), y[b * P.n_total:(b + 1) * P.n_total])
        s["y"] = y
        P.net_set_params(_weights(seed))
    return s


def run(s):
    P, c = s["P"], s["case"]
    if s["kind"] == "mgrit":
        P.mgrit_solve(s["u"], s["opts"], s["out"])
        return s["out"]
    if s["kind"] == "seq":
        P.sequential_solve(s["u"], c["dt"], c["nsteps"], s["out"], s["opts"])
        return s["out"]
    if s["kind"] == "phi":
        P.phi_batch(c["dt"], s["u"], s["out"], s["opts"], f=s["f"], n_batch=c["batch"], stats=False)
        return s["out"]
    if s["kind"] == "combine":
        return P.combine(s["u"], s["pts"], s["out"])
    if s["kind"] == "recombine":
        return P.recombine(s["u"], s["out"])
    loss, grad = P.net_loss_grad(c["dT"], s["u"], s["y"], n_batch=c["batch"])
    return {"loss": loss, "grad": grad}


# ---------------------------------------------------------------------------------------------------------------
# what one pass cannot do without
def _grids(case):
    """Level multi-indices (l_i >= L0, |l| = n + d - 1 - w) and coefficients, in the canonical order."""
    d, n, L0 = case["d"], case["n"], case["L0"]
    out = []
    for w in range(d):
        total = n + d - 1 - w

        def fill(head):
            if len(head) == d - 1:
                last = total - sum(head)
                if last >= L0:
                    yield head + [last]
                return
            for v in range(L0, total - sum(head) - L0 * (d - 1 - len(head)) + 1):
                yield from fill(head + [v])

        out += [(tuple(l), (-1.0) ** w * math.comb(d - 1, w)) for l in fill([])]
    return out


def work(case):
    """Bytes: every input read and every output written once.  Flops: per backward-Euler step one application of the
    operator to the state (its residual), per evaluation point one multilinear interpolation a grid, per node and axis
    one surplus each way, per node the products of the network forward and backward."""
    gr = _grids(case)
    nodes = sum(math.prod((1 << l) - 1 for l in lev) for lev, _ in gr)
    # operator application: 2 flops a stencil entry that exists
    stencil = sum(math.prod((1 << l) - 1 for l in lev) * (2 + 4 * sum(l > 1 for l in lev)) for lev, _ in gr)
    kind, nb = case["kind"], case.get("batch", 1)
    if kind in ("mgrit", "seq"):
        return {"bytes": 16.0 * nodes, "flops": float(stencil) * case["nsteps"]}
    if kind == "phi":
        return {"bytes": (24.0 if case["forcing"] else 16.0) * nodes * nb, "flops": float(stencil) * nb}
    if kind == "combine":
        return {"bytes": 8.0 * nodes + 8.0 * case["npts"] * (case["d"] + 1),
                "flops": 2.0 * len(gr) * case["npts"] * 2 ** case["d"]}
    if kind == "recombine":
        return {"bytes": 16.0 * nodes, "flops": 6.0 * case["d"] * nodes}
    fma = 3 * 16 * 5 + 2 * 17 * 16 * 5 + 17 * 5
    return {"bytes": 16.0 * nodes * nb, "flops": 3 * 2.0 * fma * nodes * nb}


# ---------------------------------------------------------------------------------------------------------------
# the same in 64 bits with torch and numpy alone
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _axes(case, lev):
    lo, hi = BOX[case["op"]]
    h = [(hi - lo) / (1 << l) for l in lev]
    return h, [lo + np.arange(1, 1 << l) * hh for l, hh in zip(lev, h)]


def _sample(case, ik, prm, lev):
    """sample_initial on one grid, as an array of the grid's shape."""
    d = case["d"]
    lo, hi = BOX[case["op"]]
    _, xs = _axes(case, lev)
    if ik == 0:
        v = 0.0
        for k in range(int(prm[0])):
            row = prm[1 + k * (d + 1):1 + (k + 1) * (d + 1)]
            t = np.array(row[0])
            for i in range(d):
                t = np.multiply.outer(t, np.sin(np.pi * row[1 + i] * (xs[i] - lo) / (hi - lo)))
            v = v + t
        return v
    if ik == 1:
        t = np.array(1.0)
        for i in range(d):
            z = (xs[i] - prm[i]) / prm[d + i]
            t = np.multiply.outer(t, np.exp(-0.5 * z * z) / (prm[d + i] * math.sqrt(2 * math.pi)))
        return t
    C = np.asarray(prm[d:]).reshape(d, d)
    x = np.stack(np.meshgrid(*xs, indexing="ij"), -1) - np.asarray(prm[:d])
    q = np.einsum("...i,ij,...j->...", x, np.linalg.inv(C), x)
    return np.exp(-0.5 * q) / math.sqrt((2 * math.pi) ** d * np.linalg.det(C))


def _heat_power(case, lev, u, steps):
    """(I + dt L)^-steps u of the constant-coefficient heat operator, u of shape (batch, N_1, ..), by sine transforms."""
    dev = u.device
    h, _ = _axes(case, lev)
    lam = torch.zeros([1] * (len(lev) + 1), dtype=torch.float64, device=dev)
    S = []
    for i, l in enumerate(lev):
        k = torch.arange(1, 1 << l, dtype=torch.float64, device=dev)
        ev = 4.0 / h[i] ** 2 * torch.sin(k * (math.pi / 2 / (1 << l))) ** 2
        shape = [1] * (len(lev) + 1)
        shape[i + 1] = -1
        lam = lam + ev.reshape(shape)
        S.append(torch.sin(torch.outer(k, k) * (math.pi / (1 << l))))

    def transform(v):
        for i, l in enumerate(lev):
            if l > 1:
                v = torch.movedim(torch.tensordot(v, S[i], dims=([i + 1], [0])), -1, i + 1)
        return v

    scale = math.prod(2.0 / (1 << l) for l in lev if l > 1)
    return transform(transform(u) * (1.0 + case["dt"] * lam) ** (-steps)) * scale


def _coefs(case, lev):
    """Stencil of I + dt L: centre, per-axis minus and plus coefficients (arrays of the grid's shape), mixed factor."""
    d, op, dt = case["d"], case["op"], case["dt"]
    h, xs = _axes(case, lev)
    X = np.meshgrid(*xs, indexing="ij")
    diag, cm, cp = np.ones(X[0].shape), [], []
    cross = 0.0

    def drift(vp, vm, hh, central):
        if central:
            return 0.5 * (vp - vm) / hh, -0.5 * vm / hh, 0.5 * vp / hh
        return (np.maximum(vp, 0) - np.minimum(vm, 0)) / hh, -np.maximum(vm, 0) / hh, np.minimum(vp, 0) / hh

    for i in range(d):
        hh, ih2 = h[i], 1.0 / h[i] ** 2
        if op == "varheat":
            def a(Y):
                f = 1.0
                for k in range(d):
                    f = f * (np.sin(2 * np.pi * Y[k]) if k % 2 == 0 else np.cos(2 * np.pi * Y[k]))
                return 1.0 + VAMP * f
            Xm, Xp = list(X), list(X)
            Xm[i], Xp[i] = X[i] - 0.5 * hh, X[i] + 0.5 * hh
            am, ap = a(Xm), a(Xp)
            dd, dm, dp = (am + ap) * ih2, -am * ih2, -ap * ih2
        elif op == "ou":
            dd, dm, dp = drift(-(X[i] + 0.5 * hh), -(X[i] - 0.5 * hh), hh, False)
            dd, dm, dp = dd + ih2, dm - 0.5 * ih2, dp - 0.5 * ih2
        elif op == "lsde":
            v = sum(LSDE_A[i][k] * X[k] for k in range(d))
            s2 = 0.5 * LSDE_H[i][i] * ih2
            dd, dm, dp = drift(v + 0.5 * hh * LSDE_A[i][i], v - 0.5 * hh * LSDE_A[i][i], hh, True)
            dd, dm, dp = dd + 2 * s2, dm - s2, dp - s2
        else:
            y = sum(X[k] for k in range(d) if k != i)
            a0, g = CME_RATES[0] / (CME_RATES[1] + y ** CME_RATES[2]), CME_RATES[3]
            dd, dm, dp = drift(a0 - g * (X[i] + 0.5 * hh), a0 - g * (X[i] - 0.5 * hh), hh, True)
            dd = dd + (a0 + g * X[i]) * ih2
            dm = dm - 0.5 * (a0 + g * (X[i] - hh)) * ih2
            dp = dp - 0.5 * (a0 + g * (X[i] + hh)) * ih2
        diag = diag + dt * dd
        cm.append(dt * dm * np.ones_like(diag))
        cp.append(dt * dp * np.ones_like(diag))
    if op == "lsde":
        cross = -dt * 0.5 * (LSDE_H[0][1] + LSDE_H[1][0]) / (4 * h[0] * h[1])
    return diag, cm, cp, cross


def _dense_power(diag, cm, cp, u, steps):
    shape, n = diag.shape, diag.size
    idx = np.arange(n).reshape(shape)
    A = np.zeros((n, n))
    A[idx.ravel(), idx.ravel()] = diag.ravel()
    for i in range(diag.ndim):
        lo = tuple(slice(None, -1) if k == i else slice(None) for k in range(diag.ndim))
        hi = tuple(slice(1, None) if k == i else slice(None) for k in range(diag.ndim))
        A[idx[hi].ravel(), idx[lo].ravel()] = cm[i][hi].ravel()
        A[idx[lo].ravel(), idx[hi].ravel()] = cp[i][lo].ravel()
    M = torch.linalg.inv(torch.from_numpy(A).to(_dev()))
    v = torch.from_numpy(np.ascontiguousarray(u).reshape(-1)).to(M.device)
    while steps:
        if steps & 1:
            v = M @ v
        steps >>= 1
        if steps:
            M = M @ M
    return v.cpu().numpy()


def _block_power(diag, cm, cp, cross, u, steps):
    """Two axes: block-tridiagonal elimination along the longer one."""
    if diag.shape[0] < diag.shape[1]:
        r = _block_power(diag.T, [cm[1].T, cm[0].T], [cp[1].T, cp[0].T], cross, u.T, steps)
        return r.reshape(diag.shape[1], diag.shape[0]).T.reshape(-1)
    K, m = diag.shape
    off = lambda v, k: np.diag(v, k)  # noqa: E731
    up, dn = cross * np.ones(m - 1), -cross * np.ones(m - 1)
    # c (p_{++} - p_{+-} - p_{-+} + p_{--}): row a + 1 gets +c right, -c left; row a - 1 the opposite
    D = [np.diag(diag[a]) + off(cp[1][a][:-1], 1) + off(cm[1][a][1:], -1) for a in range(K)]
    L = [np.diag(cm[0][a]) + off(-up, 1) + off(-dn, -1) for a in range(K)]
    U = [np.diag(cp[0][a]) + off(up, 1) + off(dn, -1) for a in range(K)]
    G, W, V = [], [None], []
    S = D[0]
    for a in range(K):
        if a:
            W.append(L[a] @ G[a - 1])
            S = D[a] - W[a] @ U[a - 1]
        G.append(np.linalg.inv(S))
        V.append(G[a] @ U[a])
    Gs = np.stack(G)
    x = np.array(u, dtype=np.float64)
    for _ in range(steps):
        y = x
        for a in range(1, K):
            y[a] -= W[a] @ y[a - 1]
        x = np.einsum("aij,aj->ai", Gs, y)
        for a in range(K - 2, -1, -1):
            x[a] -= V[a] @ x[a + 1]
    return x.reshape(-1)


def _hier(v, sign):
    """Hierarchical surpluses of a grid's nodal values along every axis (sign -1), or back (+1), in place."""
    for ax in range(v.ndim):
        w = np.moveaxis(v, ax, 0)
        N = w.shape[0]
        lev = (N + 1).bit_length() - 1
        for t in range(lev) if sign < 0 else range(lev - 1, -1, -1):
            st = 1 << t
            J = np.arange(st, N + 1, 2 * st)
            p = np.zeros((len(J) + 1,) + w.shape[1:])
            p[1:-1] = w[J[:-1] + st - 1]
            w[J - 1] += sign * 0.5 * (p[:-1] + p[1:])
    return v


def _increments(lev):
    """(increment, slices of its nodes) of a grid."""
    for lam in itertools.product(*[range(1, l + 1) for l in lev]):
        yield lam, tuple(slice((1 << (l - k)) - 1, None, 2 << (l - k)) for l, k in zip(lev, lam))


def _exact_recombine(case, seed, gr):
    ik, prm = _initial(case, seed)
    acc = {}
    for lev, c in gr:
        v = _hier(np.array(_sample(case, ik, prm, lev)), -1.0)
        for lam, at in _increments(lev):
            acc[lam] = acc[lam] + c * v[at] if lam in acc else c * v[at]
    out = []
    for lev, _ in gr:
        v = np.empty([(1 << l) - 1 for l in lev])
        for lam, at in _increments(lev):
            v[at] = acc[lam]
        out.append(_hier(v, 1.0).reshape(-1))
    return np.concatenate(out)


def _exact_combine(case, seed, gr):
    dev, d = _dev(), case["d"]
    lo, hi = BOX[case["op"]]
    ik, prm = _initial(case, seed)
    x = torch.from_numpy((_points(case, seed) - lo) / (hi - lo)).to(dev)
    total = torch.zeros(case["npts"], dtype=torch.float64, device=dev)
    for lev, c in gr:
        u = torch.from_numpy(np.ascontiguousarray(np.pad(_sample(case, ik, prm, lev), 1))).to(dev)
        cells, ts = [], []
        for i, l in enumerate(lev):
            s = x[:, i] * (1 << l)
            k = torch.clamp(s.floor().long(), 0, (1 << l) - 1)
            cells.append(k)
            ts.append(s - k)
        for corner in itertools.product((0, 1), repeat=d):
            w = torch.full_like(total, c)
            flat = torch.zeros_like(cells[0])
            for i in range(d):
                w = w * (ts[i] if corner[i] else 1.0 - ts[i])
                flat = flat * u.shape[i] + cells[i] + corner[i]
            total += w * u.reshape(-1)[flat]
    return total.cpu().numpy()


def _exact_netgrad(case, seed, gr):
    dev, d = _dev(), case["d"]
    w = torch.from_numpy(_weights(seed)).to(torch.bfloat16).double().to(dev).requires_grad_(True)
    layers, at = [], 0
    for cin, cout in [(3, 16), (17, 16), (17, 16), (17, 1)]:
        layers.append((w[at:at + cout * cin * 5].reshape(cout, cin, 5), w[at + cout * cin * 5:at + cout * cin * 5 + cout]))
        at += cout * cin * 5 + cout
    total = 0.0
    for b in range(case["batch"]):
        ik, pu = _initial(case, seed + 1000 * b)
        py = _modes(d, seed + 1000 * b, case["dT"])
        for lev, _ in gr:
            h, xs = _axes(case, lev)
            X = np.meshgrid(*xs, indexing="ij")
            a = np.ones(X[0].shape)
            if case["op"] == "varheat":
                for k in range(d):
                    a = a * (np.sin(2 * np.pi * X[k]) if k % 2 == 0 else np.cos(2 * np.pi * X[k]))
                a = 1.0 + VAMP * a
            u = torch.from_numpy(np.array(_sample(case, ik, pu, lev))).to(dev)
            y = torch.from_numpy(np.array(_sample(case, 0, py, lev))).to(dev)
            sig = torch.sqrt((u * u).mean())
            z = torch.stack([u / sig, torch.from_numpy(a).to(dev)])
            si = [1.0 / (1.0 + 4.0 * case["dT"] / hh ** 2) for hh in h]
            one = torch.ones_like(u)
            for k, (W, bias) in enumerate(layers):
                full = torch.cat([z, one[None]])
                taps = []
                for t in range(5):
                    acc = 0.0
                    for i in range(d):
                        N = u.shape[i]
                        src = full if t != 2 else full
                        p = torch.nn.functional.pad(torch.movedim(src, i + 1, -1), (2, 2))[..., t:t + N]
                        p = torch.movedim(p, -1, i + 1)
                        acc = acc + torch.cat([p[:-1], p[-1:] * si[i]])
                    taps.append(acc)
                z = torch.einsum("oct,tc...->o...", W, torch.stack(taps)) + bias.reshape([-1] + [1] * d)
                if k < 3:
                    z = torch.relu(z)
            total = total + ((u + sig * z[0] - y) ** 2).sum() / (y * y).sum()
    total.backward()
    return {"loss": total.item(), "grad": w.grad.cpu().numpy()}


def exact(case, seed):
    kind, gr = case["kind"], _grids(case)
    if kind == "recombine":
        return torch.from_numpy(_exact_recombine(case, seed, gr))
    if kind == "combine":
        if case["npts"] * len(gr) * 2 ** case["d"] > 4e9:
            return None
        return torch.from_numpy(_exact_combine(case, seed, gr))
    if kind == "netgrad":
        return _exact_netgrad(case, seed, gr)
    nb, steps = case.get("batch", 1), case.get("nsteps", 1)
    out = []
    if case["op"] == "heat":
        inits = [_initial(case, seed + 1000 * b) for b in range(nb)]
        forces = [_modes(case["d"], seed + 7 + 1000 * b) for b in range(nb)] if case.get("forcing") else None
        for lev, _ in gr:
            u = np.stack([_sample(case, ik, prm, lev) for ik, prm in inits])
            if forces:
                u = u + case["dt"] * np.stack([_sample(case, 0, f, lev) for f in forces])
            r = _heat_power(case, lev, torch.from_numpy(u).to(_dev()), steps)
            out.append(r.reshape(nb, -1).cpu())
        return torch.cat(out, 1).reshape(-1).contiguous()
    ik, prm = _initial(case, seed)
    for lev, _ in gr:
        diag, cm, cp, cross = _coefs(case, lev)
        u = np.array(_sample(case, ik, prm, lev))
        if case["op"] in ("lsde", "cme"):
            out.append(_block_power(diag, cm, cp, cross, u, steps))
        else:
            out.append(_dense_power(diag, cm, cp, u, steps))
    return torch.from_numpy(np.concatenate(out))
