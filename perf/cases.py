"""The calls whose speed is watched: what a program has the ETD2RKds stepper do.

A case names one use of the public binding: a solve from given initial data, a
server's tick, a batch, a monitored run, a general plan.  Grids, coefficients,
horizons and data follow the repository's own configurations (the Schnakenberg
64^2, FitzHugh-Nagumo 1024^2 and Brusselator 256^3 solves, the mixed batch, the
serving stream, the Lawson2b and general-plan options).  The products run in
split BF16 on the tensor cores unless a case says FP32 or FP64, which are the
precisions for grids whose sides are no multiples of eight and for FP64 results.

exact() repeats a case in 64 bits with plain torch operations.
"""
import math
import types

import torch

import paper_2307_10684_gb300 as adr

PREC = {"fp64": adr.FP64, "fp32": adr.FP32, "bf16x3": adr.BF16X3}
MODEL = {"schnakenberg": adr.SCHNAKENBERG, "fhn": adr.FHN, "brusselator": adr.BRUSSELATOR,
         "fhn_rho": adr.FHN_RHO}
BATCH_SIDES = (64, 96, 128, 192, 256, 384, 512)


def listed():
    return [
        # an interactive program that looks at the state every few steps: all launch latency
        dict(name="step4_128x96", kind="step", model="brusselator", precision="bf16x3",
             state="plain", scheme="etd2rkds", n1=128, n2=96, n3=0, steps=4),
        # the small reference solve in FP64 (64^2, 200 steps)
        dict(name="solve_schnakenberg_64_fp64", kind="solve", model="schnakenberg",
             precision="fp64", state="plain", scheme="etd2rkds", n1=64, n2=64, n3=0, steps=200),
        # the benchmark's 2D solve: FitzHugh-Nagumo with advection, 1024^2
        dict(name="solve_fhn_1024", kind="solve", model="fhn", precision="bf16x3", state="plain",
             scheme="etd2rkds", n1=1024, n2=1024, n3=0, steps=96),
        # the benchmark's 3D solve: advective Brusselator, 256^3, the largest work
        dict(name="solve_brusselator_256", kind="solve", model="brusselator", precision="bf16x3",
             state="plain", scheme="etd2rkds", n1=256, n2=256, n3=256, steps=32),
        # a batch of independent 2D solves of mixed, non-square sides
        dict(name="batch_32_mixed", kind="batch", precision="bf16x3", state="plain", count=32,
             pick=4, steps=32),
        # a server's tick on one 2D solve: 32 steps of a compensated state
        dict(name="tick_schnakenberg_512", kind="step", model="schnakenberg", precision="bf16x3",
             state="compensated", scheme="etd2rkds", n1=512, n2=512, n3=0, steps=32),
        # a server's tick on one 3D solve
        dict(name="tick_brusselator_160", kind="step", model="brusselator", precision="bf16x3",
             state="compensated", scheme="etd2rkds", n1=160, n2=160, n3=160, steps=32),
        # plain FP32 on a 3D grid whose sides are no multiples of eight
        dict(name="solve_fhn_rho_3d_fp32", kind="solve", model="fhn_rho", precision="fp32",
             state="plain", scheme="etd2rkds", n1=65, n2=64, n3=63, steps=32),
        # a monitored run: indicators of every step, read back every 32 steps
        dict(name="run_brusselator_200", kind="run", model="brusselator", precision="bf16x3",
             state="plain", scheme="etd2rkds", n1=200, n2=200, n3=0, steps=64),
        # the second scheme, on a non-square grid
        dict(name="solve_lawson2b_768x512", kind="solve", model="fhn", precision="bf16x3",
             state="plain", scheme="lawson2b", n1=768, n2=512, n3=0, steps=32),
        # three components, dense matrices, polynomial reactions, FP64
        dict(name="general_m3_130x72_fp64", kind="general", precision="fp64", comps=3, n1=130,
             n2=72, n3=0, steps=16),
        # host buffers in, host buffers out, a large non-square 2D grid
        dict(name="host_solve_fhn_2048x1536", kind="host", model="fhn", precision="bf16x3",
             state="plain", scheme="etd2rkds", n1=2048, n2=1536, n3=0, steps=64),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("solve2", "solve2", "solve3", "tick2", "tick3", "simt", "simt", "run",
                       "lawson", "general", "host", "batch", "step"))
    model = rng.choice(("schnakenberg", "fhn", "brusselator"))
    side8 = lambda lo, hi: 8 * max(1, round(_log(rng, lo, hi) / 8))  # noqa: E731
    c = dict(kind="solve", model=model, precision="bf16x3", state="plain", scheme="etd2rkds",
             n1=side8(64, 2048), n2=side8(64, 2048), n3=0, steps=rng.randint(33, 100))
    if kind == "solve3":
        c.update(n1=side8(32, 256), n2=side8(32, 256), n3=side8(32, 256), steps=rng.randint(8, 32))
    elif kind == "tick2":
        c.update(kind="step", state="compensated", steps=32, n1=side8(128, 1024),
                 n2=side8(128, 1024))
    elif kind == "tick3":
        c.update(kind="step", state="compensated", steps=32, n1=side8(64, 192), n2=side8(64, 192),
                 n3=side8(64, 192))
    elif kind == "simt":
        three = rng.random() < 0.5
        c.update(precision=rng.choice(("fp32", "fp64")), steps=rng.randint(8, 64))
        lo, hi = (20, 80) if three else (40, 320)
        c.update(n1=round(_log(rng, lo, hi)), n2=round(_log(rng, lo, hi)),
                 n3=round(_log(rng, lo, hi)) if three else 0)
        if rng.random() < 0.3:
            c.update(model="fhn_rho")
    elif kind == "run":
        c.update(kind="run", model="brusselator", n1=side8(64, 512), n2=side8(64, 512),
                 steps=rng.randint(32, 128))
    elif kind == "lawson":
        c.update(scheme="lawson2b", model="fhn", n1=side8(64, 1024), n2=side8(64, 1024),
                 steps=rng.randint(16, 64))
    elif kind == "general":
        three = rng.random() < 0.4
        lo, hi = (8, 40) if three else (24, 200)
        c = dict(kind="general", precision=rng.choice(("fp32", "fp64")), comps=rng.randint(1, 4),
                 n1=round(_log(rng, lo, hi)), n2=round(_log(rng, lo, hi)),
                 n3=round(_log(rng, lo, hi)) if three else 0, steps=rng.randint(6, 20))
    elif kind == "host":
        c.update(kind="host", model="fhn", n1=side8(256, 2048), n2=side8(256, 2048),
                 steps=rng.randint(32, 64))
    elif kind == "batch":
        c = dict(kind="batch", precision="bf16x3", state=rng.choice(("plain", "compensated")),
                 count=rng.randint(8, 32), pick=rng.randint(10, 10000), steps=rng.randint(16, 40))
    elif kind == "step":
        c.update(kind="step", n1=side8(64, 512), n2=side8(64, 512), steps=rng.randint(1, 16))
    # no more work than the listed cases have, by the rate that the precision runs at
    most = {"fp64": 4e9, "fp32": 1e11, "bf16x3": 3e12}[c["precision"]]
    c["steps"] = max(1, min(c["steps"], int(c["steps"] * most / work(c)["flops"])))
    return c


# ------------------------------------------------------------------ problems
def _problem(c):
    """One solve's problem: the coefficients of the repository's base configurations."""
    n = (c["n1"], c["n2"]) + ((c["n3"],) if c["n3"] else ())
    d = len(n)
    model = c["model"]
    vel, length, tau = 0.0, 1.0, 1e-2
    if model == "schnakenberg":
        diff, params = (1.0, 10.0), (1000.0, 0.1, 0.9)
        # the 64^2 reference solve's step; served and batched grids take a quarter of it
        tau = 5e-4 if c["precision"] == "fp64" else 1.25e-4
    elif model == "fhn":
        diff, params, vel, length = (1.0, 20.0), (0.05, 2.0, -0.03), 0.5, 100.0
    elif model == "brusselator":
        diff, params, vel = (0.02, 0.1), (1.0, 3.0), -0.5
    else:
        diff, params, length = (1.0, 42.1887), (24.649, 11.0, 0.1), math.pi
        tau = 5e-4
    # cell Peclet number below 1
    vmax = 0.9 * 2.0 * min(diff) * (min(n) - 1) / length
    vel = max(-vmax, min(vmax, vel))
    return types.SimpleNamespace(
        d=d, n=n, lo=(0.0,) * d, hi=(length,) * d, diff=diff, adv=((vel,) * d,) * 2,
        model=MODEL[model], params=params, tau=tau, precision=PREC[c["precision"]],
        scheme=adr.LAWSON2B if c.get("scheme") == "lawson2b" else adr.ETD2RKDS,
        state=adr.STATE_COMPENSATED if c["state"] == "compensated" else adr.STATE_PLAIN)


def _batch_problems(c):
    """Mixed batch: sides from BATCH_SIDES, half Schnakenberg, half FitzHugh-Nagumo."""
    gen = torch.Generator().manual_seed(c["pick"])
    out = []
    for q in torch.rand(c["count"], 5, generator=gen).tolist():
        n = tuple(BATCH_SIDES[int(x * len(BATCH_SIDES))] for x in q[:2])
        one = dict(c, model="schnakenberg" if q[2] < 0.5 else "fhn", n1=n[0], n2=n[1], n3=0)
        p = _problem(one)
        p.diff = (1.0, 5.0 + 35.0 * q[3])
        if q[2] < 0.5:
            gamma = 100.0 + 1900.0 * q[4]
            p.params = (gamma, 0.1, 0.9)
            p.tau = min(max(1.25e-4 * (1000.0 / gamma), 6.25e-5), 1.25e-3)
        out.append(p)
    return out


def _data(p, kind, gen):
    """Initial data: the equilibrium with a small perturbation (a wave for the monitored run)."""
    dt = torch.float64 if p.precision == adr.FP64 else torch.float32
    shape = tuple(reversed(p.n))
    if p.model == adr.FHN:
        f = [0.05 * torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
             for _ in range(2)]
    else:
        a, b = p.params[-2:]
        base = {adr.SCHNAKENBERG: (a + b, b / (a + b) ** 2), adr.BRUSSELATOR: (a, b / a),
                adr.FHN_RHO: (0.0, 0.0)}[p.model]
        f = [x + 0.01 * (2 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) - 1)
             for x in base]
        if kind == "run":  # u0 = a + sin(2 pi x1) sin(2 pi x2), as in the paper's Brusselator example
            s = torch.ones(shape, device="cuda", dtype=torch.float64)
            for mu, n in enumerate(p.n):
                x = torch.sin(2 * math.pi * torch.linspace(0, 1, n, device="cuda", dtype=torch.float64))
                s = s * x.reshape([-1 if ax == p.d - 1 - mu else 1 for ax in range(p.d)])
            f[0] = f[0] + s
    return [x.to(dt).contiguous() for x in f]


def _general(c, seed):
    """Dense directional matrices (negative definite part plus a skew part), each component
    driven by the next one and damped by its own square; data around 0.5."""
    n = (c["n1"], c["n2"]) + ((c["n3"],) if c["n3"] else ())
    m = c["comps"]
    gen = torch.Generator().manual_seed(seed)
    A = []
    for _ in range(m):
        row = []
        for k in n:
            B = torch.randn(k, k, generator=gen, dtype=torch.float64)
            row.append(3.0 * (-(B @ B.T / k + torch.eye(k, dtype=torch.float64))
                              + 0.3 * (B - B.T) / math.sqrt(k)))
        A.append(row)
    terms = []
    for i in range(m):
        e, e2 = [0] * m, [0] * m
        e[(i + 1) % m] += 1
        e2[i] = 2
        terms += [(i, tuple(e), 0.5), (i, tuple(e2), -0.3)]
    terms.append((0, (0,) * m, 0.3))
    shape = tuple(reversed(n))
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    U = [(0.5 + 0.1 * torch.randn(shape, generator=gen, dtype=torch.float64)).to(dt)
         for _ in range(m)]
    return A, terms, U


GENERAL_TAU = 1e-2


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    c, s = case, types.SimpleNamespace(case=case)
    if c["kind"] == "general":
        A, terms, U = _general(c, seed)
        s.plan = adr.GeneralPlan([[a.numpy() for a in row] for row in A], terms, GENERAL_TAU,
                                 precision=PREC[c["precision"]])
        s.u = [x.cuda() for x in U]
        return s
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if c["kind"] == "batch":
        problems = _batch_problems(c)
        fields = [_data(p, c["kind"], gen) for p in problems]
        s.u, s.v = [f[0] for f in fields], [f[1] for f in fields]
        s.plans = [adr.Plan(p) for p in problems]
        s.batch = adr.Batch(s.plans)
        return s
    p = _problem(c)
    s.u, s.v = _data(p, c["kind"], gen)
    s.plan = adr.Plan(p)
    if c["kind"] == "run":
        s.plan.set_indicators(True)
        s.t_end = c["steps"] * p.tau
    elif c["kind"] == "solve":
        s.u0, s.v0 = s.u, s.v
        s.u, s.v = torch.empty_like(s.u0), torch.empty_like(s.v0)
    elif c["kind"] == "host":
        s.u0, s.v0 = s.u.cpu().pin_memory(), s.v.cpu().pin_memory()
        s.u, s.v = torch.empty_like(s.u0).pin_memory(), torch.empty_like(s.v0).pin_memory()
    return s


def run(state):
    s, c = state, state.case
    kind = c["kind"]
    if kind == "general":
        s.plan.step(s.u, c["steps"])
        return s.u
    if kind == "batch":
        s.batch.step(s.u, s.v, c["steps"])
        return [s.u, s.v]
    if kind == "run":
        steps, ind = s.plan.run(s.u, s.v, s.t_end)
        return [s.u, s.v, steps, ind]
    if kind == "step":
        s.plan.step(s.u, s.v, c["steps"])
    else:
        s.plan.solve(s.u0, s.v0, s.u, s.v, c["steps"])
    return [s.u, s.v]


# ------------------------------------------------------------------ work
def _work_of(n, comps, steps, esize):
    """The state read and written once; per step and component two Tucker operators (a dense
    n_mu x n_mu matrix along every direction) and the directional sum of the right-hand side."""
    N = math.prod(n)
    flops = steps * comps * N * (4.0 * sum(n) + 12.0 * len(n))
    return 2.0 * comps * N * esize, flops


def work(case):
    c = case
    esize = 8 if c["precision"] == "fp64" else 4
    if c["kind"] == "batch":
        parts = [_work_of(p.n, 2, c["steps"], esize) for p in _batch_problems(c)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n = (c["n1"], c["n2"]) + ((c["n3"],) if c["n3"] else ())
    b, f = _work_of(n, c.get("comps", 2), c["steps"], esize)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64 bits
def _fd(n, lo, hi, delta, alpha):
    """delta d2/dx2 - alpha d/dx on n vertices, Neumann rows by a mirrored ghost value."""
    h = (hi - lo) / (n - 1)
    A = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    i = torch.arange(n, device="cuda")
    A[i, i] = -2 * delta / h ** 2
    A[i[1:], i[:-1]] = delta / h ** 2 + alpha / (2 * h)
    A[i[:-1], i[1:]] = delta / h ** 2 - alpha / (2 * h)
    A[0, 1] = A[n - 1, n - 2] = 2 * delta / h ** 2
    return A


def _phi(X):
    """e^X, phi_1(X), phi_2(X): Taylor on X / 2^s, then s doublings."""
    n = X.shape[0]
    one = torch.eye(n, dtype=X.dtype, device=X.device)
    norm = float(X.abs().sum(0).max())
    s = max(0, math.ceil(math.log2(norm / 0.5))) if norm > 0 else 0
    Y = X / 2.0 ** s
    p2 = one / math.factorial(17)
    for k in range(16, 1, -1):
        p2 = Y @ p2 + one / math.factorial(k)
    p1 = Y @ p2 + one
    E = Y @ p1 + one
    for _ in range(s):
        p2 = (p1 @ p1 + 2 * p2) / 4
        p1 = (E @ p1 + p1) / 2
        E = E @ E
    return E, p1, p2


def _mode(X, M, axis):
    """X x_mu M along tensor axis `axis`."""
    return torch.movedim(torch.tensordot(M, X, dims=([1], [axis])), 0, axis)


def _tucker(X, Ms):
    for mu, M in enumerate(Ms):
        X = _mode(X, M, X.dim() - 1 - mu)
    return X


def _react(p):
    q = p.params
    if p.model == adr.SCHNAKENBERG:
        return lambda u, v: (q[0] * (q[1] - u + u * u * v), q[0] * (q[2] - u * u * v))
    if p.model == adr.FHN:
        return lambda u, v: (u - u ** 3 - v, q[0] * (u - q[1] * v - q[2]))
    if p.model == adr.BRUSSELATOR:
        return lambda u, v: (q[0] - (q[1] + 1) * u + u * u * v, q[1] * u - u * u * v)
    return lambda u, v: (q[0] * (u - u ** 3 - v), q[0] * q[1] * (u - q[2] * v))


def _etd(U, A, phis, G, tau, d, steps):
    """`steps` steps of Eq. 11 for the components U; returns the last two states."""
    prev = U
    for _ in range(steps):
        prev = U
        g = G(*U)
        W = [sum(_mode(x, A[c][mu], d - 1 - mu) for mu in range(d)) + g[c]
             for c, x in enumerate(U)]
        U2 = [x + tau * _tucker(w, [f[1] for f in phis[c]]) for c, (x, w) in enumerate(zip(U, W))]
        g2 = G(*U2)
        U = [x + 2 ** (d - 1) * tau * _tucker(g2[c] - g[c], [f[2] for f in phis[c]])
             for c, x in enumerate(U2)]
    return prev, U


def _lawson(U, phis, G, tau, steps):
    """`steps` steps of Eq. 7."""
    for _ in range(steps):
        g = G(*U)
        E = [[f[0] for f in row] for row in phis]
        U2 = [_tucker(x + tau * g[c], E[c]) for c, x in enumerate(U)]
        g2 = G(*U2)
        U = [_tucker(x + tau / 2 * g[c], E[c]) + tau / 2 * g2[c] for c, x in enumerate(U)]
    return U


def _solve64(p, fields, steps):
    seen, A, phis = {}, [], []
    for c in range(2):
        A.append([])
        phis.append([])
        for mu in range(p.d):
            key = (p.n[mu], p.lo[mu], p.hi[mu], p.diff[c], p.adv[c][mu])
            if key not in seen:
                M = _fd(*key)
                seen[key] = (M, _phi(p.tau * M))
            A[c].append(seen[key][0])
            phis[c].append(seen[key][1])
    U = [x.double() for x in fields]
    if p.scheme == adr.LAWSON2B:
        return None, _lawson(U, phis, _react(p), p.tau, steps)
    return _etd(U, A, phis, _react(p), p.tau, p.d, steps)


def _indicators(p, prev, U):
    """Trapezoid-weighted means and Frobenius norms of the last increment."""
    w = torch.ones((), dtype=torch.float64, device="cuda")
    for mu, n in enumerate(p.n):
        t = torch.ones(n, dtype=torch.float64, device="cuda")
        t[0] = t[-1] = 0.5
        w = w * (t / (n - 1)).reshape([-1 if ax == p.d - 1 - mu else 1 for ax in range(p.d)])
    return ([float((w * x).sum()) for x in U]
            + [float((x - y).norm()) for x, y in zip(U, prev)])


def exact(case, seed):
    c = case
    if c["kind"] == "general":
        A, terms, U = _general(c, seed)
        A = [[a.cuda() for a in row] for row in A]
        phis = [[_phi(GENERAL_TAU * a) for a in row] for row in A]

        def G(*u):
            out = [torch.zeros_like(x) for x in u]
            for i, pw, coef in terms:
                t = torch.full_like(u[0], coef)
                for x, e in zip(u, pw):
                    t = t * x ** e
                out[i] = out[i] + t
            return out

        return _etd([x.cuda().double() for x in U], A, phis, G, GENERAL_TAU, len(A[0]),
                    c["steps"])[1]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if c["kind"] == "batch":
        problems = _batch_problems(c)
        fields = [_data(p, c["kind"], gen) for p in problems]
        out = [_solve64(p, f, c["steps"])[1] for p, f in zip(problems, fields)]
        return [[x[0] for x in out], [x[1] for x in out]]
    p = _problem(c)
    prev, U = _solve64(p, _data(p, c["kind"], gen), c["steps"])
    if c["kind"] == "run":
        return [U[0], U[1], c["steps"], _indicators(p, prev, U)]
    return U
