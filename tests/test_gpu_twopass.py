"""The library's own kernel choice of a BF16x3 plan against the FP64 oracle,
where its rule takes the two-pass launch (the x1 and x2 products of a Tucker
operator as dependent passes) and the sizes at which that launch, and the 3D
stencil on whole rows, can go wrong: tiles that span slabs, sides of one tile
and one more, columns split over narrow tiles, rows at and beyond the
stencil's limit, narrow and wide supports, two plans on two streams, and a
field that holds an infinity.

Tolerance: 1e-5 max relative error against FP64, the bound of the split
products (24 bits an operand; a step forms a few hundred products of either
sign per value)."""
import numpy as np
import pytest

import oracle
import workloads as wl
from oracle import schemes

pytestmark = pytest.mark.gpu

TOL = 1e-5
PARAMS = {wl.SCHNAKENBERG: (200.0, 0.1, 0.9), wl.FHN: (0.05, 2.0, -0.03),
          wl.BRUSSELATOR: (1.0, 3.0)}


@pytest.fixture(scope="module")
def adr():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2307_10684_gb300 import build
    build.build()
    import paper_2307_10684_gb300 as adr
    return adr


def problem(n, model, nsteps=4, scheme=wl.ETD2RKDS, state=wl.STATE_AUTO, tau=2e-3):
    d = len(n)
    return wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(0.02, 0.1),
                      adv=((0.2, -0.1, 0.3)[:d], (-0.2, 0.1, 0.05)[:d]), model=model,
                      params=PARAMS[model], tau=tau, nsteps=nsteps, precision=wl.BF16X3, seed=91,
                      scheme=scheme, state=state)


def inputs(p):
    u0, v0 = wl.initial_data(p, kind="uniform")
    return wl.round_to(u0, wl.FP32), wl.round_to(v0, wl.FP32)


def reference(p, u0, v0):
    plan = schemes.make_plan(p)
    if p.scheme == wl.LAWSON2B:
        for _ in range(p.nsteps):
            u0, v0 = schemes.lawson2b_step(plan, u0, v0)
        return u0, v0
    return schemes.etd2rkds_solve(plan, u0, v0, p.nsteps)


def run(adr, p, u0, v0, kernel=-1):
    import torch
    u = torch.tensor(u0, dtype=torch.float32, device="cuda")
    v = torch.tensor(v0, dtype=torch.float32, device="cuda")
    with adr.Plan(p, kernel=kernel) as plan:
        plan.step(u, v, p.nsteps)
        assert plan.stats()["device_error"] == 0
    return u.double().cpu().numpy(), v.double().cpu().numpy()


@pytest.mark.parametrize("n,model", [
    ((128, 128), wl.FHN), ((136, 8), wl.BRUSSELATOR), ((8, 392), wl.FHN), ((256, 264), wl.SCHNAKENBERG),
    ((648, 40), wl.FHN), ((176, 136), wl.BRUSSELATOR), ((264, 200), wl.FHN),
    ((1032, 64), wl.SCHNAKENBERG), ((40, 16, 200), wl.FHN), ((8, 8, 8), wl.SCHNAKENBERG),
    ((160, 24, 40), wl.BRUSSELATOR), ((72, 264, 16), wl.FHN), ((192, 8, 16), wl.FHN),
    ((200, 16, 24), wl.SCHNAKENBERG), ((264, 8, 16), wl.BRUSSELATOR)])
@pytest.mark.parametrize("state", [wl.STATE_PLAIN, wl.STATE_COMPENSATED])
def test_matches_oracle(adr, n, model, state):
    p = problem(n, model, state=state)
    u0, v0 = inputs(p)
    U, V = run(adr, p, u0, v0)
    assert oracle.max_rel_err(U, V, *reference(p, u0, v0)) <= TOL


@pytest.mark.parametrize("n", [(72, 136), (24, 40, 16), (264, 8, 24)])
def test_lawson_matches_oracle(adr, n):
    p = problem(n, wl.FHN, scheme=wl.LAWSON2B)
    u0, v0 = inputs(p)
    U, V = run(adr, p, u0, v0)
    assert oracle.max_rel_err(U, V, *reference(p, u0, v0)) <= TOL


@pytest.mark.parametrize("L,n", [(100.0, (1024, 384)), (10.0, (1024, 384)), (20.0, (384, 640))])
def test_supports_of_long_rows(adr, L, n):
    """FHN on a short and a long domain: wide supports (the two-pass launch,
    column tiles contracting over their own group's range) and narrow ones
    (the intermediate in TMEM)."""
    p = wl.fhn_1024(precision=wl.BF16X3, nsteps=3).replace(n=n, hi=(L, L))
    u0, v0 = wl.initial_data(p)
    u0, v0 = wl.round_to(u0, wl.FP32), wl.round_to(v0, wl.FP32)
    U, V = run(adr, p, u0, v0)
    assert oracle.max_rel_err(U, V, *reference(p, u0, v0)) <= TOL


def test_an_infinity_stays_where_its_products_reach(adr):
    """Supports bound what a non-finite point reaches in one step; the points
    beyond keep the values they have without it, bit for bit."""
    p = wl.fhn_1024(precision=wl.BF16X3, nsteps=1).replace(n=(1024, 512), hi=(30.0, 30.0))
    u0, v0 = wl.initial_data(p)
    u0, v0 = wl.round_to(u0, wl.FP32), wl.round_to(v0, wl.FP32)
    U, V = run(adr, p, u0, v0)
    u1 = u0.copy()
    u1[7, 5] = np.inf
    Ui, Vi = run(adr, p, u1, v0)
    assert not np.isfinite(Ui[7, 5])
    assert np.array_equal(Ui[:, 960:], U[:, 960:]) and np.array_equal(Vi[:, 960:], V[:, 960:])


def test_two_plans_on_two_streams(adr):
    """Units are claimed from a counter and wait for units claimed earlier:
    two plans interleaved on two streams end, with the results they have
    alone, bit for bit."""
    import torch
    ps = [problem((392, 264), wl.FHN, nsteps=40), problem((96, 72, 64), wl.BRUSSELATOR, nsteps=40)]
    init = [inputs(p) for p in ps]
    alone = [run(adr, p, *i) for p, i in zip(ps, init)]
    streams = [torch.cuda.Stream() for _ in ps]
    plans, fields = [], []
    for p, (u0, v0), s in zip(ps, init, streams):
        with torch.cuda.stream(s):
            plans.append(adr.Plan(p, stream=s))
            fields.append([torch.tensor(x, dtype=torch.float32, device="cuda") for x in (u0, v0)])
    torch.cuda.synchronize()
    for _ in range(20):
        for pl, (u, v) in zip(plans, fields):
            pl.step(u, v, 2)
    torch.cuda.synchronize()
    for pl, (u, v), (U, V) in zip(plans, fields, alone):
        assert pl.stats()["device_error"] == 0
        assert np.array_equal(u.double().cpu().numpy(), U) and np.array_equal(v.double().cpu().numpy(), V)
        pl.close()
