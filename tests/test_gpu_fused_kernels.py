"""The fused launch that keeps the intermediate in TMEM, with the kernel asked
for by number (the library's own choice takes the two-pass launch on many of
these grids): against the FP64 oracle over ragged grids, x2 ranges of several
256-column groups, wide supports, both schemes, the compensated state,
indicators and a grouped batch of uneven chunk counts.

Tolerance: 1e-5 max relative error against FP64, the bound of the split
products; where two launches compute the same products in another association,
1e-6.  Indicators as in the tests of the library's own choice: means within
1e-6, increments within 1e-3 and the states' rounding."""
import numpy as np
import pytest

import oracle
import workloads as wl
from oracle import metrics, schemes

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


def problem(n, model, nsteps=6, scheme=wl.ETD2RKDS, state=wl.STATE_PLAIN, diff=None, tau=2e-3,
            seed=151):
    d = len(n)
    return wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d,
                      diff=diff or ((0.05, 0.3) if d == 2 else (0.02, 0.1)),
                      adv=((0.2, -0.1, 0.3)[:d], (-0.2, 0.1, 0.05)[:d]), model=model,
                      params=PARAMS[model], tau=tau, nsteps=nsteps, precision=wl.BF16X3,
                      seed=seed, scheme=scheme, state=state)


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


def run(adr, p, u0, v0, kernel):
    import torch
    u = torch.tensor(u0, dtype=torch.float32, device="cuda")
    v = torch.tensor(v0, dtype=torch.float32, device="cuda")
    with adr.Plan(p, kernel=kernel) as plan:
        plan.set_timing(True)
        plan.step(u, v, p.nsteps)
        st = plan.stats()
    assert st["device_error"] == 0
    return u.double().cpu().numpy(), v.double().cpu().numpy(), st["kernels"]["mode_product_tc"]["count"]


def check(adr, p, kernel):
    u0, v0 = inputs(p)
    U, V, count = run(adr, p, u0, v0, kernel)
    assert count == (2 if p.d == 2 else 4) * p.nsteps  # one fused launch per operator (3D: and x3)
    assert oracle.max_rel_err(U, V, *reference(p, u0, v0)) <= TOL


@pytest.mark.parametrize("kernel", [0, 4])
@pytest.mark.parametrize("n,model", [((200, 136), wl.FHN), ((72, 200), wl.SCHNAKENBERG),
                                     ((128, 256), wl.BRUSSELATOR), ((8, 16), wl.FHN),
                                     ((264, 392), wl.FHN), ((256, 264), wl.SCHNAKENBERG)])
def test_2d(adr, n, model, kernel):
    check(adr, problem(n, model), kernel)


@pytest.mark.parametrize("n", [(136, 520), (200, 384)])
def test_several_x2_groups(adr, n, monkeypatch):
    monkeypatch.setenv("ADR_KSUPPORT", "0")  # every tile contracts over all of x2
    check(adr, problem(n, wl.FHN), 0)


@pytest.mark.parametrize("n", [(168, 320), (136, 264), (40, 520)])
def test_wide_supports(adr, n):
    check(adr, problem(n, wl.SCHNAKENBERG, diff=(1.0, 20.0), tau=1e-2, nsteps=4), 0)


@pytest.mark.parametrize("n", [(200, 136), (392, 264), (40, 24, 56)])
def test_lawson2b(adr, n):
    check(adr, problem(n, wl.FHN, scheme=wl.LAWSON2B), 0)


@pytest.mark.parametrize("n", [(200, 136), (392, 264), (40, 24, 56)])
def test_compensated_state(adr, n):
    check(adr, problem(n, wl.SCHNAKENBERG, state=wl.STATE_COMPENSATED, nsteps=20), 0)


@pytest.mark.parametrize("kernel", range(5))
@pytest.mark.parametrize("n,model", [((136, 24, 40), wl.FHN), ((64, 200, 72), wl.SCHNAKENBERG),
                                     ((8, 16, 8), wl.FHN), ((40, 264, 24), wl.BRUSSELATOR)])
def test_3d(adr, n, model, kernel):
    check(adr, problem(n, model, nsteps=4), kernel)


def test_3d_of_full_tiles(adr):
    check(adr, problem((128, 128, 136), wl.BRUSSELATOR, nsteps=4), 4)


@pytest.mark.parametrize("n", [(264, 392), (128, 96, 64)])
def test_agrees_with_per_direction_launches(adr, n, monkeypatch):
    p = problem(n, wl.FHN)
    u0, v0 = inputs(p)
    U, V, count = run(adr, p, u0, v0, 0)
    monkeypatch.setenv("ADR_TC_FUSED", "0")
    Ud, Vd, each = run(adr, p, u0, v0, 0)
    assert (count, each) == tuple(k * p.nsteps for k in ((2, 4) if p.d == 2 else (4, 6)))
    assert oracle.max_rel_err(U, V, Ud, Vd) <= 1e-6


@pytest.mark.parametrize("n,kernel", [((200, 200), 0), ((264, 392), 4), ((72, 40, 48), 4),
                                      ((200, 200), -1), ((264, 392), -1), ((160, 136, 24), -1)])
def test_indicators_of_every_step(adr, n, kernel):
    """Both launches (-1: the two-pass one) against the oracle's indicators."""
    import torch
    p = problem(n, wl.BRUSSELATOR, nsteps=12)
    u0, v0 = inputs(p)
    rows, prev = [], [u0, v0]

    def cb(k, U, V):
        mu, du = metrics.indicators(prev[0], U)
        mv, dv = metrics.indicators(prev[1], V)
        rows.append((mu, mv, du, dv))
        prev[0], prev[1] = U, V

    Ur, Vr = schemes.etd2rkds_solve(schemes.make_plan(p), u0, v0, p.nsteps, callback=cb)
    ref = np.array(rows)
    u = torch.tensor(u0, dtype=torch.float32, device="cuda")
    v = torch.tensor(v0, dtype=torch.float32, device="cuda")
    with adr.Plan(p, kernel=kernel) as plan:
        plan.set_indicators(True)
        plan.step(u, v, p.nsteps)
        got = plan.indicator_log()
    scale = np.abs(ref[:, :2]).max(axis=0)
    assert np.max(np.abs(got[:, :2] - ref[:, :2]) / scale) <= 1e-6
    floor = 2.0 * np.sqrt(float(np.prod(n))) * 2.0 ** -23 * np.array([np.abs(Ur).max(), np.abs(Vr).max()])
    assert np.all(np.abs(got[:, 2:] - ref[:, 2:]) <= 1e-3 * ref[:, 2:] + floor)


def test_batch_of_uneven_chunk_counts(adr):
    """A grouped launch over solves whose units have different numbers of
    64-column chunks per group: each result is the one alone, bit for bit."""
    import torch
    probs = [problem(n, m, seed=170 + i)
             for i, (n, m) in enumerate([((136, 64), wl.FHN), ((200, 256), wl.SCHNAKENBERG),
                                         ((72, 136), wl.BRUSSELATOR), ((128, 520), wl.FHN)])]
    init = [inputs(p) for p in probs]
    plans = [adr.Plan(p, kernel=0) for p in probs]
    us = [torch.tensor(u0, dtype=torch.float32, device="cuda") for u0, _ in init]
    vs = [torch.tensor(v0, dtype=torch.float32, device="cuda") for _, v0 in init]
    with adr.Batch(plans) as batch:
        assert batch.grouped
        batch.step(us, vs, 6)
        assert batch.stats()["device_error"] == 0
    for i, (p, pl, (u0, v0)) in enumerate(zip(probs, plans, init)):
        u = torch.tensor(u0, dtype=torch.float32, device="cuda")
        v = torch.tensor(v0, dtype=torch.float32, device="cuda")
        pl.step(u, v, 6)
        torch.cuda.synchronize()
        assert torch.equal(u, us[i]) and torch.equal(v, vs[i]), i
        assert oracle.max_rel_err(u.double().cpu().numpy(), v.double().cpu().numpy(),
                                  *reference(p, u0, v0)) <= TOL, i
    for pl in plans:
        pl.close()
