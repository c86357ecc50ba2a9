"""Control sets of the two-pass launch (claims and dependency counters): a
step's two operators take turns with two sets, each cleared one operator ahead.
Whatever comes between steps, every launch must find its own set cleared: single
steps, replayed graphs, timed mode products (launches without row kernels
between them), another state pair, a batch over the same plans.  The results
are those of one undisturbed run, bit for bit."""
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def adr():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2307_10684_gb300 import build
    build.build()
    import paper_2307_10684_gb300 as adr
    return adr


def problem(n, scheme, state):
    d = len(n)
    return wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(0.02, 0.1),
                      adv=((0.2, -0.1, 0.3)[:d], (-0.2, 0.1, 0.05)[:d]), model=wl.BRUSSELATOR,
                      params=(1.0, 3.0), tau=2e-3, nsteps=1, precision=wl.BF16X3, seed=17,
                      scheme=scheme, state=state)


def fields(p):
    import torch
    return [torch.tensor(wl.round_to(x, wl.FP32), dtype=torch.float32, device="cuda")
            for x in wl.initial_data(p)]


@pytest.mark.parametrize("n", [(200, 200), (1024, 136), (40, 24, 56), (136, 72, 96)])
@pytest.mark.parametrize("scheme,state", [(wl.ETD2RKDS, wl.STATE_PLAIN),
                                          (wl.ETD2RKDS, wl.STATE_COMPENSATED),
                                          (wl.LAWSON2B, wl.STATE_PLAIN)])
def test_steps_between_other_launches(adr, n, scheme, state):
    import torch
    p = problem(n, scheme, state)
    calls = (1, 1, 2, 33, 1, 64, 3)
    u, v = fields(p)
    with adr.Plan(p) as plan:
        for k in calls:
            plan.step(u, v, k)
            if state == wl.STATE_COMPENSATED:  # stepping another pair restarts the low-order words
                plan.step(*fields(p), 1)
    ua, va = fields(p)
    scratch = fields(p)
    with adr.Plan(p) as plan, adr.Plan(p) as other:
        for k in calls:
            plan.step(ua, va, k)
            plan.time_mode_products(*scratch, reps=3)
            scratch = fields(p)
            plan.step(*scratch, 1)
            with adr.Batch([plan, other]) as batch:
                w = fields(p), fields(p)
                batch.step([w[0][0], w[1][0]], [w[0][1], w[1][1]], 1)
                assert batch.stats()["device_error"] == 0
            assert torch.equal(w[0][0], w[1][0]) and torch.equal(w[0][1], w[1][1])
            assert torch.equal(w[0][0], scratch[0]) and torch.equal(w[0][1], scratch[1])
        assert plan.stats()["device_error"] == 0
    torch.cuda.synchronize()
    assert torch.isfinite(u).all() and torch.isfinite(v).all()
    assert torch.equal(u, ua) and torch.equal(v, va)
