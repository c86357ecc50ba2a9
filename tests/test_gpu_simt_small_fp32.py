"""FP32 mode products of launches with one 8 x 8 tile an SM at most (K split
four ways), on both sides of that line, with remainders in every dimension and
short and long K, against the FP64 oracle.

Tolerance: FP32 chains of K terms with random signs, 1e-5, as for the larger
tiles."""
import pytest

import oracle
import workloads as wl
from oracle import schemes

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


@pytest.mark.parametrize("n", [(3, 3), (3, 3, 3), (9, 9, 9), (8, 600), (600, 8), (5, 607), (72, 64),
                               (80, 64), (64, 77), (4, 130, 3), (16, 16, 17)])
@pytest.mark.parametrize("scheme", [wl.ETD2RKDS, wl.LAWSON2B])
def test_matches_oracle(adr, n, scheme):
    import torch
    d = len(n)
    p = wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(0.02, 0.1),
                   adv=((0.2, -0.1, 0.3)[:d], (-0.2, 0.1, 0.05)[:d]), model=wl.BRUSSELATOR,
                   params=(1.0, 3.0), tau=2e-3, nsteps=2, precision=wl.FP32, seed=19, scheme=scheme)
    u0, v0 = (wl.round_to(x, wl.FP32) for x in wl.initial_data(p, kind="uniform"))
    u, v = (torch.tensor(x, dtype=torch.float32, device="cuda") for x in (u0, v0))
    with adr.Plan(p) as plan:
        plan.step(u, v, p.nsteps)
    plan = schemes.make_plan(p)
    if scheme == wl.LAWSON2B:
        for _ in range(p.nsteps):
            u0, v0 = schemes.lawson2b_step(plan, u0, v0)
    else:
        u0, v0 = schemes.etd2rkds_solve(plan, u0, v0, p.nsteps)
    assert oracle.max_rel_err(u.double().cpu().numpy(), v.double().cpu().numpy(), u0, v0) <= 1e-5
