"""adr_plan_time_mode_products leaves the plan as it was: the indicator log and
the low-order words of a compensated state belong to the state that the plan
steps, before its first step and between steps."""
import numpy as np
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


@pytest.mark.parametrize("n,kernel", [((200, 200), -1), ((96, 128), 0), ((40, 24, 56), -1),
                                      ((40, 24, 56), 4)])
def test_log_and_words_survive(adr, n, kernel):
    import torch
    d = len(n)
    p = wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(0.02, 0.1), adv=((0.1,) * d,) * 2,
                   model=wl.BRUSSELATOR, params=(1.0, 3.0), tau=2e-3, nsteps=1, precision=wl.BF16X3,
                   seed=23, state=wl.STATE_COMPENSATED)
    out = []
    for timed in (False, True):
        u, v = (torch.tensor(wl.round_to(x, wl.FP32), dtype=torch.float32, device="cuda")
                for x in wl.initial_data(p))
        scratch = u.clone(), v.clone()
        with adr.Plan(p, kernel=kernel) as plan:
            plan.set_indicators(True)
            for k in (0, 1, 20, 3):
                plan.step(u, v, k)
                if timed:
                    ms, _ = plan.time_mode_products(*scratch, reps=2)
                    assert ms > 0
            log = plan.indicator_log()
            assert plan.stats()["device_error"] == 0
        out.append((u.cpu(), v.cpu(), log))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2].shape == (24, 4)
    # per-warp sums added in FP64 in any order: at most 2^12 of them, each rounded at 2^-53
    np.testing.assert_allclose(out[1][2], out[0][2], rtol=1e-12, atol=0)
