"""Indicator sums over the range of FP32: without reactions a solve is linear,
so fields scaled by a power of two take exactly the scaled states, and their
means and increments must be the scaled ones.  The kernels sum values of an
ordinary size in FP32 words and others in FP64 (increments below 2^-35 or from
2^40 on, values from 2^90 on); the scales put all, some or none of the points
into each.

Tolerance: both sums keep at least 53 bits of each term; at most 2^16 terms of
one sign, so 2^16 2^-53 < 1e-11."""
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


@pytest.mark.parametrize("n,kernel,state", [((200, 200), -1, wl.STATE_PLAIN),
                                            ((200, 200), -1, wl.STATE_COMPENSATED),
                                            ((128, 96), 0, wl.STATE_PLAIN),
                                            ((24, 40, 56), -1, wl.STATE_PLAIN),
                                            ((24, 40, 56), 4, wl.STATE_PLAIN)])
def test_sums_scale_with_the_fields(adr, n, kernel, state):
    import torch
    d = len(n)
    p = wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(0.02, 0.1), adv=((0.0,) * d,) * 2,
                   model=wl.NO_REACTION, params=(), tau=2e-3, nsteps=6, precision=wl.BF16X3, seed=7,
                   state=state)
    gen = torch.Generator().manual_seed(7)
    base = [0.5 + torch.rand(n[::-1], generator=gen, dtype=torch.float32) for _ in range(2)]
    logs, finals = {}, {}
    with adr.Plan(p, kernel=kernel) as plan:
        for e in (0, -30, -33, -36, 41, 60, 92):
            u, v = (torch.ldexp(x, torch.tensor(e)).cuda() for x in base)
            plan.set_indicators(True)
            plan.step(u, v, p.nsteps)
            logs[e] = plan.indicator_log() / 2.0 ** e
            finals[e] = [torch.ldexp(x.cpu(), torch.tensor(-e)) for x in (u, v)]
        assert plan.stats()["device_error"] == 0
    assert np.isfinite(logs[0]).all() and (logs[0] > 0).all()
    for e in logs:
        assert torch.equal(finals[e][0], finals[0][0]) and torch.equal(finals[e][1], finals[0][1]), e
        np.testing.assert_allclose(logs[e], logs[0], rtol=1e-11, atol=0, err_msg=str(e))
