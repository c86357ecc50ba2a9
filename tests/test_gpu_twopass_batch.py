"""Grouped batches of plans that take the two-pass launch: every solve equals
the same solve alone, bit for bit.

Each solve of a batch has dependency counters of its own.  The mixes put solves
whose x1 tiles are quick beside solves whose x1 tiles are slow, in both orders,
over one to a few units per SM, so that an x2 tile taken as ready because a
tile of another solve with the same indices was would read pieces that its own
x1 tile has not written yet.

Tolerance of the indicators: their per-warp sums are added by FP64 atomics in
any order; at most 2^14 of them, each rounded at 2^-53, stay within 1e-11."""
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


def wide(n, i, state=wl.STATE_PLAIN):
    """Schnakenberg on the unit square or cube: supports as wide as the grid."""
    d = len(n)
    return wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(1.0, 10.0),
                      adv=((0.0,) * d, (0.0,) * d), model=wl.SCHNAKENBERG,
                      params=(100.0 + 20.0 * i, 0.1, 0.9), tau=2e-4, nsteps=1,
                      precision=wl.BF16X3, seed=300 + i, state=state)


def fields(p):
    import torch
    return [torch.tensor(wl.round_to(x, wl.FP32), dtype=torch.float32, device="cuda")
            for x in wl.initial_data(p)]


MIXES = {
    "two_512": [(512, 512)] * 2,
    "eight_512": [(512, 512)] * 8,
    "twenty_136_512": [(136, 136), (512, 512)] * 10,
    "twenty_512_136": [(512, 512), (136, 136)] * 10,
    "short_then_long": [(384, 192), (1024, 1024)],
    "long_then_short": [(1024, 1024), (384, 192)],
    "cubes": [(96, 24, 40), (160, 160, 64), (24, 96, 40), (160, 160, 64)],
    "rows": [(64, 64, 64), (264, 40, 24), (192, 24, 40), (200, 64, 16)],  # both 3D stencils
    "slabs": [(64, 64, 96), (192, 136, 40), (64, 64, 96), (40, 200, 24)],
}


@pytest.mark.parametrize("mix", list(MIXES))
@pytest.mark.parametrize("option", ["plain", "compensated", "indicators"])
def test_batch_equals_each_solve_alone(adr, mix, option):
    import torch
    calls = (3, 97, 100)  # one by one, then by replayed graphs
    state = wl.STATE_COMPENSATED if option == "compensated" else wl.STATE_PLAIN
    probs = [wide(n, i, state) for i, n in enumerate(MIXES[mix])]
    plans = [adr.Plan(p) for p in probs]
    if option == "indicators":
        for pl in plans:
            pl.set_indicators(True)
    init = [fields(p) for p in probs]
    us, vs = [f[0].clone() for f in init], [f[1].clone() for f in init]
    with adr.Batch(plans) as batch:
        assert batch.grouped
        for k in calls:
            batch.step(us, vs, k)
        assert batch.stats()["device_error"] == 0
    logs = [pl.indicator_log() for pl in plans] if option == "indicators" else None
    for i, (p, (u, v)) in enumerate(zip(probs, init)):
        with adr.Plan(p) as one:
            one.set_indicators(option == "indicators")
            for k in calls:
                one.step(u, v, k)
            assert one.stats()["device_error"] == 0
            log = one.indicator_log() if logs else None
        torch.cuda.synchronize()
        assert torch.isfinite(u).all() and torch.isfinite(v).all(), i
        assert torch.equal(u, us[i]) and torch.equal(v, vs[i]), i
        if logs:
            np.testing.assert_allclose(logs[i], log, rtol=1e-11, atol=0, err_msg=str(i))
    for pl in plans:
        pl.close()
