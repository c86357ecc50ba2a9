"""Batches whose solves take different launch sequences: the parts step side by
side on streams of the batch's own, and everything stays ordered on the batch's
stream: fields written on it just before the call, results read on it just
after, uneven horizons, timing mode.  Every solve equals the solve alone, bit
for bit."""
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


def problem(n, i, precision=wl.BF16X3, state=wl.STATE_PLAIN):
    d = len(n)
    return wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(0.02, 0.1),
                      adv=((0.2, -0.1, 0.3)[:d], (-0.2, 0.1, 0.05)[:d]), model=wl.BRUSSELATOR,
                      params=(1.0, 3.0), tau=2e-3, nsteps=1, precision=precision, seed=600 + i,
                      state=state)


# plans of two and three sequences (by grid, state and precision), the last part of plans that step one by one
MIXES = {
    "small_and_large": [problem((64, 64), 0), problem((200, 200), 1), problem((96, 128), 2),
                        problem((512, 512), 3)],
    "states": [problem((64, 64), 0), problem((200, 200), 1, state=wl.STATE_COMPENSATED),
               problem((160, 160), 2), problem((96, 96), 3, state=wl.STATE_COMPENSATED)],
    "with_fp32": [problem((160, 160), 0), problem((65, 33), 1, wl.FP32), problem((64, 64), 2)],
    "cubes": [problem((40, 24, 56), 0), problem((264, 256, 160), 1), problem((64, 64, 64), 2),
              problem((256, 256, 168), 3)],
}


@pytest.mark.parametrize("mix", list(MIXES))
@pytest.mark.parametrize("uneven", [False, True])
def test_parts_are_ordered_on_the_batch_stream(adr, mix, uneven):
    import torch
    probs = MIXES[mix]
    calls = [[40] * len(probs), [3] * len(probs)]
    if uneven:
        calls = [[5 + 17 * (i % 3) for i in range(len(probs))], [0] + [2] * (len(probs) - 1)]
    if probs[0].d == 3:
        calls = [[min(k, 6) for k in c] for c in calls]
    init = [[torch.tensor(wl.round_to(x, wl.FP32), dtype=torch.float32) for x in wl.initial_data(p)]
            for p in probs]
    stream = torch.cuda.Stream()
    # the low-order words of a compensated state stay with its buffers: those are written once
    once = any(p.state == wl.STATE_COMPENSATED for p in probs)
    got = []
    with torch.cuda.stream(stream):
        plans = [adr.Plan(p, stream=stream) for p in probs]
        with adr.Batch(plans, stream=stream) as batch:
            us = [torch.empty_like(u, device="cuda") for u, _ in init]
            vs = [torch.empty_like(v, device="cuda") for _, v in init]
            for timing in (False,) if once else (False, True):
                batch.set_timing(timing)
                for rep in range(1 if once else 3):  # no wait between: written, stepped, read and written again
                    for x, y, (u0, v0) in zip(us, vs, init):
                        x.copy_(u0.cuda(non_blocking=True))
                        y.copy_(v0.cuda(non_blocking=True))
                    for c in calls:
                        batch.step(us, vs, c)
                    got.append([(x.clone(), y.clone()) for x, y in zip(us, vs)])
            assert batch.stats()["device_error"] == 0
        for pl in plans:
            pl.close()
    torch.cuda.synchronize()
    for i, (p, (u0, v0)) in enumerate(zip(probs, init)):
        u, v = u0.cuda(), v0.cuda()
        with adr.Plan(p) as one:
            for c in calls:
                if c[i]:
                    one.step(u, v, c[i])
        torch.cuda.synchronize()
        assert torch.isfinite(u).all() and torch.isfinite(v).all()
        for run in got:
            assert torch.equal(run[i][0], u) and torch.equal(run[i][1], v), i
