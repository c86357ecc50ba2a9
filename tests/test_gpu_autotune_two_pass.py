"""The autotuners time the two-pass launch where the library's choice is that
one: a problem it serves best tunes to kernel -1, a batch of such problems keeps
it, and problems that differ only in their supports are tuned apart."""
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


def wide(n):
    d = len(n)
    return wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(0.02, 0.1),
                      adv=((0.0,) * d,) * 2, model=wl.BRUSSELATOR, params=(1.0, 3.0), tau=2e-3,
                      nsteps=1, precision=wl.BF16X3, seed=1)


@pytest.mark.parametrize("n", [(512, 512), (160, 160), (40, 64, 48)])
def test_the_two_pass_launch_is_a_candidate(adr, n):
    p = wide(n)
    best, ms = adr.autotune(p, nsteps=8, cache=False)
    assert set(ms) == {-1, 0, 1, 2, 3, 4} and all(t > 0 for t in ms.values())
    assert best == min(ms, key=ms.get)
    with adr.Plan(p) as plan:
        assert plan.two_pass
        plan.set_kernel(0)
        assert not plan.two_pass
        plan.set_kernel(best)
        assert plan.two_pass == (best == -1)


def test_wide_supports_tune_to_it(adr):
    """512^2: 53 us a step with two passes against 77 with the best other kernel."""
    assert adr.autotune(wide((512, 512)), nsteps=32, cache=False)[0] == -1


def test_supports_are_part_of_the_cache_key(adr):
    p = wide((512, 512))
    narrow = p.replace(hi=(100.0, 100.0))
    assert adr.autotune(p, nsteps=4) is adr.autotune(p.replace(seed=9), nsteps=4)
    assert -1 in adr.autotune(p, nsteps=4)[1]
    assert -1 not in adr.autotune(narrow, nsteps=4)[1]


@pytest.mark.parametrize("sides", [(512, 512), (64, 512)])
def test_a_batch_keeps_it(adr, sides):
    plans = [adr.Plan(wide((k, k))) for k in sides]
    best, ms = adr.autotune_batch(plans, nsteps=4)
    assert set(ms) == {-1, 0, 1, 2, 3, 4} and best == min(ms, key=ms.get)
    assert [pl.two_pass for pl in plans] == [best == -1 and k == 512 for k in sides]
    for pl in plans:
        pl.close()


def test_other_plans_have_none(adr):
    p = wl.fhn_1024(precision=wl.BF16X3, n=64)
    for q in (p, p.replace(precision=wl.FP32)):
        with adr.Plan(q) as plan:
            assert not plan.two_pass
