"""2D grids of one tile of x2 around the line between the two launches (rows
that are and are no multiple of 16, narrow and wide supports, both schemes and
states): the library's choice and the launch that keeps the intermediate in TMEM
(kernel 0) form the same products in another association, so they agree to
rounding level."""
import pytest

import oracle
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


@pytest.mark.parametrize("n", [(256, 128), (264, 128), (512, 128), (1024, 64), (1000, 64), (2048, 24),
                               (2048, 128), (2056, 64)])
@pytest.mark.parametrize("hi", [1.0, 100.0])
@pytest.mark.parametrize("scheme,state", [(wl.ETD2RKDS, wl.STATE_PLAIN),
                                          (wl.ETD2RKDS, wl.STATE_COMPENSATED),
                                          (wl.LAWSON2B, wl.STATE_PLAIN)])
def test_both_launches_agree(adr, n, hi, scheme, state):
    import torch
    p = wl.Problem(d=2, n=n, lo=(0.0, 0.0), hi=(hi, hi * max(1.0, n[1] / n[0])), diff=(0.02, 0.1),
                   adv=((0.2, -0.1), (-0.2, 0.1)), model=wl.BRUSSELATOR, params=(1.0, 3.0), tau=2e-3,
                   nsteps=4, precision=wl.BF16X3, seed=41, scheme=scheme, state=state)
    gen = torch.Generator().manual_seed(41)
    base = [x + 0.2 * torch.rand(n[::-1], generator=gen, dtype=torch.float32) for x in (1.0, 3.0)]
    out = []
    for kernel in (-1, 0):
        u, v = (x.cuda() for x in base)
        with adr.Plan(p, kernel=kernel) as plan:
            plan.step(u, v, p.nsteps)
            assert plan.stats()["device_error"] == 0
        out.append([x.double().cpu().numpy() for x in (u, v)])
    assert oracle.max_rel_err(*out[0], *out[1]) <= 1e-6
