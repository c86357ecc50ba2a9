"""The two-pass launch on 3D grids large enough that its passes interleave (the
x2 tiles of a run of slabs follow the x1 tiles of the next run), against the
launch that keeps the intermediate in TMEM: the same products in another
association, so they agree to rounding level."""
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


@pytest.mark.parametrize("n", [(176, 176, 176), (192, 136, 264), (264, 200, 104)])
@pytest.mark.parametrize("state", [wl.STATE_PLAIN, wl.STATE_COMPENSATED])
def test_interleaved_passes(adr, n, state):
    import torch
    p = wl.Problem(d=3, n=n, lo=(0.0,) * 3, hi=(1.0,) * 3, diff=(0.02, 0.1),
                   adv=((0.2, -0.1, 0.3), (-0.2, 0.1, 0.05)), model=wl.BRUSSELATOR, params=(1.0, 3.0),
                   tau=2e-3, nsteps=3, precision=wl.BF16X3, seed=5, state=state)
    gen = torch.Generator().manual_seed(5)
    base = [x + 0.2 * torch.rand(n[::-1], generator=gen, dtype=torch.float32) for x in (1.0, 3.0)]
    out = []
    for kernel in (-1, 0):
        u, v = (x.cuda() for x in base)
        with adr.Plan(p, kernel=kernel) as plan:
            plan.step(u, v, p.nsteps)
            assert plan.stats()["device_error"] == 0
        out.append([x.double().cpu().numpy() for x in (u, v)])
    assert oracle.max_rel_err(*out[0], *out[1]) <= 1e-6
