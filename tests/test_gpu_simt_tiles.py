"""The FP64 and FP32 mode products against the FP64 oracle at sizes that take
each tile of the GEMM (8 x 8 with K split four or two ways and, beyond 8 x 65535
rows, 64 x 64 in FP64; 32 x 32, 64 x 32, 64 x 64 and 128 x 128 in FP32), with remainders in every
dimension, K on either side of a pipeline stage, and rows that do and do not
start on 16 bytes.

Tolerance: of the oracle's arithmetic in FP64 (1e-11), of FP32 chains of K
terms with random signs (1e-5), the bounds of the other parity tests."""
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


@pytest.mark.parametrize("precision,n", [
    (wl.FP64, (3, 5)), (wl.FP64, (8, 64)), (wl.FP64, (63, 66)), (wl.FP64, (129, 127)), (wl.FP64, (130, 72)),
    (wl.FP64, (40, 40, 33)), (wl.FP64, (5, 17, 131)), (wl.FP64, (700, 690)), (wl.FP64, (3, 800, 700)),
    (wl.FP32, (3, 5)), (wl.FP32, (36, 64)), (wl.FP32, (65, 130)), (wl.FP32, (300, 258)), (wl.FP32, (36, 39, 31)),
    (wl.FP32, (641, 255)), (wl.FP32, (1028, 900))])
def test_tiles_match_oracle(adr, precision, n):
    import torch
    d = len(n)
    p = wl.Problem(d=d, n=n, lo=(0.0,) * d, hi=(1.0,) * d, diff=(0.02, 0.1),
                   adv=((0.2, -0.1, 0.3)[:d], (-0.2, 0.1, 0.05)[:d]), model=wl.BRUSSELATOR,
                   params=(1.0, 3.0), tau=2e-3, nsteps=2, precision=precision, seed=17,
                   scheme=wl.ETD2RKDS)
    dt = torch.float64 if precision == wl.FP64 else torch.float32
    u0, v0 = wl.initial_data(p, kind="uniform")
    if precision == wl.FP32:
        u0, v0 = wl.round_to(u0, wl.FP32), wl.round_to(v0, wl.FP32)
    u, v = (torch.tensor(x, dtype=dt, device="cuda") for x in (u0, v0))
    with adr.Plan(p) as plan:
        plan.step(u, v, p.nsteps)
    ru, rv = schemes.etd2rkds_solve(schemes.make_plan(p), u0, v0, p.nsteps)
    err = oracle.max_rel_err(u.double().cpu().numpy(), v.double().cpu().numpy(), ru, rv)
    assert err <= (1e-11 if precision == wl.FP64 else 1e-5)
