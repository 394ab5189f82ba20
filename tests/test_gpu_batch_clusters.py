"""The batch launch with knots on both sides of the line above which a cluster takes a knot (5e4
to 8e5 multiply-adds in a small batch, by precision), against single evaluations of the same plans.

Both run the same steps; a term's error is 2^-53 in complex128, below 2^-37 on split's digits and
2^-24 in complex64, over a plan at most (steps + K) of them, widened by 2^6 for cancellation."""
import pytest

import knotgen as kg
import paper_1807_02119_gb300 as pk
from oracle.scaled import SC, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,eps", [("c128", 2.0 ** -53), ("split", 2.0 ** -37), ("c64", 2.0 ** -24)])
@pytest.mark.parametrize("q", [3, 5])
def test_small_and_large_knots(prec, eps, q):
    import torch
    ctx = pk.Context(0)
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    sizes = [(14, 16, 24), (30, 60, 99), (18, 30, 50), (46, 180, 260) if q == 3 else (33, 70, 110), (12, 12, 20)]
    plans = []
    for i, (L, lo, hi) in enumerate(sizes):
        gk = kg.random_grid_knot(L, 300 + i, True, lo, hi)
        plans.append(pk.Plan(ctx, pk.Knot.from_pd(ctx, gk.pd, outer=gk.outer), q))
    work = [sum(s["R"] * s["K"] * s["N"] for s in p.steps()) for p in plans]
    assert min(work) < 5e4 and max(work) > 8e5, work
    b = pk.Batch(plans, prec)
    ws = torch.empty(b.workspace_bytes()[0], dtype=torch.uint8, device="cuda")
    b.upload(ws)
    for _ in range(2):
        b.launch(ws)
    zs, vs = b.download(ws)[:2]
    for p, z, v in zip(plans, zs, vs):
        tol = 64 * (len(p.steps()) + max(s["K"] for s in p.steps())) * eps
        ze, ve = pk.evaluate(p, prec)
        assert rel_err(SC.of(z.mantissa, z.exp2), SC.of(ze.mantissa, ze.exp2)) <= tol
        assert rel_err(SC.of(v.mantissa, v.exp2), SC.of(ve.mantissa, ve.exp2)) <= tol
