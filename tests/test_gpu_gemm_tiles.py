"""GEMM steps on the CUDA cores in both tile sizes (64 x 64, and 32 x 32 for fewer than two tiles per
multiprocessor) against the same knot with every step on the row kernels.

A sum of K terms is off by at most K 2^-p of its terms in either path (p = 24 or 53): over a plan
(steps + K) 2^-p, widened by 2^6 for cancellation."""
import pytest

import knotgen as kg
import paper_1807_02119_gb300 as pk
from oracle.scaled import SC, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,eps", [("c64", 2.0 ** -24), ("c128", 2.0 ** -53), ("split", 2.0 ** -44)])
@pytest.mark.parametrize("q,L,seed", [(5, 40, 3), (3, 40, 1), (4, 34, 22)])
def test_matches_row_kernels(prec, eps, q, L, seed):
    import torch
    ctx = pk.Context(0)
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    gk = kg.random_grid_knot(L, seed, True, 70, 400)
    k = pk.Knot.from_pd(ctx, gk.pd, outer=gk.outer)
    p = pk.Plan(ctx, k, q, flags=pk.FLAG_NO_TC)
    gemm = [s for s in p.steps() if s["kernel"] == 2]
    tiles = [-(-s["R"] // s["Bsz"] // 64) * -(-s["N"] // 64) * s["Bsz"] for s in gemm]
    assert max(tiles) >= 304 if q == 5 else 0 < max(tiles) < 304, tiles
    tol = 64 * (len(p.steps()) + max(s["K"] for s in p.steps())) * eps
    z, v = pk.evaluate(p, prec)
    zr, vr = pk.evaluate(pk.Plan(ctx, k, q, flags=pk.FLAG_NO_TC | pk.FLAG_FORCE_ROWS), prec)
    c = lambda s: SC.of(s.mantissa, s.exp2)
    assert rel_err(c(z), c(zr)) <= tol and rel_err(c(v), c(vr)) <= tol
