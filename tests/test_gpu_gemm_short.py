"""Split GEMM steps with K <= 32 in one tensor-core kernel, against the same plans on the CUDA
cores and complex128: every step forced onto GEMM, so that K, the rows and the columns take the
powers of q around each edge (K = 8, 16, 32 and past it, one to several column tiles, ragged and
whole row blocks).

S digits leave 2^(-8S-6) of each operand's largest entry and drop levels below 2^(-8S): less than
2^(-8S+3) per term; over a plan at most (steps + K) of that, widened by 2^6 for cancellation."""
import pytest

import knotgen as kg
import paper_1807_02119_gb300 as pk
from oracle.scaled import SC, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q,L,n,want", [(2, 48, 200, {2, 8, 16, 32, 64}), (3, 34, 80, {3, 9, 27, 81}), (4, 30, 60, {4, 16}),
                                        (5, 30, 50, {5, 25, 125}), (6, 26, 40, {6, 36})])
@pytest.mark.parametrize("digits,flag", [(5, 0), (4, pk.FLAG_TC_DIGITS4)])
def test_matches_cuda_cores_and_complex128(q, L, n, want, digits, flag):
    import torch
    ctx = pk.Context(0)
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    seen = set()
    for seed in range(4):
        gk = kg.random_grid_knot(L, 70 + seed, True, n, 3 * n)
        k = pk.Knot.from_pd(ctx, gk.pd, outer=gk.outer)
        p = pk.Plan(ctx, k, q, flags=pk.FLAG_FORCE_GEMM | flag)
        steps = [s for s in p.steps() if s["kernel"] == 2]
        seen |= {s["K"] for s in steps}
        tol = 64 * (len(p.steps()) + max(s["K"] for s in steps)) * 2.0 ** (3 - 8 * digits)
        out = [pk.evaluate(p, "split"), pk.evaluate(p, "c128"),
               pk.evaluate(pk.Plan(ctx, k, q, flags=pk.FLAG_FORCE_GEMM | pk.FLAG_NO_TC), "split")]
        z = [[SC.of(x.mantissa, x.exp2) for x in o] for o in out]
        assert rel_err(z[0][0], z[1][0]) <= tol and rel_err(z[0][1], z[1][1]) <= tol, (seed, seen)
        assert rel_err(z[0][0], z[2][0]) <= tol, seed
    assert want <= seen, seen
