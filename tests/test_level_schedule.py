"""The level schedule of the light steps (several steps of one tree level per launch).

CPU: the multiplications that stand for the level kernels' index divisions, and the schedule's
memory layout (pk_plan_verify replays it) at the thresholds' ends.  GPU: every step inside a
level against the same steps launched one at a time in their own order (the finite check's
path), where each output is the same sum up to its order: K terms per output and a few hundred
steps, so a relative difference of at most about steps x K x 2^-53 (complex128) or 2^-48
(split), widened by 2^6 for cancellation between steps."""
import pytest

import knotgen as kg
import paper_1807_02119_gb300 as pk
from oracle.scaled import SC, rel_err

SHAPES = [(12, 0, 16, 16), (20, 3, 30, 60), (30, 35, 60, 160), (40, 1, 100, 400)]


def sc(s):
    return SC.of(s.mantissa, s.exp2)


def test_division_by_multiplication_is_exact_in_its_range():
    for d in [2, 3, 4, 5, 7, 9, 25, 27, 125, 729, 3125, 15625, 19683, 59049, 65535, 65536]:
        m = -(-(1 << 32) // d)
        top = ((1 << 32) - 1) // d                    # y d < 2^32
        ys = {0, 1, d - 1, d, d + 1, top, top - 1, top // 2}
        ys |= {k * d + r for k in (1, 2, top // d // 2, top // d - 1) for r in (-1, 0, 1)}
        for y in ys:
            if 0 <= y <= top:
                assert (y * m) >> 32 == y // d, (y, d)


@pytest.mark.parametrize("outs,work,k", [(1, 1, 1), (9, 81, 9), (1024, 65536, 2048), (65536, 1 << 24, 2048)])
def test_schedule_layout_verifies_at_every_threshold(outs, work, k):
    c = pk.Context(-1)
    c.set_tuning(seq_outs=outs, seq_work=work, seq_k=k)
    for L, seed, lo, hi in SHAPES[:3]:
        gk = kg.random_grid_knot(L, seed, True, lo, hi)
        kn = pk.Knot.from_pd(c, gk.pd, outer=gk.outer)
        for q in (1, 2, 5):
            for kw in ({}, {"max_log2_elems": 8.0}, {"tail_steps": 5}, {"grad": True, "checkpoint_stride": 4}):
                p = pk.Plan(c, kn, q, **kw)
                for prec in ("c128", "c64", "split"):
                    assert p.verify(prec) == "", (L, q, kw, prec, p.verify(prec))


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["c128", "split", "c64"])
@pytest.mark.parametrize("work", [81, 65536, 1 << 24])
def test_levels_match_single_steps(prec, work):
    import torch
    ctx = pk.Context(0)
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    ctx.set_tuning(seq_work=work)
    eps = {"c128": 2.0 ** -53, "split": 2.0 ** -40, "c64": 2.0 ** -24}[prec]   # split: digits of 2^-40
    for L, seed, lo, hi in SHAPES:
        gk = kg.random_grid_knot(L, seed, True, lo, hi)
        k = pk.Knot.from_pd(ctx, gk.pd, outer=gk.outer)
        for q in (2, 3, 5):
            if q == 5 and L == 40:
                continue
            p = pk.Plan(ctx, k, q)
            z, _ = pk.evaluate(p, prec)
            ctx.set_debug(pk.DEBUG_CHECK_FINITE)
            try:
                z1, _ = pk.evaluate(p, prec)
            finally:
                ctx.set_debug(0)
            kmax = max(s["K"] for s in p.steps())
            assert rel_err(sc(z), sc(z1)) <= 64 * eps * (len(p.steps()) + kmax), (L, q)


@pytest.mark.gpu
def test_noalloc_keeps_the_plans_its_workspace_held():
    """A plan whose level schedule takes more than the fixed 64 MiB while its steps' own order
    fits still runs there, with pk_eval's values."""
    import torch
    ctx = pk.Context(0)
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    for seed, prec in ((6, "split"), (16, "c128")):
        k = pk.Knot.from_grid_walk(ctx, 57, seed, True, 314, 346)
        p = pk.Plan(ctx, k, 3, restarts=16)
        assert p.workspace_bytes(prec) > 64 << 20
        z, v = pk.evaluate_noalloc(p, prec)
        z1, v1 = pk.evaluate(p, prec)
        tol = 64 * 2.0 ** (-53 if prec == "c128" else -40) * (len(p.steps()) + 729)
        assert rel_err(sc(z), sc(z1)) <= tol and rel_err(sc(v), sc(v1)) <= tol
