"""complex64 sums stay in the steps' own order wherever a step runs: inside a level, alone (the
finite check's path, one output per thread) or in the batch executor.  Every path then does the
same FP32 operations, so the values are equal bit for bit."""
import pytest

import paper_1807_02119_gb300 as pk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    c = pk.Context(0)
    c.set_stream(torch.cuda.current_stream().cuda_stream)
    return c


def bits(s):
    return (s.re, s.im, s.exp2)


@pytest.mark.parametrize("L,seed,lo,hi,q,longest", [
    (57, 9, 314, 346, 3, 81),
    (40, 12, 100, 300, 3, 81),
    (33, 4, 100, 200, 5, 125),
    (34, 22, 70, 200, 4, 16),
    (20, 3, 30, 60, 3, 9),
])
def test_levels_keep_the_order_of_single_steps(ctx, L, seed, lo, hi, q, longest):
    k = pk.Knot.from_grid_walk(ctx, L, seed, True, lo, hi)
    p = pk.Plan(ctx, k, q)
    assert any(s["K"] >= longest and s["R"] * s["N"] * s["K"] <= 1 << 22 for s in p.steps() if s["kernel"] == 0)
    z, v = pk.evaluate(p, "c64")
    ctx.set_debug(pk.DEBUG_CHECK_FINITE)
    try:
        z1, v1 = pk.evaluate(p, "c64")
    finally:
        ctx.set_debug(0)
    assert bits(z) == bits(z1) and bits(v) == bits(v1)


def test_batch_keeps_the_order_of_single_steps(ctx):
    plans = []
    for seed in range(1, 40):
        for q in (3, 4, 5):
            p = pk.Plan(ctx, pk.Knot.from_grid_walk(ctx, 20, seed, True, 20, 60), q)
            if all(s["kernel"] == 0 for s in p.steps()):   # split-K sums have an order of their own
                plans.append(p)
    assert any(s["K"] > 16 for p in plans for s in p.steps())
    zs, _ = pk.evaluate_batch(plans, "c64")
    ctx.set_debug(pk.DEBUG_CHECK_FINITE)
    try:
        one = [pk.evaluate(p, "c64")[0] for p in plans]
    finally:
        ctx.set_debug(0)
    assert [bits(z) for z in zs] == [bits(z) for z in one]
