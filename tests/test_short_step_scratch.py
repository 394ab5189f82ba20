"""Split steps with K <= 32 take no digit scratch: a plan whose tensor-core steps are all that
short has the arena alone (twice complex64's), and gives the same Z there."""
import pytest

import paper_1807_02119_gb300 as pk


@pytest.mark.parametrize("L,seed,q", [(33, 2, 3), (30, 3, 4), (33, 1, 5)])
def test_arena_alone(L, seed, q):
    ctx = pk.Context(-1)
    p = pk.Plan(ctx, pk.Knot.from_grid_walk(ctx, L, seed, True, 10, 400), q)
    ks = [s["K"] for s in p.steps() if s["tc"]]
    assert ks and max(ks) <= 32
    assert p.state_bytes("split")[1] == 2 * p.state_bytes("c64")[1]
    assert p.verify("split") == ""


@pytest.mark.gpu
@pytest.mark.parametrize("L,seed,q", [(33, 2, 3), (30, 3, 4), (33, 1, 5)])
def test_value(L, seed, q):
    import torch
    from oracle.scaled import SC, rel_err
    ctx = pk.Context(0)
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    p = pk.Plan(ctx, pk.Knot.from_grid_walk(ctx, L, seed, True, 10, 400), q)
    assert pk.profile(p, "split", _uploaded(p))["gemm_tc"]["launches"] > 0
    z, zd = pk.evaluate(p, "split")[0], pk.evaluate(p, "c128")[0]
    assert rel_err(SC.of(z.mantissa, z.exp2), SC.of(zd.mantissa, zd.exp2)) <= 1e-6   # as for split elsewhere


def _uploaded(p):
    import torch
    ws = torch.empty(p.workspace_bytes("split"), dtype=torch.uint8, device="cuda")
    pk.upload(p, "split", ws)
    return ws
