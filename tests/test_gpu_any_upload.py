"""One upload serves launches in every precision: each level schedule's records have their own
place in the workspace, and neither an evaluation in one call nor the exact residues disturb them."""
import pytest

import paper_1807_02119_gb300 as pk

pytestmark = pytest.mark.gpu

ALL = ("c128", "c64", "split")


@pytest.mark.parametrize("L,seed,q,opts", [
    (40, 1, 3, {}),                          # a schedule of its own for every precision
    (16, 3, 3, {}),                          # small steps alone: shared records
    (40, 1, 3, dict(max_log2_elems=14.0)),   # slices
])
def test_any_upload(L, seed, q, opts):
    import torch
    ctx = pk.Context(0)
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    k = pk.Knot.from_grid_walk(ctx, L, seed, True, 10, 400)
    p = pk.Plan(ctx, k, q, **opts)
    n = max(p.workspace_bytes(x) for x in ALL)

    def buffer():
        return torch.zeros(n, dtype=torch.uint8, device="cuda")

    want = {x: pk.evaluate(pk.Plan(ctx, k, q, **opts), x, buffer()) for x in ALL}
    residues = pk.evaluate_exact(p, (2147483647,), buffer())
    for up in ALL:
        ws = buffer()
        pk.upload(p, up, ws)
        for x in ALL + ALL[::-1]:
            pk.launch(p, x, ws)
            assert pk.download(p, x, ws) == want[x], (up, x)
    for up in ALL:
        ws = buffer()
        assert pk.evaluate(p, up, ws) == want[up]
        assert pk.evaluate_exact(p, (2147483647,), ws) == residues
        for x in ALL:
            pk.upload_inputs(p, x, ws)
            pk.launch(p, x, ws)
            assert pk.download(p, x, ws) == want[x], (up, x)
