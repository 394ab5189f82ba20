"""A plan whose steps are all forced on one kernel has no complex128 step on the tensor cores:
the same launches and workspace as with PK_FLAG_NO_TC besides."""
import pytest

import paper_1807_02119_gb300 as pk


@pytest.mark.parametrize("force", [pk.FLAG_FORCE_ROWS, pk.FLAG_FORCE_GEMM])
@pytest.mark.parametrize("L,seed,q", [(33, 21, 5), (40, 1, 3)])
def test_no_tensor_core_step(force, L, seed, q):
    ctx = pk.Context(-1)
    k = pk.Knot.from_grid_walk(ctx, L, seed, True, 70, 400)

    def plan(flags):
        p = pk.Plan(ctx, k, q, flags=flags, grad=True, checkpoint_stride=4)
        return p.launches("c128"), p.workspace_bytes("c128"), p.grad_workspace_bytes("c128")

    assert plan(0)[1] > plan(pk.FLAG_NO_TC)[1]   # the knot has such steps
    assert plan(force) == plan(force | pk.FLAG_NO_TC)
