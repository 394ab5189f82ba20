"""complex128 with clause weights whose powers of two lie far apart: an output that is small
against its row's and column's largest entries keeps its digits on the tensor-core path.

All weights are positive, so no sum cancels and the relative errors of all steps add up: FP64's
are at most (K + 8) 2^-53 per step.  The tensor cores keep outputs above 2^-8 of the product of
the maxima, or with a term above 2^-10 of it; their dropped digits are at most K 7 2^14 2^48 / 2^124
= K 2^-59.2 of it, hence 14 K 2^-53 of the output."""
import math

import numpy as np
import pytest

import knotgen as kg
import paper_1807_02119_gb300 as pk
from oracle.scaled import SC, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    c = pk.Context(0)
    c.set_stream(torch.cuda.current_stream().cuda_stream)
    return c


def sc(s):
    return SC.of(s.mantissa, s.exp2)


def graded(n, J, seed):
    rng = kg.SplitMix64(seed)
    return [(math.exp((1 if rng.below(2) else -1) * J * (0.5 + rng.below(1000) / 2000)) + 0j, 1 + 0j) for _ in range(n)]


def bound(ks):
    return sum(15 * k + 16 for k in ks) * 2.0 ** -53


def conversions(p):
    import torch
    ws = torch.empty(p.workspace_bytes("c128"), dtype=torch.uint8, device="cuda")
    pk.upload(p, "c128", ws)
    return pk.profile(p, "c128", ws)["digits"]["launches"]


@pytest.mark.parametrize("q,L,seed", [(5, 33, 21), (3, 40, 1), (7, 30, 3)])
@pytest.mark.parametrize("J", [10, 20, 30, 40, 60])
def test_evaluate(ctx, q, L, seed, J):
    k = pk.Knot.from_grid_walk(ctx, L, seed, True, 60, 400)
    w = graded(k.info()["n_c"], J, J + q)
    p, pn = pk.Plan(ctx, k, q, weights=w), pk.Plan(ctx, k, q, weights=w, flags=pk.FLAG_NO_TC)
    assert conversions(p) > 0 and conversions(pn) == 0
    z, zn = pk.evaluate(p, "c128")[0], pk.evaluate(pn, "c128")[0]
    assert rel_err(sc(z), sc(zn)) <= bound(s["K"] for s in p.steps())


@pytest.mark.parametrize("q,L,seed", [(5, 33, 21), (3, 40, 1)])
def test_zeros(ctx, q, L, seed):
    """Weights of 0 (colourings): outputs without a term are 0, not formed again."""
    k = pk.Knot.from_grid_walk(ctx, L, seed, True, 60, 400)
    w = [(d, 0j if i % 3 == 0 else o) if i % 5 else (0j, o) for i, (d, o) in enumerate(graded(k.info()["n_c"], 3, 1))]
    p, pn = pk.Plan(ctx, k, q, weights=w), pk.Plan(ctx, k, q, weights=w, flags=pk.FLAG_NO_TC)
    z, zn = pk.evaluate(p, "c128")[0], pk.evaluate(pn, "c128")[0]
    assert zn.mantissa and rel_err(sc(z), sc(zn)) <= bound(s["K"] for s in p.steps())


@pytest.mark.parametrize("J", [0, 20, 60])
def test_recorded_launches_follow_new_weights(ctx, J):
    """A plan with the standard weights of q = 3, launched once, then given graded ones: Z, and
    every adjoint of the reverse pass."""
    k = pk.Knot.from_grid_walk(ctx, 53, 7, True, 300, 300)
    w = graded(k.info()["n_c"], J, 9)
    out = []
    for f in (0, pk.FLAG_NO_TC):
        p = pk.Plan(ctx, k, 3, grad=True, checkpoint_stride=4, flags=f)
        pk.evaluate(p, "c128")
        pk.grad(p, "c128")
        p.set_weights(w)
        z, _, d, _ = pk.grad(p, "c128")
        out.append((sc(pk.evaluate(p, "c128")[0]), sc(z), d))
    tol = 2 * bound([s["K"] for s in p.steps()] * 4)   # the reverse program: at most four steps for one
    for a, b in zip(out[0][:2], out[1][:2]):
        assert rel_err(a, b) <= tol
    assert np.all(np.abs(out[0][2] - out[1][2]) <= tol * np.abs(out[1][2]))
