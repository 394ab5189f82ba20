"""With the standard weights and q <= 4 the nonzero entries of every tensor have one magnitude
(Gauss sums): the ground on which complex128's fixed point needs no second look there."""
import numpy as np
import pytest

import paper_1807_02119_gb300 as pk
import plan_replay as pr


def word(p):
    return int(np.frombuffer(p.debug_blob(0), dtype=np.int32)[-64])   # first of the program's last 256 bytes


@pytest.mark.parametrize("q", [1, 2, 3, 4])
@pytest.mark.parametrize("L,seed", [(16, 3), (20, 5), (26, 8)])
def test_one_magnitude(q, L, seed, monkeypatch):
    ctx = pk.Context(-1)
    p = pk.Plan(ctx, pk.Knot.from_grid_walk(ctx, L, seed, True, 10, 140), q)
    assert word(p) == 1
    step, seen = pr._step, []

    def watched(st, arena, out, mx, ex):
        step(st, arena, out, mx, ex)
        x = np.abs(out[st.off_c:st.off_c + st.R * st.N])
        x = x[x > 1e-9 * x.max()]
        seen.append(float(x.max() / x.min() - 1) if x.size else 0.0)

    monkeypatch.setattr(pr, "_step", watched)
    pr.replay(p)
    assert seen and max(seen) <= 1e-9


def test_word_follows_weights():
    ctx = pk.Context(-1)
    k = pk.Knot.from_grid_walk(ctx, 16, 3, True, 10, 140)
    assert word(pk.Plan(ctx, k, 5)) == 0
    p = pk.Plan(ctx, k, 3, grad=True)
    assert word(p) == 1
    p.set_weights([(2 + 0j, 1 + 0j)] * k.info()["n_c"])
    assert word(p) == 0
    p.set_weights(None)
    assert word(p) == 1


def test_stored_evaluations_keep_their_fingerprint():
    """The word lies behind the offsets that plan_fingerprint covers: widening records follow
    the slots (48 bytes each), rounded up to 256, also where these fill their last 256 bytes."""
    ctx = pk.Context(-1)
    full = 0
    for L in (10, 12, 14, 16, 18, 20):
        for seed in range(1, 9):
            p = pk.Plan(ctx, pk.Knot.from_grid_walk(ctx, L, seed, True, 3, 150), 3)
            sc = [int(v) for v in np.frombuffer(p.debug_blob(3), dtype=np.int64)]
            end = sc[7] + 48 * max(1, sc[8])
            full += end % 256 == 0
            assert sc[13] == (end + 255) // 256 * 256
    assert full
