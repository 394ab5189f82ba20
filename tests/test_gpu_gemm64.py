"""complex128 GEMM steps on the tensor cores (64-bit fixed point in eight BF16 digits): against
the same plans on the FP64 units (PK_FLAG_NO_TC) and the CPU oracle.

The digits keep 2^-62 of a row's and a column's largest entries, so a step is no further from
the exact sum than FP64's own rounding (K terms of 2^-53); the two paths may then differ by the
FP64 path's error, at most steps x K x 2^-53 of the result, widened by 2^6 for the cancellation
between steps."""
import pytest

import knotgen as kg
import oracle
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


def tc64_steps(p):
    """Steps of the size and shape that complex128 runs on the tensor cores."""
    return [s for s in p.steps() if s["b"] >= 0 and s["kernel"] != 1 and s["R"] // s["Bsz"] >= 64 and
            s["N"] >= 4 and 4 <= s["K"] <= 4096 and
            s["R"] * s["K"] * s["N"] >= (1 << 19 if s["kernel"] == 2 else 1 << 20)]


@pytest.mark.parametrize("L,seed,q,least", [
    (40, 1, 3, 1),     # ragged tiles: 243 rows, 27 and 81 columns
    (33, 21, 5, 4),    # K from 5 (one padded chunk) to 125 (three flush groups)
    (29, 57, 5, 4),
    (34, 22, 4, 1),    # powers of two: no ragged edge
    (40, 3, 5, 6),     # batch indices outside the tile, K = 625
])
def test_matches_fp64_and_oracle(ctx, L, seed, q, least):
    gk = kg.random_grid_knot(L, seed, True, 70, 400)
    k = pk.Knot.from_pd(ctx, gk.pd, outer=gk.outer)
    p, pn = pk.Plan(ctx, k, q), pk.Plan(ctx, k, q, flags=pk.FLAG_NO_TC)
    steps = tc64_steps(p)
    assert len(steps) >= least, len(steps)
    tol = 64 * 2.0 ** -53 * (len(p.steps()) + max(s["K"] for s in p.steps()))
    z, v = pk.evaluate(p, "c128")
    zn, vn = pk.evaluate(pn, "c128")
    assert rel_err(sc(z), sc(zn)) <= tol and rel_err(sc(v), sc(vn)) <= tol
    g = oracle.tait_graph(gk.pd, outer=gk.outer)
    if q ** max(s["rank_c"] for s in p.steps()) <= 3 ** 12:
        assert rel_err(sc(z), oracle.z_complex(g.n_v, g.edges, q)) <= 1e-10


def test_reverse_pass_uses_it(ctx):
    """300 crossings at q = 3: the adjoint steps' wide contractions, against the FP64 units."""
    import numpy as np
    k = pk.Knot.from_grid_walk(ctx, 53, 7, True, 300, 300)
    out = [pk.grad(pk.Plan(ctx, k, 3, grad=True, checkpoint_stride=4, flags=f), "c128")
           for f in (0, pk.FLAG_NO_TC)]
    assert rel_err(sc(out[0][0]), sc(out[1][0])) <= 64 * 2.0 ** -53 * 1500
    scale = max(1.0, float(np.max(np.abs(out[1][2]))))
    assert float(np.max(np.abs(out[0][2] - out[1][2]))) <= 64 * 2.0 ** -53 * 3000 * scale


def test_weights_of_every_size(ctx):
    """Clause weights scaled by powers of two up to 2^1000: rows whose exponents lie far apart."""
    k = pk.Knot.from_grid_walk(ctx, 33, 21, True, 70, 140)
    rng = kg.SplitMix64(5)
    one, big, tot = [], [], 0
    for i in range(k.info()["n_c"]):
        d = complex(1 + rng.below(100) / 50, rng.below(100) / 50 - 1)
        s = int(rng.below(2001)) - 1000
        one.append((d, 1 - 0.5j))
        big.append((d * 2.0 ** s, (1 - 0.5j) * 2.0 ** s))
        tot += s
    pa, pb = pk.Plan(ctx, k, 5, weights=one), pk.Plan(ctx, k, 5, weights=big)
    assert tc64_steps(pa)
    za, zb = pk.evaluate(pa, "c128")[0], pk.evaluate(pb, "c128")[0]
    assert rel_err(sc(zb), sc(za) * SC.of(1.0 + 0j, tot)) <= 64 * 2.0 ** -53 * 1000


def test_nan_stays_nan(ctx):
    """A NaN planted in one uploaded clause value reaches Z through the tensor-core steps."""
    import ctypes as C
    import math
    import struct
    import torch
    k = pk.Knot.from_grid_walk(ctx, 33, 21, True, 70, 140)
    p = pk.Plan(ctx, k, 5)
    assert tc64_steps(p)
    scal = struct.unpack(f"<{len(p.debug_blob(3)) // 8}q", p.debug_blob(3))
    off_slots, n_slots = scal[7], scal[8]
    prog = p.debug_blob(0)
    at = next(off_slots + 48 * i for i in range(n_slots)
              if struct.unpack_from("<4i", prog, off_slots + 48 * i)[2] == 1) + 16
    ws = pk.workspace(p, "c128")
    pk.upload(p, "c128", ws)
    ws[at:at + 8].copy_(torch.tensor(list(struct.pack("<d", math.nan)), dtype=torch.uint8, device="cuda"))
    pk.launch(p, "c128", ws)
    z, v = pk.pk_scaled(), pk.pk_scaled()
    assert pk.lib().pk_download(ctx.h, p.h, 0, C.c_void_p(ws.data_ptr()), C.byref(z), C.byref(v)) == 0
    assert math.isnan(z.re) or math.isnan(z.im)
