"""The work that a user of this package gives it, as cases to be timed: evaluations of single
knots in every precision, groups and batches of knots, reverse passes, exact residues.

A case fixes the shapes (a random grid-walk diagram, q, the planner's options); the seed of
prepare() draws every crossing's over / under bit, so another seed is another knot on the
same shadow.  What prepare() returns is what a program keeps between calls: the context, the
plan, its device workspace (and the group or batch made of them).
"""
import math
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_1807_02119_gb300 as pk

DEVICE = "cuda:0"
QS = (2, 3, 5)                              # the q of the paper's evaluations
PRIMES = (2147483647, 2147483629, 2147483587, 2147483579)   # the largest below 2^31


def listed():
    return [
        # the smallest call: a textbook-size knot, default precision (latency and launches)
        dict(name="eval_tiny_c128", kind="eval", crossings=16, knot=0, q=3, precision="c128"),
        # the ordinary call: one 205-crossing knot, every option at its default
        dict(name="eval_q3_c128", kind="eval", crossings=205, knot=1, q=3, precision="c128"),
        # one knot of the paper's size at q = 5 in the throughput precision, planned with effort
        dict(name="eval_q5_split", kind="eval", crossings=167, knot=2, q=5, precision="split",
             restarts=64, refine=8),
        # the same kind of knot in the reference precision: a screening result confirmed
        dict(name="eval_q5_c128", kind="eval", crossings=167, knot=2, q=5, precision="c128",
             restarts=64, refine=8),
        # plain complex64 on a knot at the upper end of the paper's sizes
        dict(name="eval_q3_c64", kind="eval", crossings=330, knot=3, q=3, precision="c64", restarts=32),
        # a 491-crossing knot cut into slices to bound the memory of its tensors
        dict(name="eval_sliced_split", kind="eval", crossings=420, knot=1, q=3, precision="split",
             restarts=32, max_log2_elems=19.0),
        # many knots at q = 2, 3, 5 as concurrent branches of one graph (a survey of knots)
        dict(name="group_split", kind="group", knots=16, lo=100, hi=400, side=40, knot=1,
             precision="split", restarts=64, refine=8),
        # many small knots in one persistent launch, in the throughput precision
        dict(name="batch_q3_split", kind="batch", knots=1024, lo=20, hi=120, knot=1, q=3,
             precision="split"),
        # fewer of them in the reference precision at q = 5
        dict(name="batch_q5_c128", kind="batch", knots=192, lo=20, hi=60, knot=7, q=5,
             precision="c128"),
        # the reverse pass over a 300-crossing knot: a gradient step of a Potts fit
        dict(name="grad_q3_c128", kind="grad", crossings=300, knot=7, q=3, precision="c128", stride=4),
        # the reverse pass in the throughput precision on a wider network
        dict(name="grad_q5_split", kind="grad", crossings=99, knot=1, q=5, precision="split", stride=4),
        # Z(q) modulo four primes: one node of the interpolation of a 36-crossing knot's polynomial
        dict(name="exact_q10", kind="exact", crossings=36, knot=2, q=10),
    ]


# Complex multiply-adds that a drawn case may need, by kind: below the largest listed one.
MOST = {"eval": 4e9, "group": 3e9, "batch": 4e8, "grad": 2.5e8, "exact": 2.4e6}


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(("eval", "eval", "eval", "group", "batch", "grad", "exact"))
        c = dict(kind=kind, knot=rng.randrange(1, 10000))
        if kind in ("eval", "grad", "exact"):
            c["q"] = rng.choice((2, 3, 4, 5)) if kind != "exact" else rng.randrange(2, 13)
            most = {"eval": (400, 400, 200, 170), "grad": (300, 300, 150, 110)}.get(kind)
            c["crossings"] = spread(12, most[c["q"] - 2] if most else 45)
        if kind == "eval":
            c["precision"] = rng.choice(("c128", "c128", "split", "split", "c64"))
            if rng.random() < 0.5:
                c.update(restarts=rng.choice((16, 32, 64)))
                if c["precision"] == "split":
                    c["refine"] = 8
            if rng.random() < 0.15:
                c["max_log2_elems"] = 20.0
        elif kind == "grad":
            c.update(precision=rng.choice(("c128", "split")), stride=rng.choice((1, 2, 4)))
        elif kind == "group":
            side = rng.randrange(20, 41)
            c.update(knots=spread(2, 16), side=side, lo=max(8, side * side // 16), hi=side * side // 4,
                     precision="split", restarts=rng.choice((16, 64)), refine=8)
        elif kind == "batch":
            lo = rng.randrange(10, 30)
            c.update(knots=spread(5, 800), lo=lo, hi=lo + rng.randrange(10, 60), q=rng.choice((2, 3, 4)),
                     precision=rng.choice(("split", "c128", "c64")))
        if _work_of(c)["cmacs"] <= MOST[kind]:
            return c


# ------------------------------------------------------------------ inputs

_shadows = {}


def _shadow(ctx, side, knot, lo, hi):
    """PD code of a random grid walk with lo..hi crossings (grid side 0: from the crossings)."""
    key = (side, knot, lo, hi)
    if key not in _shadows:
        L = side or max(6, round(math.sqrt((lo + hi) / 0.2)))
        _shadows[key] = pk.Knot.from_grid_walk(ctx, L, knot, True, lo, hi).pd()
    return _shadows[key]


def _with_bits(pd, bits):
    """The diagram with over and under exchanged where the bit is 1.  (a, b, c, d): a the
    incoming under-arc, then counter-clockwise; arcs are numbered along the knot."""
    out = []
    for (a, b, c, d), x in zip(pd, bits):
        if not x:
            out.append((a, b, c, d))
        elif (d + 1) % (2 * len(pd)) == b:   # the over-strand enters through d
            out.append((d, a, b, c))
        else:
            out.append((b, c, d, a))
    return out


def _shadows_of(ctx, case):
    if case["kind"] in ("eval", "grad", "exact"):
        n = case["crossings"]
        return [_shadow(ctx, 0, case["knot"], n - n // 20, n + n // 20)]
    if case["kind"] == "group":
        return [_shadow(ctx, case["side"], case["knot"] + i, case["lo"], case["hi"])
                for i in range(case["knots"])]
    out = []   # batch: targets spread evenly over lo..hi
    for i in range(case["knots"]):
        n = case["lo"] + (i * 37) % (case["hi"] - case["lo"] + 1)
        out.append(_shadow(ctx, 0, case["knot"] + i, n - 2, n + 2))
    return out


def _diagrams(ctx, case, seed):
    r = np.random.RandomState(seed % (1 << 31))
    return [_with_bits(pd, r.randint(0, 2, len(pd))) for pd in _shadows_of(ctx, case)]


def _plans(ctx, case, pds):
    kw = {k: case[k] for k in ("restarts", "refine", "max_log2_elems") if k in case}
    if case["kind"] == "grad":
        kw.update(grad=True, checkpoint_stride=case["stride"])
    jobs = [(pk.Knot.from_pd(ctx, pd), q) for pd in pds
            for q in (QS if case["kind"] == "group" else (case["q"],))]
    if len(jobs) == 1:
        return [pk.Plan(ctx, jobs[0][0], jobs[0][1], **kw)]
    with ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as ex:
        return list(ex.map(lambda j: pk.Plan(ctx, j[0], j[1], **kw), jobs))


def _buffer(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device=DEVICE)


def prepare(case, seed):
    ctx = pk.Context(0, torch.cuda.current_stream().cuda_stream)
    plans = _plans(ctx, case, _diagrams(ctx, case, seed))
    s = dict(kind=case["kind"], precision=case.get("precision"), ctx=ctx, plans=plans, plan=plans[0])
    if case["kind"] == "eval":
        s["ws"] = _buffer(plans[0].workspace_bytes(case["precision"]))
    elif case["kind"] == "grad":
        s["ws"] = _buffer(plans[0].grad_workspace_bytes(case["precision"]))
    elif case["kind"] == "exact":
        s["ws"] = _buffer(plans[0].workspace_bytes("c64"))
    elif case["kind"] == "group":
        s["ws"] = [_buffer(p.workspace_bytes(case["precision"])) for p in plans]
        s["group"] = pk.Group(plans, case["precision"], s["ws"])
        s["group"].upload()
    else:
        s["batch"] = pk.Batch(plans, case["precision"])
        s["ws"] = _buffer(s["batch"].workspace_bytes()[0])
        s["batch"].upload(s["ws"])
    return s


# ------------------------------------------------------------------ one pass

def _values(precision, zs, vs):
    """The values as numbers: complex64 results in complex64, the others in complex128."""
    t = np.complex64 if precision == "c64" else np.complex128
    # Z leaves the range of complex64 for larger knots: there it stays in V alone
    out = {"v": np.array([v.to_complex() for v in vs], dtype=t)}
    if precision != "c64":
        out["z"] = np.array([z.to_complex() for z in zs], dtype=t)
    return out


def run(state):
    kind, precision = state["kind"], state["precision"]
    if kind == "eval":
        z, v = pk.evaluate(state["plan"], precision, state["ws"])
        return _values(precision, [z], [v])
    if kind == "grad":
        z, v, dlogz, dlogv = pk.grad(state["plan"], precision, state["ws"])
        return dict(_values(precision, [z], [v]), dlogz=dlogz, dlogv=np.array([dlogv]))
    if kind == "exact":
        return np.array(pk.evaluate_exact(state["plan"], PRIMES, state["ws"]), dtype=np.int64)
    if kind == "group":
        state["group"].launch()
        zv = state["group"].download()
        out = {}
        for i, q in enumerate(QS):
            out["q%d" % q] = _values(precision, [z for z, _ in zv[i::len(QS)]], [v for _, v in zv[i::len(QS)]])
        return out
    state["batch"].launch(state["ws"])
    return _values(precision, *state["batch"].download(state["ws"]))


# ------------------------------------------------------------------ what a pass cannot do without

_work = {}


def _work_of(case):
    """Complex multiply-adds of the plans (the shadows as they are), edges and evaluations."""
    key = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _work:
        ctx = pk.Context(-1)
        pds = _shadows_of(ctx, case)
        plans = _plans(ctx, case, pds)
        if case["kind"] == "grad":
            g = plans[0].grad_stats()
            cm = (g["cmacs_forward"] + g["cmacs_adjoint"]) * g["slices"]
        else:
            cm = sum(p.stats()["cmacs"] for p in plans)
        _work[key] = {"cmacs": cm, "edges": sum(len(p) for p in pds) * len(plans) // len(pds), "evals": len(plans)}
    return _work[key]


def work(case):
    """A clause matrix (its diagonal and its off-diagonal weight, complex128) per crossing is
    read and Z and V (24 bytes each) are written per evaluation; 8 flops per complex
    multiply-add of the plan's contraction.  Reverse pass: forward and adjoint
    contractions, and a q x q adjoint per edge written.  Exact: per prime, on pairs of residues."""
    w = _work_of(case)
    flops, nbytes = 8.0 * w["cmacs"], 32.0 * w["edges"] + 48.0 * w["evals"]
    if case["kind"] == "grad":
        nbytes += 16.0 * w["edges"] * case["q"] ** 2
    if case["kind"] == "exact":
        flops *= len(PRIMES)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ the same in plain numpy and torch

def _tait(pd):
    """Signed Tait graph of a knot diagram: (n_v, edges (u, v, eps), writhe), black being the
    colour of the region right of arc 0."""
    n = len(pd)
    parent = list(range(4 * n))

    def find(x):
        while parent[x] != x:
            parent[x] = parent[parent[x]]
            x = parent[x]
        return x

    # corner 4 i + p lies between the arms p and p + 1 (counter-clockwise) of crossing i
    side, out_arm, right0 = {}, [], None
    for i, (a, b, c, d) in enumerate(pd):
        leaves = 1 if (d + 1) % (2 * n) == b else 3   # the arm the over-strand leaves through
        out_arm.append(leaves)
        for p, arc in enumerate((a, b, c, d)):
            ccw, cw = 4 * i + p, 4 * i + (p - 1) % 4
            left, right = (ccw, cw) if p in (2, leaves) else (cw, ccw)
            if arc == 0 and p in (2, leaves):
                right0 = right
            for key, corner in (((arc, 0), left), ((arc, 1), right)):
                if key in side:
                    parent[find(corner)] = find(side[key])
                else:
                    side[key] = corner
    colour, todo = {find(right0): 1}, [find(right0)]
    regions = {}
    for i in range(n):
        for p in range(4):
            regions.setdefault(find(4 * i + p), []).append((i, p))
    while todo:
        x = todo.pop()
        for i, p in regions[x]:
            for y in (find(4 * i + (p + 1) % 4), find(4 * i + (p - 1) % 4)):
                if y not in colour:
                    colour[y] = 1 - colour[x]
                    todo.append(y)
    number = {x: k for k, x in enumerate(sorted(x for x in regions if colour[x]))}
    edges, writhe = [], 0
    for i in range(n):
        p = 0 if colour[find(4 * i)] else 1
        eps = 1 if colour[find(4 * i + out_arm[i])] else -1   # left of the leaving over-strand
        edges.append((number[find(4 * i + p)], number[find(4 * i + p + 2)], eps))
        writhe += 1 if out_arm[i] == 1 else -1
    return len(number), edges, writhe


def _order(n_v, edges):
    """(width, order): a min-fill order of the spins, best of a dozen random tie breaks."""
    best = None
    for s in range(12):
        r = np.random.RandomState(s)
        nb = [set() for _ in range(n_v)]
        for u, v, _ in edges:
            if u != v:
                nb[u].add(v)
                nb[v].add(u)
        left, order, width = set(range(n_v)), [], 0
        while left:
            def fill(x):
                l = list(nb[x])
                return sum(l[j] not in nb[l[i]] for i in range(len(l)) for j in range(i))
            few = min((fill(x), len(nb[x]), r.rand(), x) for x in left)
            x = few[3]
            width = max(width, len(nb[x]) + 1)
            for y in nb[x]:
                nb[y] |= nb[x]
                nb[y] -= {x, y}
            left.discard(x)
            order.append(x)
        if best is None or width < best[0]:
            best = (width, order)
    return best


def _einsum(factors, out):
    letter = {i: chr(97 + k) if k < 26 else chr(39 + k) for k, i in enumerate(sorted({i for f in factors for i in f[0]}))}
    return torch.einsum(",".join("".join(letter[i] for i in idx) for idx, _ in factors) + "->" +
                        "".join(letter[i] for i in out), *[t for _, t in factors])


def _log_z(n_v, edges, q, mats, order):
    """(mantissa, log of its factor): Z = sum over spins of the product of the clause matrices
    mats[e] (complex128 torch), one spin summed out after another."""
    factors, log = [], 0.0
    for (u, v, _), m in zip(edges, mats):
        factors.append(((u,), torch.diagonal(m)) if u == v else ((u, v), m))
    scalar = torch.ones((), dtype=torch.complex128)
    for x in order:
        mine = [f for f in factors if x in f[0]]
        factors = [f for f in factors if x not in f[0]]
        if not mine:
            scalar = scalar * q
            continue
        names = sorted({i for f in mine for i in f[0]} - {x})
        mine.sort(key=lambda f: f[1].dim())
        while len(mine) > 2:   # small factors first; the last two are contracted over x
            (i1, t1), (i2, t2) = mine[:2]
            idx = tuple(sorted(set(i1) | set(i2)))
            mine[:2] = [(idx, _einsum([(i1, t1), (i2, t2)], idx))]
            mine.sort(key=lambda f: f[1].dim())
        prod = _einsum(mine, names)
        top = prod.detach().abs().max()
        if top > 0:
            prod = prod / top
            log += math.log(float(top))
        if names:
            factors.append((tuple(names), prod))
        else:
            scalar = scalar * prod
    for _, t in factors:
        scalar = scalar * t
    return scalar, log


def _t(q):
    return ((q - 2) + 1j * math.sqrt(q * (4 - q))) / 2 if q < 4 else ((q - 2) + math.sqrt(q * (q - 4))) / 2 + 0j


def _reference(pd, q, grad=False, widest=6e7):
    """(Z, V) of a knot diagram in 64 bits, with grad also d log Z / dT (edges, q, q) and
    d log V / dt at fixed q; None where a factor would have more than `widest` entries."""
    n_v, edges, w = _tait(pd)
    width, order = _order(n_v, edges)
    if float(q) ** (width - 1) > widest:
        return None
    t, tau = _t(q), sum(e for _, _, e in edges)
    eye = torch.eye(q, dtype=torch.complex128)
    mats = [((1 - eye) - eye * t ** -e).requires_grad_(grad) for _, _, e in edges]
    m, log = _log_z(n_v, edges, q, mats, order)
    num = 3 * w + tau + 2 * n_v + 2
    zc = complex(m.detach())
    z = zc * math.exp(log)
    la = (num // 4) * np.log(complex(t)) - (n_v + 1) * np.log(t + 1)
    v = (-1) ** (w + n_v + 1) * zc * complex(np.exp(la + log))
    if not grad:
        return z, v
    torch.log(m).backward(torch.ones((), dtype=torch.complex128))
    d = torch.stack([x.grad.conj() for x in mats]).numpy()   # of a holomorphic function
    dv = (num // 4) / t - (n_v + 1) / (t + 1)
    dv += sum(e * t ** (-e - 1) * np.trace(d[i]) for i, (_, _, e) in enumerate(edges))
    return z, v, d, dv


def exact(case, seed):
    kind = case["kind"]
    if kind == "exact":
        return None
    pds = _diagrams(pk.Context(-1), case, seed)   # the inputs alone
    if kind in ("eval", "grad"):
        r = _reference(pds[0], case["q"], kind == "grad", 1e7 if kind == "grad" else 6e7)
        if r is None:
            return None
        out = {"v": np.array([r[1]])} | ({} if case.get("precision") == "c64" else {"z": np.array([r[0]])})
        return out | ({"dlogz": r[2], "dlogv": np.array([r[3]])} if kind == "grad" else {})
    out = {}
    for q in QS if kind == "group" else (case["q"],):
        r = None if kind == "group" and q > 3 else [_reference(pd, q) for pd in pds]
        known = r is not None and all(x is not None for x in r)
        o = {"v": np.array([x[1] for x in r]) if known else None, "z": np.array([x[0] for x in r]) if known else None}
        if case["precision"] == "c64":
            del o["z"]
        out["q%d" % q] = o
    return out if kind == "group" else out["q%d" % case["q"]]
