"""The work that a user of this framework has it do, as cases to be timed.

A sparse matrix comes in as a CSR pattern on the GPU; the framework builds its
hypergraph model, lays the model out in R^d (multilevel steepest descent),
bisects the coordinates recursively and returns permutations.  The cases are
that whole path at its smallest and its batched form, the layout at the sizes
of the benchmark, and each part through its own entry point: one layout step,
the recursive ordering of given coordinates, the ordering with a strengthened
diagonal, the model's construction and the m-way k-means++.

Sizes are those of workloads.CONFIGS, of the benchmark's legs and of the tests.
Patterns and coordinates are made on the GPU from the seed (torch's generator)
with the degree structure of workloads: stencils, power-law and uniform random
patterns.
"""
from __future__ import annotations

import math

import torch

import paper_1105_4490_gb300 as V

DEV = "cuda"
U64 = (1 << 64) - 1


# ------------------------------- patterns -----------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _csr(m, n, rows, cols):
    """CSR (int32, ascending distinct columns) of the entries (rows, cols)."""
    key = torch.unique(rows.long() * n + cols.long())
    r = key // n
    ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.bincount(r, minlength=m), 0)
    return ptr.int(), (key - r * n).int()


def _grid(side, d, reach):
    """Stencil on a side^d grid: the 2d + 1 points of the Laplacian (reach
    "star") or the full 3^d box ("box")."""
    k = side ** d
    v = torch.arange(k, device=DEV)
    c = [(v // side ** m) % side for m in range(d)]
    rows, cols = [], []
    for o in range(3 ** d):
        off = [(o // 3 ** m) % 3 - 1 for m in range(d)]
        if reach == "star" and sum(abs(t) for t in off) > 1:
            continue
        ok = torch.ones(k, dtype=torch.bool, device=DEV)
        for m in range(d):
            ok &= (c[m] + off[m] >= 0) & (c[m] + off[m] < side)
        r = v[ok]
        rows.append(r)
        cols.append(r + sum(off[m] * side ** m for m in range(d)))
    return (k, k) + _csr(k, k, torch.cat(rows), torch.cat(cols))


def _powerlaw_degrees(n, dmin, gen):
    """Degrees with P(d) ~ d^-2.5 on [dmin, 2000]."""
    sup = torch.arange(dmin, 2001, dtype=torch.float64, device=DEV)
    cdf = torch.cumsum(sup ** -2.5, 0)
    u = torch.rand(n, generator=gen, device=DEV, dtype=torch.float64) * cdf[-1]
    return (dmin + torch.searchsorted(cdf, u)).clamp(max=2000)


def _powerlaw(n, gen):
    """Symmetric pattern with power-law degrees (mean about 11), full diagonal."""
    cw = torch.cumsum(_powerlaw_degrees(n, 4, gen).double(), 0)
    e = int(float(cw[-1]) / 2)
    a, b = (torch.searchsorted(cw, torch.rand(e, generator=gen, device=DEV, dtype=torch.float64) * cw[-1])
            .clamp(max=n - 1) for _ in range(2))
    keep = a != b
    a, b, i = a[keep], b[keep], torch.arange(n, device=DEV)
    return (n, n) + _csr(n, n, torch.cat([a, b, i]), torch.cat([b, a, i]))


def _rect(m, n, gen):
    """m x n pattern with power-law column degrees (mean about 16)."""
    deg = _powerlaw_degrees(n, 6, gen)
    cols = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    return (m, n) + _csr(m, n, torch.randint(0, m, (cols.numel(),), generator=gen, device=DEV), cols)


def _random_symmetric(n, per_row, gen):
    e = int(n * (per_row - 1.0) / 2)
    a, b = (torch.randint(0, n, (e,), generator=gen, device=DEV) for _ in range(2))
    keep = a != b
    a, b, i = a[keep], b[keep], torch.arange(n, device=DEV)
    return (n, n) + _csr(n, n, torch.cat([a, b, i]), torch.cat([b, a, i]))


def _pattern(case, gen):
    """(m, n, rowptr, colidx) of the case's matrix."""
    p, n = case["pattern"], case["n"]
    if p == "grid2d":
        return _grid(n, 2, "star")
    if p == "grid3d":
        return _grid(n, 3, "star")
    if p == "stencil27":
        return _grid(n, 3, "box")
    if p == "powerlaw":
        return _powerlaw(n, gen)
    if p == "random":
        return _random_symmetric(n, case["per_row"], gen)
    return _rect(n, n * 3 // 4, gen)


def _renumbered(m, n, ptr, col, gen):
    """The same matrix with its rows and columns in another order (a square
    pattern's alike), as meshes and graphs come from their generators."""
    rows = torch.repeat_interleave(torch.arange(m, device=DEV), (ptr[1:] - ptr[:-1]).long())
    p = torch.randperm(m, generator=gen, device=DEV)
    q = p if m == n else torch.randperm(n, generator=gen, device=DEV)
    return (m, n) + _csr(m, n, p[rows], q[col.long()])


def _coords(case, k, gen):
    """Coordinates as a layout leaves them (mean point spacing about 1): a
    jittered grid for a stencil, a cloud that is dense in the middle for the
    irregular patterns; float32 [k, 4], components from d on zero."""
    d = case["d"]
    x = torch.zeros((k, 4), dtype=torch.float32, device=DEV)
    if case["pattern"] in ("grid2d", "grid3d"):
        side, gd = case["n"], 2 if case["pattern"] == "grid2d" else 3
        v = torch.arange(k, device=DEV)
        for m in range(min(gd, d)):
            x[:, m] = ((v // side ** m) % side).float()
        x[:, :d] += 0.4 * (torch.rand((k, d), generator=gen, device=DEV) - 0.5)
    else:
        x[:, :d] = torch.randn((k, d), generator=gen, device=DEV) * (0.25 * k ** (1.0 / d))
    return x


# --------------------------------- cases ------------------------------------
def listed():
    return [
        # The smallest job: build, lay out and order a 64 x 64 grid (the
        # smallest configuration).  Launches and their latency decide.
        dict(name="whole_grid2d_64", kind="whole", pattern="grid2d", n=64, d=2, min_part=64, max_depth=62),
        # The layout of a regular mesh and of an irregular matrix with hub
        # rows at the sizes of the medium configuration: nearly all of the
        # time of an ordering from scratch.
        dict(name="layout_grid3d_64", kind="layout", pattern="grid3d", n=64, d=3),
        dict(name="layout_powerlaw_500k", kind="layout", pattern="powerlaw", n=500_000, d=3),
        # Many matrices of uneven size in one call (the batch configuration's mix).
        dict(name="batch_256", kind="batch", count=256, nmin=200, nmax=20000, d=3),
        # One step of steepest descent: binning, attraction, repulsion and
        # update, at the smallest and at the medium size.
        dict(name="step_grid2d_64", kind="step", pattern="grid2d", n=64, d=2, weighted=False),
        dict(name="step_powerlaw_500k", kind="step", pattern="powerlaw", n=500_000, d=3, weighted=False),
        # Recursive bisection of given coordinates: a user who keeps a layout
        # and orders it (BBD to depth 10; SBD of a rectangular matrix to 64 parts).
        dict(name="order_grid3d_64", kind="order", pattern="grid3d", n=64, d=3, model="symmetric", sbd=False,
             min_part=64, max_depth=10, sep_recursion=0, cut_order=0),
        dict(name="order_sbd_rect_400k", kind="order", pattern="rect", n=400_000, d=2, model="bipartite", sbd=True,
             min_part=1, max_depth=6, sep_recursion=0, cut_order=0),
        # Unsymmetric matrix with a strengthened diagonal (ordering before an
        # LU factorisation), rows and matched columns kept together.
        dict(name="matched_mesh_200", kind="matched", pattern="grid2d", n=200, d=2, min_part=64),
        # The model of a matrix: a 27-point mesh of a million nodes (the
        # largest requests that are served) and the bipartite model of the
        # rectangular matrix.
        dict(name="build_stencil27_100", kind="build", pattern="stencil27", n=100, model="symmetric"),
        dict(name="build_rect_400k", kind="build", pattern="rect", n=400_000, model="bipartite"),
        # One-shot 64-way partition of a million points.
        dict(name="kmeans_1m_64", kind="kmeans", n=1_000_000, m=64, d=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["whole", "layout", "batch", "step", "order", "order", "matched", "build", "build", "kmeans"])
    if kind == "whole":
        if rng.random() < 0.5:
            return dict(kind=kind, pattern="grid2d", n=_log(rng, 14, 140), d=2, min_part=rng.choice([16, 64]),
                        max_depth=62)
        return dict(kind=kind, pattern="random", n=_log(rng, 200, 20000), per_row=round(rng.uniform(3, 30), 2),
                    d=rng.choice([2, 3]), min_part=rng.choice([16, 64]), max_depth=62)
    if kind == "batch":
        return dict(kind=kind, count=_log(rng, 8, 256), nmin=200, nmax=20000, d=rng.choice([2, 3]))
    if kind == "kmeans":
        return dict(kind=kind, n=_log(rng, 3000, 1_000_000), m=_log(rng, 2, 256), d=rng.choice([2, 3, 4]))
    if kind == "matched":
        return dict(kind=kind, pattern="grid2d", n=_log(rng, 20, 200), d=rng.choice([2, 3]),
                    min_part=rng.choice([16, 64]))
    if kind == "build":
        pat = rng.choice(["stencil27", "powerlaw", "rect"])
        n = _log(rng, 12, 100) if pat == "stencil27" else _log(rng, 5000, 500_000 if pat == "powerlaw" else 400_000)
        models = ["bipartite", "rownet", "colnet", "finegrain"] + (["symmetric"] if pat != "rect" else [])
        return dict(kind=kind, pattern=pat, n=n, model=rng.choice(models))
    pat = rng.choice(["grid2d", "grid3d", "powerlaw", "rect"])
    n = {"grid2d": _log(rng, 40, 500), "grid3d": _log(rng, 12, 64), "powerlaw": _log(rng, 5000, 500_000),
         "rect": _log(rng, 3000, 400_000)}[pat]
    d = {"grid2d": 2, "grid3d": 3, "rect": 2}.get(pat) or rng.choice([2, 3, 4])
    if kind == "layout":
        return dict(kind=kind, pattern=pat, n=n, d=min(d, 3))
    if kind == "step":
        return dict(kind=kind, pattern=pat, n=n, d=d, weighted=rng.random() < 0.5)
    sep = rng.choice([0, 0, 1])
    return dict(kind="order", pattern=pat, n=n, d=d, model="bipartite" if pat == "rect" else "symmetric",
                sbd=rng.random() < 0.5, min_part=rng.choice([1, 16, 64]), max_depth=rng.choice([6, 10, 62]),
                sep_recursion=sep, cut_order=0 if sep else rng.choice([0, 0, 2]))


# -------------------------------- inputs ------------------------------------
def _inputs(case, seed):
    """Everything of a case that comes from the seed, as plain tensors."""
    gen, kind = _gen(seed), case["kind"]
    if kind == "kmeans":
        n, d = case["n"], case["d"]
        x = torch.zeros((n, 4), dtype=torch.float32, device=DEV)
        x[:, :d] = torch.randn((n, d), generator=gen, device=DEV) * (0.25 * n ** (1.0 / d))
        return dict(x=x, verts=torch.randperm(n, generator=gen, device=DEV).int())
    if kind == "batch":
        rate = (3 + 27 * torch.rand(case["count"], generator=gen, device=DEV, dtype=torch.float64)).tolist()
        mats = []
        for i, r in enumerate(rate):
            t = (0.5 + i * 0.6180339887498949) % 1.0  # sizes spread evenly over their logarithm
            n = int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** t))
            m, _, ptr, col = _grid(max(2, round(math.sqrt(n))), 2, "star") if i % 2 == 0 \
                else _random_symmetric(n, r, gen)
            mats.append((ptr, col, m))
        return dict(mats=mats)
    if kind == "matched":
        m, _, ptr, col = _pattern(case, gen)
        rows = torch.repeat_interleave(torch.arange(m, device=DEV), (ptr[1:] - ptr[:-1]).long())
        keep = (rows == col) | (torch.rand(rows.numel(), generator=gen, device=DEV) < 0.7)
        pi = torch.randperm(m, generator=gen, device=DEV)
        ptr, col = _csr(m, m, rows[keep], pi[col[keep].long()])
        x = _coords(case, m, gen)
        y = x.clone()
        y[:, :case["d"]] += 0.2 * (torch.rand((m, case["d"]), generator=gen, device=DEV) - 0.5)
        both = torch.empty((2 * m, 4), dtype=torch.float32, device=DEV)
        both[:m] = x
        both[m + pi] = y  # column pi[i] beside row i
        return dict(m=m, n=m, ptr=ptr, col=col, match=pi.int(), x=both)
    if kind == "build":  # one matrix of the size, in another numbering for every seed
        m, n, ptr, col = _renumbered(*_pattern(case, _gen(0)), gen)
    else:
        m, n, ptr, col = _pattern(case, gen)
    got = dict(m=m, n=n, ptr=ptr, col=col)
    if kind in ("step", "order"):
        k = m + n if case["pattern"] == "rect" else m
        got["x"] = _coords(case, k, gen)
        if case.get("weighted"):
            got["w"] = torch.randint(1, 9, (k,), generator=gen, device=DEV).float()
    return got


def _params(case, seed):
    return V.Params(d=case["d"], seed=int(seed) % (1 << 31) + 1,
                    **{f: case[f] for f in ("min_part", "max_depth", "sep_recursion", "cut_order") if f in case})


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"], kind = case, case["kind"]
    if kind not in ("build", "kmeans"):
        s["params"] = _params(case, seed)
    if kind == "kmeans":
        s["seed"] = int(seed) + 77
    if kind in ("layout", "step", "order", "matched"):
        model = "bipartite" if case["pattern"] == "rect" or kind == "matched" else "symmetric"
        s["hg"] = V.Hypergraph(s["ptr"], s["col"], s["m"], s["n"], model, s.get("w"))
    return s


def _tree(tree, k):
    """The tree's records, with zeros up to the most that k vertices can have."""
    cap = 2 * k + 16
    ints = torch.stack([tree[f] for f in ("offset", "n1", "n2", "nsep", "depth", "comp")])
    return [torch.nn.functional.pad(t, (0, cap - t.shape[-1])) for t in (tree["heap"], ints)]


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "whole":
        hg = V.Hypergraph(s["ptr"], s["col"], s["m"], s["n"], "symmetric")
        x = hg.layout(s["params"])
        rp, cp, tree = hg.order(s["params"], coords=x)
        return dict(x=x, rows=rp, cols=cp, tree=_tree(tree, hg.k))
    if kind == "layout":
        return s["hg"].layout(s["params"])
    if kind == "batch":
        x, _ = V.batch_layout(s["mats"], s["params"])
        perm, _ = V.batch_order(s["mats"], s["params"], coords=x)
        return dict(x=x, perm=perm)
    if kind == "step":
        x, y, keys, _ = s["hg"].layout_step(s["x"], 1.0, s["params"])
        return dict(x=x, y=y, keys=keys)
    if kind == "order":
        rp, cp, tree = s["hg"].order(s["params"], coords=s["x"], sbd=case["sbd"])
        return dict(rows=rp, cols=cp, tree=_tree(tree, s["hg"].k))
    if kind == "matched":
        rp, cp, vp, tree = s["hg"].order_matched(s["match"], s["params"], coords=s["x"])
        return dict(rows=rp, cols=cp, verts=vp, tree=_tree(tree, s["hg"].k))
    if kind == "build":
        return V.Hypergraph(s["ptr"], s["col"], s["m"], s["n"], case["model"]).arrays()
    labels, centres, nonempty = V.kmeans(s["x"], s["verts"], case["m"], s["seed"], d=case["d"])
    return dict(labels=labels, centres=centres, nonempty=nonempty)


# ---------------------------------- work ------------------------------------
# Sources that act on a point in one step: the points of its own and the
# adjacent cells (3^d cells of about 4 points) and, on each of the grid's
# levels but the two coarsest, the cells that are adjacent to its parent's
# cell and not to its own; about 18 operations each for d = 3.
_OPS = {2: 10, 3: 18, 4: 23}


def _levels(k, d):
    L = 1
    while L < {2: 15, 3: 10, 4: 7}[d] and 8 * 2 ** (d * L) < k:
        L += 1
    return L


def _step_flops(k, d):
    sources = min(k, 4 * 3 ** d) + max(0, _levels(k, d) - 1) * 0.6 * (6 ** d - 3 ** d)
    return k * min(k, sources) * _OPS[d]


def _size(case):
    """About (vertices, entries) of the case's matrix, or all of them together."""
    if case["kind"] == "batch":
        mean = (case["nmax"] - case["nmin"]) / math.log(case["nmax"] / case["nmin"])
        return int(case["count"] * mean), int(case["count"] * mean * 10.5)
    p, n = case["pattern"], case["n"]
    k, per = {"grid2d": (n * n, 5), "grid3d": (n ** 3, 7), "stencil27": (n ** 3, 26.5), "powerlaw": (n, 11),
              "random": (n, case.get("per_row")), "rect": (n + n * 3 // 4, 6.7)}[p]
    if case["kind"] == "matched":
        return 2 * k, int(k * 3.8)
    return k, int(k * per)


def work(case):
    kind = case["kind"]
    if kind == "kmeans":
        n, m, d = case["n"], case["m"], case["d"]
        # seeding: a distance to every centre; 20 rounds and the labels: the same
        return dict(bytes=24 * n + 16 * m, flops=float(n) * m * (3 * d) * 22)
    k, nnz = _size(case)
    csr = 4 * nnz + 4 * k
    if kind == "build":
        graph = case["model"] in ("symmetric", "bipartite")
        # graph models: adjacency, nets of two pins, incidence; else pins and incidence
        return dict(bytes=csr + (4 * nnz * (2 if graph else 1) * 3.5 + 12 * k), flops=0)
    d = case["d"]
    if kind == "step":
        return dict(bytes=csr + 16 * k * 3 + 4 * k, flops=_step_flops(k, d) + nnz * 8)
    depth = min(case.get("max_depth", 62), max(1, math.ceil(math.log2(max(2, k / max(1, case.get("min_part", 64)))))))
    order = float(k) * depth * 20 * 7 * d  # 20 rounds of two distances and the sums on each level
    if kind in ("order", "matched"):
        return dict(bytes=csr + 16 * k + 8 * k, flops=order)
    # 100 steps on every level of the hierarchy, about half as many vertices on each
    steps, kk = 0.0, float(k if kind != "batch" else k / case["count"])
    while kk > 64:
        steps += _step_flops(kk, d) * 100
        kk /= 1.8
    steps *= case["count"] if kind == "batch" else 1
    return dict(bytes=csr + 16 * k + (8 * k if kind != "layout" else 0), flops=steps + (order if kind != "layout" else 0))


# ---------------------------------- exact -----------------------------------
def _exact_step(case, seed):
    """One step in 64 bits: the grid and its cells from the 32-bit coordinates
    (they decide which sources are points and which are cells), then pulls,
    pushes and the update in double precision."""
    s = _inputs(case, seed)
    d, x32 = case["d"], s["x"]
    k = x32.shape[0]
    L = _levels(k, d)
    c = x32[:, :d]
    lo = c.amin(0)
    scale = torch.tensor(float(1 << L), device=DEV) / (c.amax(0) - lo).max()
    cell = torch.floor((c - lo) * scale).long().clamp(max=(1 << L) - 1)
    x = c.double()
    w = s["w"].double() if "w" in s else torch.ones(k, dtype=torch.float64, device=DEV)
    F = torch.zeros((k, d), dtype=torch.float64, device=DEV)

    def index(q, side):
        r = q[:, d - 1]
        for m in range(d - 2, -1, -1):
            r = r * side + q[:, m]
        return r

    def push(t, src, ws):  # F[t] += w r^-d (src - x[t]), each t once
        dx = src - x[t]
        r2 = (dx * dx).sum(1)
        g = torch.where(r2 > 0, ws * r2.clamp(min=1e-300) ** (-0.5 * d), torch.zeros_like(r2))
        F[t] += g[:, None] * dx

    # near field: every point of the 3^d cells around the point's own
    side = 1 << L
    key = index(cell, side)
    order = torch.argsort(key)
    cnt = torch.bincount(key, minlength=side ** d)
    first = torch.cumsum(cnt, 0) - cnt
    for o in range(3 ** d):
        q = cell + torch.tensor([(o // 3 ** m) % 3 - 1 for m in range(d)], device=DEV)
        t = torch.nonzero(((q >= 0) & (q < side)).all(1)).squeeze(1)
        b = index(q[t], side)
        a, n = first[b], cnt[b]
        j = 0
        while True:
            t, a, n = t[n > j], a[n > j], n[n > j]
            if t.numel() == 0:
                break
            u = order[a + j]
            push(t, x[u], w[u])
            j += 1
    # far field: on every level from 2 on the children of the cells around the
    # parent's, but not the cells around the point's own
    every = torch.arange(k, device=DEV)
    for l in range(2, L + 1):
        sl = 1 << l
        me = cell >> (L - l)
        mine = index(me, sl)
        W = torch.zeros(sl ** d, dtype=torch.float64, device=DEV).index_add_(0, mine, w)
        S = torch.zeros((sl ** d, d), dtype=torch.float64, device=DEV).index_add_(0, mine, x * w[:, None])
        Z = S / W.clamp(min=1e-300)[:, None]
        for o in range(6 ** d):
            q = 2 * (me >> 1) - 2 + torch.tensor([(o // 6 ** m) % 6 for m in range(d)], device=DEV)
            ok = ((q >= 0) & (q < sl)).all(1) & ((q - me).abs() > 1).any(1)
            t = every[ok]
            b = index(q[t], sl)
            keep = W[b] > 0
            push(t[keep], Z[b[keep]], W[b[keep]])
    # pulls of the adjacency (off-diagonal pairs), half of each difference
    rows = torch.repeat_interleave(torch.arange(s["m"], device=DEV), (s["ptr"][1:] - s["ptr"][:-1]).long())
    cols = s["col"].long() + (s["m"] if case["pattern"] == "rect" else 0)
    if case["pattern"] == "rect":
        rows, cols = torch.cat([rows, cols]), torch.cat([cols, rows])
    y = F * (1.0 if d == 2 else d - 2.0) * w[:, None]
    y.index_add_(0, rows, 0.5 * (x[rows] - x[cols]))
    out = [torch.zeros((k, 4), dtype=torch.float64, device=DEV) for _ in range(2)]
    out[0][:, :d] = x - y / y.norm(dim=1, keepdim=True).clamp(min=1e-300)
    out[1][:, :d] = y
    return dict(x=out[0], y=out[1], keys=None)


def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & U64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & U64
    return z ^ (z >> 31)


def _rand(seed, a, b):
    G = 0x9E3779B97F4A7C15
    return _mix((_mix((seed + G * (a + 1)) & U64) + G * (b + 1)) & U64)


def _exact_kmeans(case, seed):
    """Centres as the means of their points in 64 bits; the draws, distances
    and labels are 32-bit decisions and are taken as such."""
    s = _inputs(case, seed)
    m, d = case["m"], case["d"]
    p = s["x"][s["verts"].long()]
    n = p.shape[0]
    tag = (int(seed) + 77) ^ 0x6B6D65616E730000
    e = math.frexp(float(p[:, :d].abs().max()))[1]
    scale = torch.tensor(2.0 ** (34 - 2 * e), device=DEV)

    def dist(z):
        q = p[:, 0] - z[0]
        r = q * q
        for c in range(1, d):
            q = p[:, c] - z[c]
            r = r + q * q
        return r

    z = [p[(n * _rand(tag, 1, 0)) >> 64].clone()]
    dm = None
    for c in range(1, m):
        dd = dist(z[-1])
        dm = dd if dm is None else torch.minimum(dm, dd)
        pre = torch.cumsum(torch.floor(dm * scale).long(), 0)
        total = int(pre[-1])
        if total == 0:
            break
        z.append(p[int(torch.searchsorted(pre, (total * _rand(tag, 1, c)) >> 64, right=True))].clone())
    z = torch.stack(z + [z[0]] * (m - len(z)))
    mean, last = z.double(), None
    for _ in range(20):
        best, lab = dist(z[0]), torch.zeros(n, dtype=torch.int64, device=DEV)
        for j in range(1, m):
            dj = dist(z[j])
            near = dj < best
            best, lab = torch.where(near, dj, best), torch.where(near, j, lab)
        if last is not None and torch.equal(lab, last):
            break
        last = lab
        cnt = torch.bincount(lab, minlength=m)
        S = torch.zeros((m, 4), dtype=torch.float64, device=DEV).index_add_(0, lab, p.double())
        mean = torch.where((cnt > 0)[:, None], S / cnt.clamp(min=1)[:, None], mean)
        z = mean.float()
    return dict(labels=None, centres=mean, nonempty=None)


def exact(case, seed):
    if case["kind"] == "step":
        return _exact_step(case, seed)
    if case["kind"] == "kmeans":
        return _exact_kmeans(case, seed)
    # a layout of hundreds of steps has no such value (a rounding moves points
    # into other cells); the other outputs are whole numbers
    return None
