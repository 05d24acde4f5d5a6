"""Components by lossless links where chains and hubs are worst: a long path
with random numbering, a star around its largest vertex, many small
components with isolated vertices, hypergraph nets; and separators of rows
around the length from which a warp tests them."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1105_4490_gb300 as P
    assert torch.cuda.is_available()
    return P


@pytest.fixture(scope="module")
def O():
    import oracle
    oracle.build()
    return oracle


def _sym(n, a, b):
    return W.csr_from_coo(n, n, np.concatenate([a, b]), np.concatenate([b, a]), "sym")


def _matrices():
    rng = np.random.default_rng(0)
    n = 50000
    p = rng.permutation(n)
    yield _sym(n, p[:-1], p[1:])
    yield _sym(n, np.arange(n - 1), np.arange(1, n))
    yield _sym(n, np.full(n - 1, n - 1), np.arange(n - 1))
    a = np.arange(0, n - 7, 7)
    yield _sym(n, a, a + rng.integers(1, 7, len(a)))
    yield _sym(3, np.zeros(0, int), np.zeros(0, int))
    yield W.random_symmetric(n, 2.2, 4)


def test_components(V, O):
    for A in _matrices():
        hg, ref = V.Hypergraph.from_matrix(A), O.build_from_matrix("symmetric", A)
        assert np.array_equal(hg.components().cpu().numpy(), O.components(ref))
    R = W.random_pattern(20000, 30000, 18000, 5)
    for model in ("rownet", "colnet", "bipartite", "finegrain"):
        hg, ref = V.Hypergraph.from_matrix(R, model), O.build_from_matrix(model, R)
        assert np.array_equal(hg.components().cpu().numpy(), O.components(ref)), model


@pytest.mark.parametrize("deg", [63, 64, 65, 97, 800])
def test_separator_row_lengths(V, O, deg):
    rng = np.random.default_rng(deg)
    n = 3000
    hub = rng.choice(n, 40, replace=False)
    A = _sym(n, np.repeat(hub, deg), np.concatenate([rng.choice(n, deg, replace=False) for _ in hub]))
    x = np.zeros((n, 4), dtype=np.float32)
    x[:, :2] = rng.standard_normal((n, 2))
    hg, ref = V.Hypergraph.from_matrix(A), O.build_from_matrix("symmetric", A)
    p = V.Params(d=2, min_part=16, seed=2)
    perm, tree = hg.order_vertices(p, torch.as_tensor(x).cuda())
    want, tree_o = O.order(ref, 2, x, seed=2, min_part=16)
    assert np.array_equal(perm.cpu().numpy(), want)
    assert np.array_equal(tree["nsep"].cpu().numpy(), tree_o["nsep"])


def _chains(n):
    a = np.arange(n - 1)
    yield "ascending", _sym(n, a, a + 1)
    yield "descending", _sym(n, n - 1 - a, n - 2 - a)
    yield "comb", _sym(n, np.concatenate([a[::2], a[:-2:2]]), np.concatenate([a[::2] + 1, a[:-2:2] + 2]))
    yield "grid", _sym(n, np.concatenate([a, a[:-99]]), np.concatenate([a + 1, a[:-99] + 100]))


@pytest.mark.parametrize("model", ("symmetric", "bipartite", "rownet", "colnet", "finegrain"))
def test_components_of_chains(V, O, model):
    for name, A in _chains(20000):
        B = W.csr_from_coo(A.m, A.n, np.concatenate([np.repeat(np.arange(A.m), np.diff(A.rowptr)), np.arange(A.m)]),
                           np.concatenate([A.colidx, np.arange(A.m)]), "diag")
        hg, ref = V.Hypergraph.from_matrix(B, model), O.build_from_matrix(model, B)
        assert np.array_equal(hg.components().cpu().numpy(), O.components(ref)), name


def test_chains_take_no_longer_than_other_patterns(V):
    """A tridiagonal pattern, whose edges all link at once, costs about what a
    random one of the same size does (it took 30 times as long)."""
    n = 1_000_000
    a = np.arange(n - 1)
    d = np.arange(n)
    best = []
    for p, q in ((a, a + 1), (np.random.default_rng(1).integers(0, n, n - 1), np.random.default_rng(2).integers(0, n, n - 1))):
        A = W.csr_from_coo(n, n, np.concatenate([p, q, d]), np.concatenate([q, p, d]), "chain")
        hg = V.Hypergraph.from_matrix(A, "bipartite")
        t = []
        for _ in range(5):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            ev[0].record()
            hg.components()
            ev[1].record()
            torch.cuda.synchronize()
            t.append(ev[0].elapsed_time(ev[1]))
        best.append(min(t))
    assert best[0] < 5 * best[1], best
