"""Models of patterns with ascending rows (built without the pair sort) and of
the patterns next to them that must not take that way: every model against the
oracle for empty and full rows around the tile of 2,048 entries, thousands of
empty rows, entries on one side of the diagonal, as many left as right of it
without being symmetric, a row out of order, duplicates, no entries, no rows."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
MODELS = ("symmetric", "bipartite", "rownet", "colnet", "finegrain")


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


def _coo(m, n, rows, cols):
    return W.csr_from_coo(m, n, np.asarray(rows), np.asarray(cols), "t")


def _raw(m, n, lists):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in lists])]).astype(np.int32)
    return W.Matrix("raw", m, n, rp, np.concatenate([np.asarray(r, dtype=np.int32) for r in lists]).astype(np.int32))


def _patterns():
    rng = np.random.default_rng(3)
    yield "grid", W.grid_laplacian_3d(11)
    yield "random", W.random_symmetric(3000, 9, 1)
    n = 9000
    a, b = rng.integers(0, 40, 4000), rng.integers(0, n, 4000)
    yield "long rows", _coo(n, n, np.concatenate([a, b]), np.concatenate([b, a]))
    k = np.arange(0, 20000, 9973)
    yield "empty rows", _coo(20000, 20000, k, k[::-1])
    yield "full rows", _coo(70, 70, np.repeat(np.arange(70), 70), np.tile(np.arange(70), 70))
    yield "upper", _coo(500, 500, np.arange(499), np.arange(1, 500))
    yield "cycle", _coo(7, 7, [0, 1, 2, 2, 0], [1, 2, 0, 1, 0])       # 2 right, 2 left, (2, 0) without (0, 2)
    yield "out of order", _raw(4, 4, [[1, 0], [0, 1], [3], [2, 3]])
    yield "duplicates", _raw(4, 4, [[0, 1, 1], [0], [3, 3], [2]])
    yield "no entries", _raw(5, 5, [[], [], [], [], []])
    yield "2049", _coo(2049, 2049, np.arange(2049), np.arange(2049)[::-1])
    yield "rectangular", W.random_pattern(700, 40000, 5000, 8)
    yield "one column", _coo(3000, 1, np.arange(3000), np.zeros(3000, int))


@pytest.mark.parametrize("model", MODELS)
def test_models(V, O, model):
    for name, A in _patterns():
        if model == "symmetric" and A.m != A.n:
            continue
        hg, ref = V.Hypergraph.from_matrix(A, model), O.build_from_matrix(model, A)
        got = {k: v.cpu().numpy() for k, v in hg.arrays().items()}
        assert hg.k == ref.k and hg.nets == ref.l, name
        for f in ("net_ptr", "pins", "vtx_ptr", "vnets"):
            assert np.array_equal(got[f], getattr(ref, f)), (name, f)
        if model in ("symmetric", "bipartite"):
            assert np.array_equal(got["adj_ptr"], ref.adj_ptr) and np.array_equal(got["adj"], ref.adj), name
