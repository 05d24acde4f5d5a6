"""2-means of a node by one cluster against the oracle, bit for bit, at the
sizes where its shape changes: one block of 128, 512 and 1,024 threads,
clusters of 2 to 16 blocks with uneven shares, points streamed instead of held
in shared memory, the largest node a cluster takes and the launch sequence
above it; no, one and 20 rounds; coincident points; nodes of very uneven size
in one launch."""
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


def _check(V, O, hg, x, verts, d, km, seed):
    from paper_1105_4490_gb300 import vmo
    ok_o, lab_o, z1_o, z2_o = O.bisect(d, x, verts, seed=seed, key=5, km_iters=km)
    runs = [hg.bisect(torch.as_tensor(x).cuda(), torch.as_tensor(verts), seed=seed, key=5, km_iters=km, d=d)]
    if len(verts) <= 131072:
        runs.append(vmo.bisect_noalloc(torch.as_tensor(x).cuda(), torch.as_tensor(verts), seed=seed, key=5,
                                       km_iters=km, d=d))
    for ok, lab, z1, z2 in runs:
        assert ok == bool(ok_o)
        assert np.array_equal(lab.cpu().numpy(), lab_o)
        assert np.array_equal(z1.cpu().numpy()[:d], np.asarray(z1_o, dtype=np.float32)[:d])
        if ok:
            assert np.array_equal(z2.cpu().numpy()[:d], np.asarray(z2_o, dtype=np.float32)[:d])


@pytest.mark.parametrize("d", [2, 3, 4])
@pytest.mark.parametrize("n", [2, 3, 127, 129, 512, 513, 2049, 4096, 4097, 8193, 33001, 65537, 290001])
def test_node_sizes(V, O, d, n):
    hg = V.Hypergraph.from_matrix(W.grid_laplacian_2d(4))
    rng = np.random.default_rng(n + d)
    x = np.zeros((n + 5, 4), dtype=np.float32)
    x[:, :d] = rng.standard_normal((n + 5, d)) * 37.0
    verts = rng.permutation(n + 5)[:n].astype(np.int32)
    for km in (0, 1, 20):
        _check(V, O, hg, x, verts, d, km, seed=n)


@pytest.mark.parametrize("n", [1802111, 1802113])
def test_largest_node(V, O, n):
    hg = V.Hypergraph.from_matrix(W.grid_laplacian_2d(4))
    x = np.zeros((n, 4), dtype=np.float32)
    x[:, :2] = np.random.default_rng(n).standard_normal((n, 2)) * 300.0
    _check(V, O, hg, x, np.arange(n, dtype=np.int32), 2, 3, seed=3)


@pytest.mark.parametrize("d,n", [(3, 1600000), (3, 1600001), (4, 1250000), (4, 1250001)])
def test_largest_node_of_more_dimensions(V, O, d, n):
    hg = V.Hypergraph.from_matrix(W.grid_laplacian_2d(4))
    x = np.zeros((n, 4), dtype=np.float32)
    x[:, :d] = np.random.default_rng(n).standard_normal((n, d)) * 300.0
    _check(V, O, hg, x, np.arange(n, dtype=np.int32), d, 3, seed=3)


def test_coincident_points(V, O):
    hg = V.Hypergraph.from_matrix(W.grid_laplacian_2d(4))
    for n in (2, 700, 20000):
        x = np.ones((n, 4), dtype=np.float32)
        x[:, 3] = 0.0
        _check(V, O, hg, x, np.arange(n, dtype=np.int32), 3, 20, seed=1)
        x[n - 1, 0] = 2.0
        _check(V, O, hg, x, np.arange(n, dtype=np.int32), 3, 20, seed=1)


def test_uneven_nodes(V, O):
    """Matrices of 3 to 40,000 rows in one ordering of given coordinates."""
    mats = [W.random_symmetric(n, 4, n) for n in (40000, 3, 130, 66, 9000, 700, 2500)] + \
        [W.grid_laplacian_2d(9) for _ in range(300)]
    rng = np.random.default_rng(2)
    xs = [np.zeros((A.m, 4), dtype=np.float32) for A in mats]
    for x in xs:
        x[:, :3] = rng.standard_normal((len(x), 3)) * 10
    p = V.Params(d=3, min_part=8, seed=6)
    perm, offs = V.batch_order(mats, p, coords=torch.as_tensor(np.concatenate(xs)).cuda())
    perm = perm.cpu().numpy()
    for i in (0, 1, 2, 4, 6, 11, 306):
        ref = O.build_from_matrix("symmetric", mats[i])
        want, _ = O.order(ref, 3, xs[i], seed=6, min_part=8)
        assert np.array_equal(perm[offs[i]:offs[i + 1]], want), i


@pytest.mark.parametrize("d", [2, 3, 4])
def test_large_nodes_among_many(V, O, d):
    """Levels of more than 512 nodes with a few of more than 16,384 points, which
    have a launch of their own."""
    mats = [W.random_symmetric(n, 4, n) for n in (70000, 16384, 16385, 40000)] + \
        [W.random_symmetric(70 + i % 9, 4, i) for i in range(540)]
    rng = np.random.default_rng(d)
    xs = [np.zeros((A.m, 4), dtype=np.float32) for A in mats]
    for x in xs:
        x[:, :d] = rng.standard_normal((len(x), d)) * 10
    perm, offs = V.batch_order(mats, V.Params(d=d, min_part=60, max_depth=3, seed=6),
                               coords=torch.as_tensor(np.concatenate(xs)).cuda())
    perm = perm.cpu().numpy()
    for i in (0, 1, 2, 3, 4, 100, 543):
        ref = O.build_from_matrix("symmetric", mats[i])
        want, _ = O.order(ref, d, xs[i], seed=6, min_part=60, max_depth=3)
        assert np.array_equal(perm[offs[i]:offs[i + 1]], want), i
