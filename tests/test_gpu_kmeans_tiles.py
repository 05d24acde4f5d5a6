"""m-way k-means++ against the oracle, bit for bit, around the tiles of its
kernels: a seeding tile (2,048 points), an assignment tile (1,024), one more
than a block keeps before it flushes its 32-bit sums (8,192 of 7.5 million),
and a draw in the first, a middle and the last tile."""
import numpy as np
import pytest
import torch

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


@pytest.mark.parametrize("n,d,m,km", [(1, 3, 4, 3), (2, 2, 2, 5), (1023, 3, 5, 20), (1025, 4, 7, 20), (2047, 2, 9, 6),
                                      (2048, 3, 256, 4), (2049, 3, 33, 6), (70001, 4, 40, 5), (7700001, 2, 3, 2)])
def test_tiles(V, O, n, d, m, km):
    rng = np.random.default_rng(n + m)
    x = np.zeros((n, 4), dtype=np.float32)
    x[:, :d] = (rng.standard_normal((n, d)) * 50).astype(np.float32)
    verts = np.arange(n, dtype=np.int32)[::-1].copy()
    for seed in ((1, 2, 3) if n < 100000 else (1,)):
        lab, z, ne = V.kmeans(torch.as_tensor(x).cuda(), torch.as_tensor(verts), m, seed=seed, key=9, km_iters=km, d=d)
        lab_o, z_o, ne_o = O.kmeans(d, x, verts, m, seed=seed, key=9, km_iters=km)
        assert ne == ne_o
        assert np.array_equal(lab.cpu().numpy(), lab_o)
        assert np.array_equal(z.cpu().numpy().view(np.uint32), z_o.view(np.uint32))
