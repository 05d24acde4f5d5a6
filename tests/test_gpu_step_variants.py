"""The layout step's kernels (terms split over threads, two far-field rows in
flight, two targets per thread) against the one of one target per thread,
which the interaction count forces: the same bits, at the edges of each
kernel's range, with one, two and four lanes per target, unit and given
weights, cells of one point and of hundreds."""
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
    yield P
    P.stats_reset(False, False)


def _points(k, d, seed, share):
    rng = np.random.default_rng(seed)
    x = np.zeros((k, 4), dtype=np.float32)
    side = float(k) ** (1.0 / d)
    x[:, :d] = rng.random((k, d)) * side
    n = int(share * k)
    x[:n, :d] = 0.4 * side + 0.05 * side * rng.standard_normal((n, d))
    return torch.as_tensor(x[rng.permutation(k)]).cuda()


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("d,k", [(2, 3), (2, 512), (2, 9001), (2, 200003), (3, 2), (3, 33), (3, 511), (3, 513),
                                 (3, 4097), (3, 12160), (3, 12191), (3, 196607), (3, 196609), (4, 300), (4, 3001),
                                 (4, 9000), (4, 200001)])
def test_step_kernels_agree(V, d, k, weighted):
    A = W.random_symmetric(k, 5, seed=k)
    w = torch.randint(1, 5, (k,), generator=torch.Generator().manual_seed(k)).float() if weighted else None
    hg = V.Hypergraph.from_matrix(A, weights=w)
    for share in (0.0, 0.2):
        x = _points(k, d, k + d, share)
        out = []
        for count in (False, True):
            V.stats_reset(False, count)
            out.append([t.cpu().numpy().view(np.uint32) for t in hg.layout_step(x, 0.3, V.Params(d=d))[:2]])
        V.stats_reset(False, False)
        assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1]), (share,)


def test_step_kernels_agree_in_a_batch(V):
    """Problems of every lane count and isolated vertices in one launch."""
    mats = W.batch_mix(60, 9, nmin=300, nmax=15000)
    for d in (2, 3):
        out = []
        for count in (False, True):
            V.stats_reset(False, count)
            out.append(V.batch_layout(mats, V.Params(d=d, iters=3, seed=5))[0].cpu().numpy().view(np.uint32))
        V.stats_reset(False, False)
        assert np.array_equal(out[0], out[1])
