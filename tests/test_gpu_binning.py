"""Device-wide binning of a layout step (cell counts, scan, vertex order within
the cell, cell sums by bricks) at the sizes where it can go wrong: grids of
fewer levels than a brick, one and several levels above the bricks, tables of
one scan tile, of several and of more than one cluster takes, cells of one
point, of just over the serial limit and of thousands, and, with all points in
one problem of at most 2,048 vertices, the same bits as the one-block binning."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-4  # normwise, the stated tolerance of one layout step


@pytest.fixture(scope="module")
def V():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1105_4490_gb300 as P
    assert torch.cuda.is_available()
    t0 = P.get_tuning()
    yield P
    P.set_tuning(**t0)


@pytest.fixture(scope="module")
def O():
    import oracle
    oracle.build()
    return oracle


def _clustered(k, d, seed, share):
    """`share` of the points in three tight clusters, the others uniform."""
    rng = np.random.default_rng(seed)
    x = np.zeros((k, 4), dtype=np.float32)
    side = float(k) ** (1.0 / d)
    x[:, :d] = rng.random((k, d)) * side
    n = int(share * k)
    x[:n, :d] = side * (0.2 + 0.3 * rng.integers(0, 3, n)[:, None]) + 0.02 * side * rng.standard_normal((n, d))
    return x[rng.permutation(k)]


@pytest.mark.parametrize("d,k,occ,share", [
    (2, 3, 8, 0.0), (2, 33, 8, 0.0), (2, 2049, 8, 0.3), (2, 9000, 1, 0.5),
    (3, 17, 8, 0.0), (3, 65, 8, 0.0), (3, 2600, 8, 0.9), (3, 30000, 8, 0.2), (3, 40000, 1, 0.1),
    (4, 40, 8, 0.0), (4, 5000, 8, 0.5), (4, 70000, 1, 0.02)])
def test_device_wide_binning(V, O, d, k, occ, share):
    A = W.random_symmetric(k, 6, seed=k)
    hg, ref = V.Hypergraph.from_matrix(A), O.build_from_matrix("symmetric", A)
    x = _clustered(k, d, k + d, share)
    p = V.Params(d=d, occupancy=occ)
    V.set_tuning(19456, 10, 4, 0)
    xg, yg, kg, L = hg.layout_step(torch.as_tensor(x).cuda(), 0.25, p)
    xo, yo, ko, Lo = O.layout_step(ref, d, x.astype(np.float64), 0.25, occ=occ)
    assert L == Lo
    assert np.array_equal(kg.cpu().numpy().view(np.uint32), ko)
    yg = yg.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(yg[:, :d] - yo[:, :d]) <= TOL * np.linalg.norm(yo[:, :d])
    if k <= 2048:
        V.set_tuning(19456, 10, 4, 2048)
        xs, ys, ks, _ = hg.layout_step(torch.as_tensor(x).cuda(), 0.25, p)
        assert np.array_equal(ys.cpu().numpy().view(np.uint32), yg.astype(np.float32).view(np.uint32))
        assert np.array_equal(xs.cpu().numpy(), xg.cpu().numpy()) and np.array_equal(ks.cpu().numpy(), kg.cpu().numpy())


def test_device_wide_binning_many_problems(V):
    """A batch of matrices with isolated vertices: the two binnings agree."""
    mats = W.batch_mix(12, 5, nmin=200, nmax=1800)
    for d in (2, 3):
        out = []
        for small in (0, 2048):
            V.set_tuning(19456, 10, 4, small)
            out.append(V.batch_layout(mats, V.Params(d=d, iters=9, seed=4))[0].cpu().numpy())
        assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))


@pytest.mark.parametrize("d,k,sizes", [
    (2, 2100, (65, 64)), (2, 3000, (1024, 1025)), (2, 4096, (4096,)), (2, 4095, (2000, 2000)), (2, 4097, (4097,)),
    (2, 9000, (1025, 1100, 4000)), (3, 5000, (2500, 2499)), (3, 2049, (1025,)), (4, 6000, (3000, 1024))])
def test_crowded_cells(V, O, d, k, sizes):
    """Cells of hundreds and thousands of points, side by side in the sorted order:
    the vertex order within them shows in the bits of the sums, so the step is
    compared with the oracle's and, where a problem fits one block, with that
    binning bit by bit."""
    A = W.random_symmetric(k, 6, seed=k)
    hg, ref = V.Hypergraph.from_matrix(A), O.build_from_matrix("symmetric", A)
    rng = np.random.default_rng(k + d)
    side = float(k) ** (1.0 / d)
    x = np.zeros((k, 4), dtype=np.float32)
    x[:, :d] = rng.random((k, d)) * side
    n = 0
    for i, size in enumerate(sizes):
        x[n:n + size, :d] = side * (0.3 + 0.2 * i) + 1e-3 * rng.standard_normal((size, d))
        n += size
    x = x[rng.permutation(k)]
    p = V.Params(d=d)
    V.set_tuning(19456, 10, 4, 0)
    xg, yg, kg, L = hg.layout_step(torch.as_tensor(x).cuda(), 0.25, p)
    xo, yo, ko, Lo = O.layout_step(ref, d, x.astype(np.float64), 0.25)
    assert L == Lo and np.array_equal(kg.cpu().numpy().view(np.uint32), ko)
    yn = yg.cpu().numpy().astype(np.float64)
    # (TOL is for clouds about their own width from the origin; where the cloud is the
    # cluster itself, 1e-3 wide at 20, single-precision cell centres alone are 1e-3 off)
    if sum(sizes) < k:
        assert np.linalg.norm(yn[:, :d] - yo[:, :d]) <= TOL * np.linalg.norm(yo[:, :d])
    V.set_tuning(19456, 10, 4, 2048)
    xs, ys, ks, _ = hg.layout_step(torch.as_tensor(x).cuda(), 0.25, p)
    assert torch.equal(ys.view(torch.int32), yg.view(torch.int32))
    assert torch.equal(xs.view(torch.int32), xg.view(torch.int32)) and torch.equal(ks, kg)


@pytest.mark.parametrize("d,k,sizes", [(2, 1025, (64, 65)), (2, 2048, (2048,)), (2, 2000, (1000, 66, 900)),
                                       (3, 2048, (1200, 700)), (3, 1500, (1024, 65)), (4, 2000, (1999,))])
def test_crowded_cells_of_one_block(V, d, k, sizes):
    """Problems of 1,025 to 2,048 points, whose crowded cells one block sorts by
    bits: steps from the crowded cloud and a few after it, as device-wide."""
    hg = V.Hypergraph.from_matrix(W.random_symmetric(k, 6, seed=k))
    rng = np.random.default_rng(k + d)
    side = float(k) ** (1.0 / d)
    x = np.zeros((k, 4), dtype=np.float32)
    x[:, :d] = rng.random((k, d)) * side
    n = 0
    for i, size in enumerate(sizes):
        x[n:n + size, :d] = side * (0.3 + 0.2 * i) + 1e-3 * rng.standard_normal((size, d))
        n += size
    x = torch.as_tensor(x[rng.permutation(k)]).cuda()
    runs = []
    for small in (0, 2048):
        V.set_tuning(19456, 10, 4, small)
        runs.append((hg.layout_step(x, 0.25, V.Params(d=d))[:3], hg.layout(V.Params(d=d, iters=9), x.clone())))
    for a, b in zip(runs[0][0] + (runs[0][1],), runs[1][0] + (runs[1][1],)):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))


@pytest.mark.parametrize("d", [2, 3])
def test_one_block_binning_with_two_targets_per_thread(V, d):
    """A batch whose problems each fit one block and whose levels have more than
    196,608 step threads, so that the blocks number their problems' chunks of two
    points: as the device-wide binning, and as with one target per thread (the
    counting kernel), bit for bit."""
    rng = np.random.default_rng(d)
    mats = [W.random_symmetric(int(n), 6, seed=i) for i, n in enumerate(rng.integers(500, 2049, 220))]
    p = V.Params(d=d, seed=3, iters=12)
    try:
        runs = []
        for small in (2048, 0):
            V.set_tuning(19456, 10, 4, small)
            runs.append(V.batch_layout(mats, p)[0])
        V.set_tuning(19456, 10, 4, 2048)
        V.stats_reset(time_step_kernel=False, count_interactions=True)
        runs.append(V.batch_layout(mats, p)[0])
        assert V.stats()["step_interactions"] > 0
    finally:
        V.stats_reset(time_step_kernel=False, count_interactions=False)
    for x in runs[1:]:
        assert torch.equal(x.view(torch.int32), runs[0].view(torch.int32))
