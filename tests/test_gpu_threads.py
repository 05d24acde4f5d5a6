"""Host threads that lay out at the same time, as the request server's slots do:
every result is the one of the same call alone, bit for bit.  The problems'
sizes differ, so that the threads' levels take launches of different shared
memory from the same kernels."""
import threading
import time

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

# rows of the two threads' matrices in turn, per d; one problem or a batch
ONE = {2: ((4096, 2100), (1500, 2048), (520, 1000)), 3: ((2048, 1100), (1030, 1900), (520, 1000)), 4: ((2048, 1100),)}


@pytest.fixture(scope="module")
def V():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1105_4490_gb300 as P
    assert torch.cuda.is_available()
    return P


def _together(jobs, rounds):
    """Runs the jobs' functions in one thread each, `rounds` times, on a stream
    of the thread's own; the results per job and round."""
    out, errors = [[] for _ in jobs], []
    gate = threading.Barrier(len(jobs))

    def work(i, job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(rounds):
                    gate.wait(60.0)
                    out[i].append(job().cpu().numpy())
        except Exception as e:  # noqa: BLE001 - reported by the test
            errors.append(e)
            gate.abort()

    threads = [threading.Thread(target=work, args=(i, j)) for i, j in enumerate(jobs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    return out


@pytest.mark.parametrize("d", (2, 3, 4))
def test_layouts_of_two_threads(V, d):
    for pair in ONE[d]:
        jobs = []
        for i, rows in enumerate(pair):
            hg = V.Hypergraph.from_matrix(W.random_symmetric(rows, 6, seed=rows))
            jobs.append(lambda hg=hg, i=i: hg.layout(V.Params(d=d, seed=3 + i)))
        alone = [j().cpu().numpy() for j in jobs]
        torch.cuda.synchronize()
        for ref, got in zip(alone, _together(jobs, 6)):
            assert all(np.array_equal(ref, x) for x in got), (d, pair)


@pytest.mark.parametrize("d", (2, 3))
def test_batches_of_two_threads(V, d):
    sets = [[W.random_symmetric(n, 6, seed=n) for n in range(a, b, 97)] for a, b in ((1200, 2048), (300, 1100))]
    sets = [s * (70 // len(s) + 1) for s in sets]  # more than 64 problems a level
    jobs = [lambda s=s: V.batch_order(s, V.Params(d=d, seed=3))[0] for s in sets]
    alone = [j().cpu().numpy() for j in jobs]
    torch.cuda.synchronize()
    for ref, got in zip(alone, _together(jobs, 4)):
        assert all(np.array_equal(ref, x) for x in got)


@pytest.mark.parametrize("d,sizes", ((3, (1200, 1999)), (2, (1500, 4000))))
def test_two_server_slots(V, d, sizes):
    lo, hi = sizes
    mats = [W.random_symmetric(lo + (i * 463) % (hi - lo + 1), 6, seed=i) for i in range(24)]
    ref = []
    for A in mats:
        rp, _, _ = V.Hypergraph.from_matrix(A).order(V.Params(d=d, seed=3), None, sbd=False, with_tree=False)
        ref.append(rp.cpu().numpy())
    with V.Server(V.Params(d=d, seed=3), slots=2, max_batch=1) as srv:
        ids = [srv.submit_matrix(A) for A in mats]
        for r, want in zip(ids, ref):
            info = srv.wait(r, 60.0)
            assert info["state"] == "done", info
            assert np.array_equal(srv.result(r), want)


def test_four_server_slots_under_load(V):
    """Four slots that take requests of the small mix as they come, each a layout of
    ten levels whose steps are queued far ahead: they all finish, with the plain
    ordering's permutations."""
    mats = W.batch_mix(180, 5)
    with V.Server(V.Params(d=3, seed=1), slots=4) as srv:
        for rnd in range(3):
            ids = []
            for i, A in enumerate(mats):
                ids.append(srv.submit_matrix(A))
                if i % 4 == 3:
                    time.sleep(0.02)
            for r in ids:
                assert srv.wait(r, 60.0)["state"] == "done"
            got = {i: srv.result(ids[i]).copy() for i in range(rnd, len(ids), 23)}
    for i, perm in got.items():
        rp, _, _ = V.Hypergraph.from_matrix(mats[i]).order(V.Params(d=3, seed=1), None, sbd=False, with_tree=False)
        assert np.array_equal(perm, rp.cpu().numpy()), i
