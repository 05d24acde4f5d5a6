"""Destroying a handle: its arrays stay valid for work that is still queued on
any stream, and other threads' layouts go on undisturbed."""
import threading

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


def test_destroy_waits_for_work_on_other_streams(V):
    for _ in range(3):
        hg = V.Hypergraph.from_matrix(W.grid_laplacian_2d(64))
        done = torch.cuda.Event()
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            torch.cuda._sleep(100_000_000)  # about 50 ms, in place of a user's kernel that reads the arrays
            done.record()
        del hg
        assert done.query()


def test_destroy_beside_layouts_of_another_thread(V):
    hg = V.Hypergraph.from_matrix(W.random_symmetric(3000, 6, seed=5))
    small = W.grid_laplacian_2d(20)
    rp, ci = torch.as_tensor(small.rowptr).cuda(), torch.as_tensor(small.colidx).cuda()
    ref = hg.layout(V.Params(d=3, seed=2)).cpu().numpy()
    stop, errors = threading.Event(), []

    def handles():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                while not stop.is_set():
                    V.Hypergraph(rp, ci, small.m, small.n)  # built, and destroyed at once
        except Exception as e:  # noqa: BLE001 - reported by the test
            errors.append(e)

    th = threading.Thread(target=handles)
    th.start()
    try:
        with torch.cuda.stream(torch.cuda.Stream()):
            got = [hg.layout(V.Params(d=3, seed=2)) for _ in range(20)]
    finally:
        stop.set()
        th.join()
    torch.cuda.synchronize()
    assert not errors, errors
    assert all(np.array_equal(ref, x.cpu().numpy()) for x in got)


def test_level_arrays_are_given_back(V):
    """A layout's level arrays of more than 1 GiB return to the device with the
    call's end, as far as they exceed what the library keeps."""
    n = 20000  # a full pattern: 1.6 GB of adjacency, next to nothing per vertex
    rowptr = torch.arange(n + 1, dtype=torch.int32, device="cuda") * n
    colidx = torch.arange(n, dtype=torch.int32, device="cuda").repeat(n)
    hg = V.Hypergraph(rowptr, colidx, n, n)
    del colidx
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    hg.layout(V.Params(d=3, iters=0, multilevel=False))
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= (1 << 30) + (256 << 20)
