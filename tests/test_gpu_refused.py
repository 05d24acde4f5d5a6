"""A refused CUDA call stops a launch sequence: no later kernel of it runs on
what the refused one should have written, and the call returns the error."""
import ctypes

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


def test_nothing_is_launched_after_a_refused_call(V):
    lib = V.load()
    hg = V.Hypergraph.from_matrix(W.random_symmetric(2000, 6, seed=5))
    want = hg.components()
    labels = torch.full((hg.k,), -7, dtype=torch.int32, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    cudart = ctypes.CDLL("libcudart.so.13")  # the copy that the library uses is loaded already
    assert cudart.cudaSetDevice(12345) != 0  # refused by the runtime; the device stays
    assert lib.vmo_components(hg._h, ctypes.c_void_p(labels.data_ptr()), stream) != 0
    torch.cuda.synchronize()
    assert bool((labels == -7).all())
    assert lib.vmo_components(hg._h, ctypes.c_void_p(labels.data_ptr()), stream) == 0  # the error was collected
    assert torch.equal(labels, want)
