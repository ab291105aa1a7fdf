"""The workspace pool gives its memory back: what it holds after calls that failed under a stream
capture (where device memory can be neither allocated nor freed) is freed later all the same."""
import ctypes

import pytest
import torch

from paper_1511_07042_gb300 import inputs

pytestmark = pytest.mark.gpu


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_failed_call_under_capture_loses_no_buffer(gpu_bmg):
    rt = ctypes.CDLL("libcudart.so.13")
    # workspaces of 31 and 62 MB (smaller ones do not change the free bytes that CUDA reports)
    small, large = (torch.zeros((n, 160), dtype=torch.float64, device="cuda") for n in (9600, 20000))
    G = torch.empty((160, 160), dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()

    def trim():
        p = gpu_bmg.Problem(*inputs.icosahedron(), 1)
        p.close()                      # closing a problem empties the pool

    for X in (small, large):           # first calls: one-time allocations of the runtime
        gpu_bmg.gram(X, X, 160, G)
    trim()
    before = free_bytes()
    gpu_bmg.gram(small, small, 160, G)
    assert free_bytes() < before       # the pool holds a workspace
    with torch.cuda.stream(stream):
        graph = ctypes.c_void_p()
        assert rt.cudaStreamBeginCapture(ctypes.c_void_p(stream.cuda_stream), 0) == 0
        with pytest.raises(gpu_bmg.BmgError):
            gpu_bmg.gram(large, large, 160, G)
        rt.cudaStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph))
        rt.cudaGetLastError()
    trim()
    assert free_bytes() >= before
    gpu_bmg.gram(large, large, 160, G)
    assert torch.equal(G, torch.zeros_like(G))


def test_destroying_nothing_empties_the_pool(gpu_bmg):
    """A program that only calls steps has no problem to destroy."""
    X = torch.zeros((9600, 160), dtype=torch.float64, device="cuda")
    G = torch.empty((160, 160), dtype=torch.float64, device="cuda")
    gpu_bmg.gram(X, X, 160, G)
    gpu_bmg.LIB.bmg_destroy(None)
    before = free_bytes()
    gpu_bmg.gram(X, X, 160, G)
    assert free_bytes() < before
    gpu_bmg.LIB.bmg_destroy(None)
    assert free_bytes() >= before
