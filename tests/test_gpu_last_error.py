"""A CUDA call that fails inside the library is reported by the status only: the
runtime's last error is clear afterwards, so the next sort does not report it."""
from __future__ import annotations

import ctypes

import pytest

pytestmark = pytest.mark.gpu


def test_failure_leaves_no_last_error():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_05245_gb300 as ps
    from paper_2305_05245_gb300 import _lib
    lib = _lib.load()
    rt = ctypes.CDLL("libcudart.so.13")
    x = torch.randint(0, 100, (1000,), dtype=torch.int32, device="cuda")
    off = torch.tensor([0, 500, 1000], device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    h = ctypes.c_void_p(s.cuda_stream)
    assert rt.cudaGetLastError() == 0
    assert rt.cudaStreamBeginCapture(h, 2) == 0
    rc = lib.ps_sort_batch(off.data_ptr(), 2, x.data_ptr(), 0, 1, h)  # has to read the offsets back: not while capturing
    left = rt.cudaPeekAtLastError()
    graph = ctypes.c_void_p()
    rt.cudaStreamEndCapture(h, ctypes.byref(graph))
    rt.cudaGetLastError()
    assert rc == -4 and lib.ps_last_cuda_error() != 0
    assert left == 0
    ps.sort(x)
    torch.cuda.synchronize()
    assert bool((x[1:] >= x[:-1]).all())
