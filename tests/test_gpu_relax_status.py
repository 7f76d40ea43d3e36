"""What a relaxation that cannot finish reports, and what it leaves behind."""
import numpy as np
import pytest
import torch

import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import Disk, Nanodisk

pytestmark = pytest.mark.gpu


def test_error_in_a_later_class_leaves_the_stream_ordered():
    """A class on a side stream still relaxes when the launch of the next class
    is refused (more replicas than a grid has rows): what the caller's stream
    does after the error sees that class's relaxation finished."""
    disks = [Disk(30e-9, 6e-9), Disk(33e-9, 6e-9)]            # P = 64 on chip, P = 128 grid-wide in FP64
    h, one = Nanodisk(disks, [1, 65536], nd.ND_FP64), Nanodisk(disks[:1], [1], nd.ND_FP64)
    X = np.zeros((h.B, 2))
    X[0] = 8e-9, 0.0
    m, start = h.empty_device(), one.empty_device()
    one.init_vortex(start, np.zeros((1, 2)))
    n = start.numel()
    m[:n] = start
    at_return, at_end = torch.empty_like(start), torch.empty_like(start)
    stream = torch.cuda.Stream()
    for d, B in ((disks[0], 1), (disks[1], 32)):              # both forms' kernels are loaded (loading one waits for the GPU)
        w = Nanodisk([d], [B], nd.ND_FP64)
        mw = w.empty_device()
        w.init_vortex(mw, np.zeros((B, 2)))
        w.relax(mw, np.zeros((B, 2)), tol=1e-300, max_iter=1)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        with pytest.raises(nd.NDError):
            h.relax(m, X, tol=1e-300, max_iter=5000, stream=stream)
        at_return.copy_(m[:n])
    torch.cuda.synchronize()
    at_end.copy_(m[:n])
    assert torch.equal(at_return, at_end)
    ref = start.clone()
    one.relax(ref, X[:1], tol=1e-300, max_iter=5000)
    assert torch.equal(at_end, ref)
