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


@pytest.mark.parametrize("R,prec,B", [(30e-9, nd.ND_FP32, 3), (30e-9, nd.ND_FP32, 20), (60e-9, nd.ND_FP32, 2), (30e-9, nd.ND_FP64, 2)])
def test_expired_wait_of_a_relaxation_is_reported_as_one(R, prec, B):
    """Turns that never come: the call says so, nd_check_status once more, no
    state is touched, and the same handle relaxes normally afterwards."""
    h = Nanodisk([Disk(R, 0.2 * R)], [B], prec)
    m, X = h.empty_device(), np.zeros((B, 2))
    h.init_vortex(m, np.full((B, 2), 1e-9))
    before = m.clone()
    assert nd.nd_check_status(h.h) == nd.ND_OK
    assert nd.nd_selftest_relax_timeout(h.h, m, X) == nd.ND_ERR_TIMEOUT
    assert torch.equal(m, before)
    assert nd.nd_check_status(h.h) == nd.ND_ERR_TIMEOUT
    assert nd.nd_check_status(h.h) == nd.ND_OK
    rc, U, lam, it = h.relax(m, X, tol=1e-300, max_iter=3)
    assert rc == nd.ND_ERR_NOT_CONVERGED and np.all(it == 3) and not torch.equal(m, before)
    assert nd.nd_check_status(h.h) == nd.ND_OK
