"""A hand-over wait lasts as long as the other side works: the time that a
replica's second part waits grows with the steps of a call, and the limit counts
from the other side's last progress."""
import numpy as np
import pytest
import torch

import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import Disk, Nanodisk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("plan", [0, 200, 201])
@pytest.mark.parametrize("R,n", [(50e-9, 6001), (14e-9, 10002)])
def test_wait_outlasts_its_limit_while_the_other_side_steps(R, n, plan):
    h = Nanodisk([Disk(R, 0.2 * R, alpha=0.02)], [2])
    dt = 1e-14
    m = h.empty_device()
    h.init_vortex(m, np.array([[1e-9, 0.0], [0.0, 1e-9]]))
    ref, other = m.clone(), m.clone()
    start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    h.rk4(other, 3, dt)                                      # (the kernels are loaded)
    nd.nd_set_plan(h.h, 0, nd.ND_METHOD_RK4, plan)
    start.record()
    h.rk4(ref, n, dt)
    end.record()
    torch.cuda.synchronize()
    assert start.elapsed_time(end) > 100.0                    # ms: the first half outlasts the 17 ms limit
    nd.nd_selftest_handover_progress(h.h, m, n, dt, plan)
    assert nd.nd_check_status(h.h) == nd.ND_OK
    half = m.numel() // 2
    assert torch.equal(m[:half], ref[:half])
    assert not torch.equal(m[half:], ref[half:])              # the second replica was left alone
