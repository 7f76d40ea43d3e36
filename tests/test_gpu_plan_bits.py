"""Every stepping plan of a size rounds alike: the one-CTA kernel in each thread
count, the global path and both cluster plans end bit for bit together, and the
default takes the plan that it is said to take."""
import numpy as np
import pytest
import torch

import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import Disk, Nanodisk

pytestmark = pytest.mark.gpu

ONE, GLOBAL, C8, C16 = 0, 100, 200, 201


def end(disks, reps, prec, plan, method, steps=4, T=None, grid3x=False):
    """The state after a few steps on a plan, or None where the size has no such plan."""
    h = Nanodisk(disks, reps, prec, grid3x=grid3x)
    if plan is not None:
        try:
            nd.nd_set_plan(h.h, 0, method, plan)
        except nd.NDError:
            return None
    X0 = np.stack([np.linspace(-2e-9, 2e-9, h.B), np.full(h.B, 0.5e-9)], 1)
    m = h.empty_device()
    h.init_vortex(m, X0)
    if method == nd.ND_METHOD_HEUN:
        T = np.linspace(0.0, 300.0, h.B) if T is None else T
        h.heun(m, steps, 1e-14, T, np.arange(h.B, dtype=np.uint64) + 7, step0=3)
    else:
        h.rk4(m, steps, 1e-14)
    torch.cuda.synchronize()
    assert nd.nd_check_status(h.h) == nd.ND_OK
    return m


@pytest.mark.parametrize("method", [nd.ND_METHOD_HEUN, nd.ND_METHOD_RK4])
@pytest.mark.parametrize("prec", [nd.ND_FP32, nd.ND_FP64])
@pytest.mark.parametrize("R,B,grid3x", [(7e-9, 5, False), (8e-9, 18, False), (15e-9, 18, False), (31e-9, 18, False),
                                        (33e-9, 3, False), (50e-9, 18, False), (64e-9, 3, False), (90e-9, 9, True),
                                        (100e-9, 9, False)])
def test_plans_of_a_size_end_bit_for_bit_together(R, B, grid3x, prec, method):
    disks = [Disk(R, 0.2 * R, alpha=0.02, hext=(0.0, 5e3, 0.0))]
    states = {p: end(disks, [B], prec, p, method, grid3x=grid3x) for p in (ONE, 1, 2, GLOBAL, C8, C16)}
    states = {p: m for p, m in states.items() if m is not None}
    assert GLOBAL in states                                   # every size has it
    assert R > 64.5e-9 or C8 in states                        # and every one up to P = 128 a cluster plan
    for p, m in states.items():
        assert torch.equal(m, states[GLOBAL]), p


@pytest.mark.parametrize("R,B,prec,threads", [
    # threads of the plan: clusters of 16 and 8 CTAs of 256 threads (512 at P = 256), one CTA, 0 for the global path
    (7e-9, 3, nd.ND_FP32, 128), (15e-9, 3, nd.ND_FP32, 16 * 256), (30e-9, 3, nd.ND_FP32, 8 * 256),
    (30e-9, 20, nd.ND_FP32, 8 * 256), (30e-9, 65, nd.ND_FP32, 384), (60e-9, 2, nd.ND_FP32, 16 * 256),
    (60e-9, 16, nd.ND_FP32, 8 * 256), (60e-9, 65, nd.ND_FP32, 512), (100e-9, 4, nd.ND_FP32, 16 * 512),
    (100e-9, 65, nd.ND_FP32, 0), (250e-9, 1, nd.ND_FP32, 0), (9e-9, 2, nd.ND_FP64, 16 * 256),
    (30e-9, 16, nd.ND_FP64, 8 * 256), (30e-9, 65, nd.ND_FP64, 384), (60e-9, 2, nd.ND_FP64, 16 * 256),
    (60e-9, 65, nd.ND_FP64, 0)])
def test_the_default_takes_clusters_for_few_replicas(R, B, prec, threads):
    h = Nanodisk([Disk(R, 0.2 * R)], [B], prec)
    info = nd.nd_plan_info(h.h, 0)
    assert info["plan_heun"] == info["plan_rk4"] == -1
    assert info["threads_heun"] == threads and info["threads_rk4"] == threads


@pytest.mark.parametrize("method", [nd.ND_METHOD_HEUN, nd.ND_METHOD_RK4])
def test_hand_overs_between_replicas_of_unequal_cost(method):
    """FP64, one class of D = 33 and 64, thermal and T = 0: the slots' shares are
    equal in steps, not in time, so hand-overs are waited for."""
    disks, reps = [Disk(64e-9, 8e-9, alpha=0.02), Disk(33e-9, 8e-9, alpha=0.02)], [15, 3]
    T = np.array([300.0] * 9 + [0.0] * 9)
    a, b = (end(disks, reps, nd.ND_FP64, p, method, steps=150, T=T) for p in (C8, GLOBAL))
    assert torch.equal(a, b)


@pytest.mark.parametrize("R,B,prec", [
    (7e-9, 3, nd.ND_FP32), (30e-9, 3, nd.ND_FP32), (30e-9, 70, nd.ND_FP32), (61e-9, 2, nd.ND_FP32), (61e-9, 70, nd.ND_FP32),
    (70e-9, 2, nd.ND_FP32), (70e-9, 20, nd.ND_FP32), (15e-9, 2, nd.ND_FP64), (30e-9, 70, nd.ND_FP64), (37e-9, 2, nd.ND_FP64),
    (37e-9, 30, nd.ND_FP64)])
def test_field_writes_whole_blocks_whatever_kernel_runs(O, R, B, prec):
    """Cells outside a mask that is no disk, and the padding, are written as zero
    by the cluster, the one-CTA and the global form; inside, the oracle's field."""
    disk = Disk(R, 0.2 * R, hext=(0.0, 5e3, 0.0))
    h, model = Nanodisk([disk], [B], prec), O.Model(disk.R, disk.L, hext=disk.hext)
    mask = np.random.default_rng(2).random((model.D, model.D)) < 0.7
    h.set_mask(0, mask)
    model.set_mask(mask)
    g = torch.Generator(device="cuda").manual_seed(1)
    D, Dp = h.layout[0]["D"], h.layout[0]["Dpad"]
    inside = torch.as_tensor(mask).cuda()
    m = torch.randn(B, 3, D, Dp, device="cuda", dtype=h.empty_device().dtype, generator=g)
    m = m / m.norm(dim=1, keepdim=True)
    m[..., D:] = 0.0
    b = torch.full_like(m, float("nan"))
    h.field(m.view(-1), b.view(-1))
    assert torch.equal(b[..., D:], torch.zeros_like(b[..., D:]))
    assert torch.all(b[..., :D][:, :, ~inside] == 0.0)
    grids, out = h.unpack(m.view(-1)), h.unpack(b.view(-1))
    tol = 1e-11 if prec == nd.ND_FP64 else 1e-5               # relative L2, of the package's field comparisons
    for r in (0, B - 1):
        ref = model.field(grids[r] * mask) * mask
        assert np.linalg.norm(out[r] - ref) < tol * np.linalg.norm(ref)
