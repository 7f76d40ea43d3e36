"""The default stepping plan: few replicas step on thread-block clusters, more
than the resident clusters time-sliced over them, many on the one-CTA kernel
or the global path.  Every plan of a size rounds alike, so a replica ends bit
for bit where the plain plan puts it, whatever shares its handle."""
import numpy as np
import pytest
import torch

import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import Disk, Nanodisk

pytestmark = pytest.mark.gpu


def states(disks, reps, prec, plan, method, steps=5):
    h = Nanodisk(disks, reps, prec)
    if plan is not None:
        nd.nd_set_plan(h.h, 0, method, plan)
    X0 = np.stack([np.linspace(-3e-9, 3e-9, h.B), np.full(h.B, 0.5e-9)], 1)
    m = h.empty_device()
    h.init_vortex(m, X0)
    if method == nd.ND_METHOD_HEUN:
        h.heun(m, steps, 1e-14, np.linspace(0.0, 300.0, h.B), np.arange(h.B, dtype=np.uint64) + 7, step0=3)
    else:
        h.rk4(m, steps, 1e-14)
    torch.cuda.synchronize()
    assert nd.nd_check_status(h.h) == nd.ND_OK
    return m


@pytest.mark.parametrize("method", [nd.ND_METHOD_HEUN, nd.ND_METHOD_RK4])
@pytest.mark.parametrize("R,prec,B,plain", [
    (7e-9, nd.ND_FP32, 3, 0), (16e-9, nd.ND_FP32, 9, 0), (32e-9, nd.ND_FP32, 17, 0), (33e-9, nd.ND_FP32, 1, 0),
    (50e-9, nd.ND_FP32, 33, 0), (64e-9, nd.ND_FP32, 8, 0), (65e-9, nd.ND_FP32, 9, 100), (128e-9, nd.ND_FP32, 2, 100),
    (9e-9, nd.ND_FP64, 16, 0), (31e-9, nd.ND_FP64, 18, 0), (34e-9, nd.ND_FP64, 2, 100), (64e-9, nd.ND_FP64, 17, 100)])
def test_default_plan_gives_the_plain_plans_trajectory(R, prec, B, plain, method):
    disks = [Disk(R, 0.2 * R, alpha=0.02, hext=(0.0, 5e3, 0.0))]
    assert torch.equal(states(disks, [B], prec, None, method), states(disks, [B], prec, plain, method))


@pytest.mark.parametrize("method", [nd.ND_METHOD_HEUN, nd.ND_METHOD_RK4])
def test_time_sliced_clusters_with_disks_of_different_sizes(method):
    """One class (P = 128) of disks with different rows per CTA, more replicas
    than clusters: the clusters pass replicas of every size on."""
    disks = [Disk(r * 1e-9, 8e-9, alpha=0.02) for r in (33, 41, 50, 57, 64)]
    reps = [4, 3, 5, 4, 3]
    assert torch.equal(states(disks, reps, nd.ND_FP32, 200, method), states(disks, reps, nd.ND_FP32, 0, method))
    assert torch.equal(states(disks, reps, nd.ND_FP32, 201, method), states(disks, reps, nd.ND_FP32, 0, method))


@pytest.mark.parametrize("prec", [nd.ND_FP32, nd.ND_FP64])
@pytest.mark.parametrize("tol,max_iter", [(1e-12, 300), (2e-3, 5000)])
def test_replicas_relaxing_in_turns_end_where_they_do_alone(prec, tol, max_iter):
    """More replicas than clusters relax in turns of some sweeps: each ends
    with the state, multipliers and sweep count it has in a small handle,
    whether its sweeps run out or it converges."""
    disk = Disk(30e-9, 6e-9)
    B = 20
    X = np.stack([np.linspace(0.0, 12e-9, B), np.linspace(-2e-9, 2e-9, B)], 1)

    def relax(sel):
        h = Nanodisk([disk], [len(sel)], prec)
        m = h.empty_device()
        h.init_vortex(m, np.zeros((len(sel), 2)))
        rc, U, lam, it = h.relax(m, X[sel], tol=tol, max_iter=max_iter)
        assert nd.nd_check_status(h.h) == nd.ND_OK
        assert rc == (nd.ND_ERR_NOT_CONVERGED if (it == max_iter).any() else nd.ND_OK)
        return m, U, lam, it

    m, U, lam, it = relax(np.arange(B))
    assert (it == max_iter).all() if tol < 1e-9 else len(set(it)) > 1
    parts = [relax(np.arange(k, k + 5)) for k in range(0, B, 5)]
    assert torch.equal(m, torch.cat([p[0] for p in parts]))
    assert np.array_equal(lam, np.concatenate([p[2] for p in parts]))
    assert np.array_equal(it, np.concatenate([p[3] for p in parts]))


def test_graph_of_time_sliced_clusters_outlives_other_schedules():
    """A graph keeps the schedule it was captured with when direct calls of
    other lengths replace the handle's cached one."""
    disk = Disk(40e-9, 8e-9, alpha=0.02)
    B = 20                                                   # more than the resident clusters
    T, seeds, dt = np.full(B, 300.0), np.arange(B, dtype=np.uint64), 1e-14
    a, b = Nanodisk([disk], [B]), Nanodisk([disk], [B])
    ma, mb, mc = a.empty_device(), b.empty_device(), a.empty_device()
    for h, m in ((a, ma), (b, mb), (a, mc)):
        h.init_vortex(m, np.zeros((B, 2)))
    g = nd.nd_graph_create(a.h, ma, nd.ND_METHOD_HEUN, 6, dt, T, seeds, step0=0)
    try:
        for k in range(3):
            nd.nd_graph_launch(g)
            a.heun(mc, 3 + k, dt, T, seeds)                  # another schedule each time
            b.heun(mb, 6, dt, T, seeds, step0=6 * k)
        torch.cuda.synchronize()
        assert torch.equal(ma, mb)
    finally:
        nd.nd_graph_destroy(g)
    assert nd.nd_check_status(a.h) == nd.ND_OK
