"""Every form of the relaxation sweep against the oracle, sweep by sweep: the
thread-block cluster (few replicas), the one-CTA kernel and the grid-wide passes
(more replicas), in both precisions, with disks and (FP64) with masks that are
not disks."""
import numpy as np
import pytest

import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import Disk, Nanodisk

pytestmark = pytest.mark.gpu

TOL = {nd.ND_FP64: 1e-11, nd.ND_FP32: 2e-5}       # of the package's other sweep comparisons with the oracle


def rough_mask(D, seed):
    """An elongated cell set with holes, symmetric in nothing."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[:D, :D] - 0.5 * (D - 1)
    m = ((x / (0.5 * D)) ** 2 + (y / (0.36 * D)) ** 2 <= 1.0) & (rng.random((D, D)) > 0.06)
    m[D // 2 - 2:D // 2 + 2, D // 2 - 2:D // 2 + 2] = True
    return m


def sweeps_against_oracle(O, R, prec, B, mask, nsweep):
    disk = Disk(R, 0.25 * R)
    h, model = Nanodisk([disk], [B], prec), O.Model(disk.R, disk.L)
    if mask:
        m0 = rough_mask(model.D, 7)
        h.set_mask(0, m0)
        model.set_mask(m0)
    # three different replicas, repeated
    X = np.array([[2.5e-9, 1.0e-9], [0.0, 0.0], [-1e-9, 2e-9]])
    starts = [model.init_vortex(0.0, 0.0), model.init_vortex(-1e-9, 2e-9), model.init_vortex(1e-9, 0.0)]
    m = h.to_device([starts[r % 3] for r in range(B)])
    start = h.unpack(m)
    first = m.clone()
    rc, U, lam, it = h.relax(m, X[np.arange(B) % 3], tol=1e-300, max_iter=nsweep)
    assert rc == nd.ND_ERR_NOT_CONVERGED and np.all(it == nsweep)
    assert nd.nd_check_status(h.h) == nd.ND_OK
    out = h.unpack(m)
    tol = TOL[prec]
    for r in range(min(B, 3)):
        mm, lm = start[r], np.zeros(2)
        for _ in range(nsweep):
            mm, lm, _ = model.relax_sweep(mm, X[r], lm)
        assert np.max(np.abs(out[r] - mm)) < 10 * tol
        assert np.allclose(lam[r], lm, rtol=100 * tol, atol=100 * tol * max(1e-3, np.abs(lm).max()))
    for r in range(3, B):                           # the same replica ends alike wherever it ran
        assert np.array_equal(out[r], out[r % 3]) and np.array_equal(lam[r], lam[r % 3])
    return h, first, X[np.arange(B) % 3]


@pytest.mark.parametrize("R,prec,B", [
    (17e-9, nd.ND_FP32, 3), (33e-9, nd.ND_FP32, 8), (33e-9, nd.ND_FP32, 2), (65e-9, nd.ND_FP32, 2),
    (9e-9, nd.ND_FP64, 2), (17e-9, nd.ND_FP64, 3), (34e-9, nd.ND_FP64, 2)])
def test_cluster_sweeps_with_ctas_that_own_no_rows(O, R, prec, B):
    """The smallest disk of a size class leaves some CTAs of a cluster without
    rows: they exchange sums with the others all the same, sweep after sweep."""
    h, m, X = sweeps_against_oracle(O, R, prec, B, False, 4)
    ends = []
    for _ in range(3):
        mm = m.clone()
        rc, U, lam, it = h.relax(mm, X, tol=1e-300, max_iter=700)
        assert rc == nd.ND_ERR_NOT_CONVERGED and np.all(it == 700)
        ends.append((mm.cpu().numpy(), lam))
    assert nd.nd_check_status(h.h) == nd.ND_OK
    for mm, lam in ends[1:]:
        assert np.array_equal(mm, ends[0][0]) and np.array_equal(lam, ends[0][1])


@pytest.mark.parametrize("R,grid3x", [(70e-9, False), (90e-9, True), (120e-9, False)])
def test_multipliers_above_128_are_held_in_more_than_fp32(O, R, grid3x):
    """FP32 sweeps above P = 128 hold the multipliers in more bits in every form:
    on clusters (2 replicas) and in grid-wide passes (24) they are no widened
    floats and follow the oracle's."""
    disk, model = Disk(R, 0.1 * R), O.Model(R, 0.1 * R)
    X = np.array([2.5e-9, 1.0e-9])
    for B in (2, 24):
        h = Nanodisk([disk], [B], nd.ND_FP32, grid3x=grid3x)
        m = h.empty_device()
        h.init_vortex(m, np.zeros((B, 2)))
        mm, lm = h.unpack(m)[0], np.zeros(2)
        rc, U, lam, it = h.relax(m, np.tile(X, (B, 1)), tol=1e-300, max_iter=4)
        for _ in range(4):
            mm, lm, _ = model.relax_sweep(mm, X, lm)
        assert np.all(lam != lam.astype(np.float32))
        assert np.allclose(lam[0], lm, rtol=100 * TOL[nd.ND_FP32], atol=100 * TOL[nd.ND_FP32] * np.abs(lm).max())


FORMS = [
    # one CTA per replica (its threads), grid-wide passes (0), clusters of 8 and 16 CTAs
    (7e-9, nd.ND_FP32, 3, 128), (15e-9, nd.ND_FP32, 65, 256), (30e-9, nd.ND_FP32, 65, 384), (61e-9, nd.ND_FP32, 65, 512),
    (15e-9, nd.ND_FP64, 65, 256), (30e-9, nd.ND_FP64, 65, 384),
    (70e-9, nd.ND_FP32, 65, 0), (37e-9, nd.ND_FP64, 65, 0), (66e-9, nd.ND_FP64, 3, 0),
    (15e-9, nd.ND_FP32, 3, 16 * 256), (30e-9, nd.ND_FP32, 3, 8 * 256), (61e-9, nd.ND_FP32, 3, 16 * 256),
    (61e-9, nd.ND_FP32, 17, 8 * 256), (70e-9, nd.ND_FP32, 3, 16 * 512), (7e-9, nd.ND_FP64, 3, 8 * 256),
    (30e-9, nd.ND_FP64, 17, 8 * 256), (37e-9, nd.ND_FP64, 3, 16 * 256)]


@pytest.mark.parametrize("R,prec,B,threads", FORMS)
def test_every_form_of_the_sweep_matches_the_oracle(O, R, prec, B, threads):
    h, m, X = sweeps_against_oracle(O, R, prec, B, False, 3)
    assert nd.nd_plan_info(h.h, 0)["threads_heun"] == threads   # the form that ran


@pytest.mark.parametrize("R,prec,B,threads", [f for f in FORMS if f[1] == nd.ND_FP64])
def test_every_form_of_the_sweep_follows_masks_that_are_not_disks(O, R, prec, B, threads):
    """In FP64: a cell without neighbours inside the mask has a field of a
    hundredth of the others', whose direction FP32 transforms do not fix to the
    tolerance (their error is relative to the largest field)."""
    h, m, X = sweeps_against_oracle(O, R, prec, B, True, 3)
    assert nd.nd_plan_info(h.h, 0)["threads_heun"] == threads
