"""The core estimator's winding test reads signs where single precision
settles them and falls back to FP64 turns where corners are nearly
antiparallel or nearly out of plane: random, lattice-aligned and nearly
antiparallel states against the oracle, in one strip and in several (D > 64)."""
import numpy as np
import pytest

import ndsynth
import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import Disk, Nanodisk

pytestmark = pytest.mark.gpu


def states(D, kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "random":
        return ndsynth.random_unit_vectors(D, seed)
    if kind == "lattice":                                  # angles at multiples of 45 degrees
        phi = rng.integers(0, 8, (D, D)) * (np.pi / 4) + 1e-6 * rng.standard_normal((D, D))
    else:                                                  # corners along one axis, either way
        phi = 0.3 + np.pi * rng.integers(0, 2, (D, D)) + 1e-4 * rng.standard_normal((D, D))
    mz = rng.uniform(-0.9, 0.9, (D, D))
    if kind == "axis":
        mz[rng.random((D, D)) < 0.02] = 1.0                # no in-plane part at all
    s = np.sqrt(1.0 - mz * mz)
    return np.stack([s * np.cos(phi), s * np.sin(phi), mz])


@pytest.mark.parametrize("prec", [nd.ND_FP32, nd.ND_FP64])
@pytest.mark.parametrize("kind", ["random", "lattice", "axis"])
@pytest.mark.parametrize("D", [2, 9, 64, 65, 130])
def test_core_of_rough_states_matches_oracle(O, D, kind, prec):
    disk = Disk(D * 1e-9, 4e-9)
    model = O.Model(disk.R, disk.L)
    assert model.D == D
    h = Nanodisk([disk], [3], prec)
    m = h.to_device([states(D, kind, s) for s in range(3)])
    Xc, st = h.vortex_core(m)
    for r, g in enumerate(h.unpack(m)):
        found, ref, _ = model.vortex_core(g)
        assert (st[r] == nd.ND_OK) == (found == 0)
        if found == 0:
            assert np.max(np.abs(Xc[r] - ref)) <= 1e-12 * disk.R
