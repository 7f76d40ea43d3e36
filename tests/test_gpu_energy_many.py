"""Energies of more replicas than a grid has rows, in turns over a bounded
workspace: every replica has the energy that it has in a small handle."""
import numpy as np
import pytest
import torch

import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import Disk, Nanodisk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,B,prec", [(7e-9, 65537, nd.ND_FP32), (7e-9, 65600, nd.ND_FP64), (64e-9, 1400, nd.ND_FP32)])
def test_energies_in_turns_match_a_small_handle(O, R, B, prec):
    disk = Disk(R, 0.2 * R, hext=(0.0, 5e3, 0.0))
    h = Nanodisk([disk], [B], prec)
    D, Dp = h.layout[0]["D"], h.layout[0]["Dpad"]
    g = torch.Generator(device="cuda").manual_seed(3)
    m = torch.randn(B, 3, D, Dp, device="cuda", dtype=h.empty_device().dtype, generator=g)
    m /= m.norm(dim=1, keepdim=True)
    sel = np.unique(np.r_[0, 1, 1279, 1280, B - 2, B - 1, np.random.default_rng(5).integers(0, B, 40)])
    small = Nanodisk([disk], [len(sel)], prec)
    ms = m[torch.as_tensor(sel).cuda()].contiguous()
    free0 = torch.cuda.mem_get_info()[0]
    E, dL = nd.nd_energy(h.h, m.view(-1), B, with_dL=True)
    assert free0 - torch.cuda.mem_get_info()[0] < 400e6       # 256 MB of spectra and the partial sums
    Es, dLs = nd.nd_energy(small.h, ms.view(-1), len(sel), with_dL=True)
    assert np.array_equal(E[sel], Es) and np.array_equal(dL[sel], dLs)
    model = O.Model(disk.R, disk.L, hext=disk.hext)
    for k, r in enumerate(sel[:3]):
        assert E[r] == pytest.approx(model.energy(small.unpack(ms.view(-1))[k]), rel=1e-12)
