"""Graphs of one handle in a joined graph share the handle's working memory
(accumulators, hand-over flags, tickets), so the joined graph runs them one
after another; parts of other handles stay side by side."""
import numpy as np
import pytest
import torch

import paper_1207_2192_gb300 as nd
from paper_1207_2192_gb300 import Disk, Nanodisk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,B", [(40e-9, 20), (50e-9, 160), (70e-9, 3)])   # time-sliced clusters, time-sliced CTAs, clusters
@pytest.mark.parametrize("nested", [False, True])
def test_parts_of_one_handle_replay_as_their_own_graphs_do(R, B, nested):
    dt, n = 1e-14, 5
    T, seeds = np.full(B, 300.0), np.arange(B, dtype=np.uint64)

    def run(joined):
        a, other = (Nanodisk([Disk(R, 0.2 * R, alpha=0.02)], [B]) for _ in range(2))
        ms, gs = [], []
        for k, h in enumerate((a, a, other) if B < 152 else (a, a)):   # (above, a launch takes the whole GPU)
            m = h.empty_device()
            h.init_vortex(m, np.full((B, 2), k * 1e-9))
            gs.append(nd.nd_graph_create(h.h, m, nd.ND_METHOD_HEUN, n, dt, T, seeds + k, step0=0))
            ms.append(m)
        tops = list(gs)
        if joined:
            first = [nd.nd_graph_join(gs[:1])] + gs[1:] if nested else gs
            tops = [nd.nd_graph_join(first)]
            assert nd.nd_graph_nodes(tops[0]) == sum(nd.nd_graph_nodes(g) for g in gs)
        for _ in range(3):
            for g in tops:
                nd.nd_graph_launch(g)
        torch.cuda.synchronize()
        assert nd.nd_check_status(a.h) == nd.ND_OK and nd.nd_check_status(other.h) == nd.ND_OK
        if joined:
            nd.nd_graph_destroy(tops[0])
            if nested:
                nd.nd_graph_destroy(first[0])
        for g in gs:
            nd.nd_graph_destroy(g)
        return ms

    for x, y in zip(run(True), run(False)):
        assert torch.equal(x, y)
