"""GPU vs CPU oracle, exact: nodes rated by one thread each (degree <= 32) at the edges of the degree
classes, with arrays that start on and off a 16-byte boundary and rows that end with the arrays."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle as orc
from tests.test_gpu_parity import HOST_PATH

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


def _shifted(gp, g, shift):
    """The device graph with adjncy and adjwgt starting `shift` words past an aligned address."""
    import torch
    dg = gp.DeviceGraph.from_host(g)

    def move(t):
        b = torch.full((t.numel() + 8,), -7, dtype=torch.int32, device="cuda")
        b[shift:shift + t.numel()] = t
        return b[shift:shift + t.numel()]
    return gp.DeviceGraph(dg.n, dg.m2, dg.xadj, move(dg.adjncy), dg.vwgt, move(dg.adjwgt))


def _degrees(wmax):
    """Nodes of every degree from 0 to 40 (joined to a pool of 60 nodes), and a last row of odd length."""
    rng = np.random.default_rng(4)
    u, v = [], []
    for d in range(41):
        for r in range(12):
            node = 60 + d * 12 + r
            u += [node] * d
            v += list(rng.choice(60, d, replace=False))
    g = gg.from_pairs(60 + 41 * 12, np.array(u), np.array(v))
    return gg.with_node_weights(gg.with_edge_weights(g, wmax), 3) if wmax > 1 else g


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("wmax", [1, 6])
@pytest.mark.parametrize("U", [2, 9, 400])
def test_clustering_rows(ctx, shift, wmax, U):
    import paper_2504_17615_gb300 as gp
    g = _degrees(wmax)
    cmap, nc, st = ctx.gp_coarsen(_shifted(gp, g, shift), U, 1, 5, gp.default_config(**HOST_PATH))
    ocmap, onc, ost = orc.coarsen(g, U, 1, 5)
    assert nc == onc and np.array_equal(cmap.cpu().numpy(), ocmap)


@pytest.mark.parametrize("shift", [0, 3])
@pytest.mark.parametrize("wmax", [1, 6])
@pytest.mark.parametrize("k", [2, 128, 255, 256])
def test_refinement_rows(ctx, shift, wmax, k):
    import torch
    import paper_2504_17615_gb300 as gp
    g = _degrees(wmax)
    blk = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    lmax = int(np.bincount(blk, weights=g.vwgt, minlength=k).max()) + 1
    t = torch.from_numpy(blk.copy()).cuda()
    moves = ctx.gp_refine(_shifted(gp, g, shift), k, lmax, 1, 3, t, gp.default_config(**HOST_PATH))
    oblk, omoves = orc.refine(g, k, lmax, 1, 3, blk)
    assert moves == omoves and np.array_equal(t.cpu().numpy(), oblk)
