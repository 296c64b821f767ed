"""GPU vs CPU oracle, exact: the sub-rounds of the persistent label propagation in every way they
can go -- no proposal, no overflowing target, overflow sets ordered by one block or target by
target, and the 2.5x cap with few and with many emptied clusters."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


def _astray(g, k, share, seed):
    """Ranges of consecutive nodes as blocks, a share of the nodes in random ones."""
    rng = np.random.default_rng(seed)
    base = (np.arange(g.n, dtype=np.int64) * k // g.n).astype(np.int32)
    return np.where(rng.random(g.n) < share, rng.integers(0, k, g.n), base).astype(np.int32)


# the overflow set: below and above 1024 entries, labels on both sides of 256 and of 1024
@pytest.mark.parametrize("k", [2, 5, 255, 256, 300, 1024, 1025])
@pytest.mark.parametrize("n,share", [(3001, 0.1), (20011, 0.6)])
def test_refine_overflow_sets(ctx, k, n, share):
    import torch
    import paper_2504_17615_gb300 as gp
    nx = int(n ** 0.5)
    g = gg.with_edge_weights(gg.grid2d(nx, n // nx), 5)
    blk = _astray(g, k, share, k)
    lmax = int(np.bincount(blk, minlength=k).max())  # no block may grow beyond the heaviest one
    t = torch.from_numpy(blk.copy()).cuda()
    moves = ctx.gp_refine(gp.DeviceGraph.from_host(g), k, lmax, 1, 3, t)
    oblk, omoves = orc.refine(g, k, lmax, 1, 3, blk)
    assert moves == omoves
    assert np.array_equal(t.cpu().numpy(), oblk)


# the cap stops a clustering at ceil(2n/5): few emptied clusters (ranked directly) and many (digits first)
@pytest.mark.parametrize("n", [37, 300, 641, 5003, 60001])
@pytest.mark.parametrize("cmax", [1, 4])
def test_clustering_cap(ctx, n, cmax):
    import paper_2504_17615_gb300 as gp
    g = gg.er(n, 8 * n, 5)
    if cmax > 1:
        g = gg.with_node_weights(g, cmax)
    U = max(2, int(g.vwgt.sum()) // 8)
    cmap, nc, st = ctx.gp_coarsen(gp.DeviceGraph.from_host(g), U, 1, 9)
    ocmap, onc = orc.coarsen(g, U, 1, 9)[:2]
    assert nc == onc == -(-2 * n // 5)
    assert np.array_equal(cmap.cpu().numpy(), ocmap)
