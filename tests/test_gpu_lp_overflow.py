"""GPU vs CPU oracle, exact: refinement whose proposals nearly all overflow their targets -- few proposals, decided by a warp
each; many, resolved a target per block with fewer and with more labels than blocks; and sets that one block sorts."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle as orc
from tests._util import star

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


GRAPHS = {"rmat": lambda: gg.with_node_weights(gg.with_edge_weights(gg.rmat(13, 8, seed=5), 3), 4),
          "grid": lambda: gg.grid2d(93, 87), "star": lambda: star(1500), "er": lambda: gg.er(700, 3000, 2)}


# one sub-round a round: every node is active, so that up to n proposals meet; 1024 labels keep their weights in
# shared memory; 33 blocks of 256 threads at 8192 nodes, 32 labels a block at most are resolved target by target
@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("S", [1, 8])
@pytest.mark.parametrize("k", [2, 3, 31, 34, 500, 1024, 1025, 2000])
def test_overflow(ctx, name, S, k):
    import torch
    import paper_2504_17615_gb300 as gp
    g = GRAPHS[name]()
    if k > g.n:
        pytest.skip("more blocks than nodes")
    blk = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    for room in (0, 7):
        lmax = int(np.bincount(blk, weights=g.vwgt, minlength=k).max()) + room
        t = torch.from_numpy(blk.copy()).cuda()
        moves = ctx.gp_refine(gp.DeviceGraph.from_host(g), k, lmax, 1, 3, t, gp.default_config(lp_subrounds=S))
        oblk, omoves = orc.refine(g, k, lmax, 1, 3, blk, orc.Config.default(lp_subrounds=S))
        assert moves == omoves and np.array_equal(t.cpu().numpy(), oblk)
