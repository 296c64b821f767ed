"""GPU vs CPU oracle, exact: nodes of more than 128 neighbours in label propagation (a block with a shared
table each up to 18432; hubs by many blocks: counted per label up to 1024 labels, hash tables beyond)
and coarse nodes with long segments in contraction."""
from __future__ import annotations

import dataclasses

import numpy as np
import pytest

import graphgen as gg
import oracle as orc
from tests._util import star
from tests.test_gpu_parity import HOST_PATH, canon

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


def _hubs(n, degs, extra, wmax):
    """Hubs 0, 1, .. of the given degrees over a sparse random graph."""
    rng = np.random.default_rng(n)
    u = [np.full(d, h) for h, d in enumerate(degs)] + [rng.integers(0, n, extra)]
    v = [rng.choice(np.arange(len(degs), n), d, replace=False) for d in degs] + [rng.integers(0, n, extra)]
    u, v = np.concatenate(u), np.concatenate(v)
    g = gg.from_pairs(n, u[u != v], v[u != v])
    return gg.with_node_weights(gg.with_edge_weights(g, wmax), 3) if wmax > 1 else g


def _clique(n):
    i, j = np.triu_indices(n, 1)
    return gg.from_pairs(n, i, j)


# the classes end at 128, 512, 2048, 6144 and 18432 neighbours; a hub's chunks have 2048 entries
GRAPHS = {"star": star(2049), "edges": _hubs(9000, [128, 129, 512, 513, 2048, 2049, 6144, 6145, 8000], 9000, 1),
          "weighted": _hubs(40000, [39000, 18433, 18432, 12345, 2500, 2049], 20000, 50), "clique": _clique(2500)}


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("U", [3, 400])
def test_clustering_with_hubs(ctx, name, U):
    import paper_2504_17615_gb300 as gp
    g = GRAPHS[name]
    cmap, nc, st = ctx.gp_coarsen(gp.DeviceGraph.from_host(g), U, 1, 5, gp.default_config(**HOST_PATH))
    ocmap, onc, ost = orc.coarsen(g, U, 1, 5)
    assert nc == onc and np.array_equal(cmap.cpu().numpy(), ocmap)


# nodes that no cluster can have room for are left out: weights around the bound and around half of it, with
# and without light nodes to take in; the per-phase and the persistent path
@pytest.mark.parametrize("cfg", [HOST_PATH, {}])
@pytest.mark.parametrize("weights", [(1, 2, 20, 21, 38, 39, 40), (20, 21, 40), (21, 39, 40), (40,)])
def test_clustering_with_full_nodes(ctx, weights, cfg):
    import paper_2504_17615_gb300 as gp
    for name in ("edges", "star"):
        g = GRAPHS[name]
        vw = np.random.default_rng(len(weights)).choice(np.array(weights, dtype=g.vwgt.dtype), g.n)
        g = dataclasses.replace(g, vwgt=vw)
        cmap, nc, st = ctx.gp_coarsen(gp.DeviceGraph.from_host(g), 40, 1, 5, gp.default_config(**cfg))
        ocmap, onc, ost = orc.coarsen(g, 40, 1, 5)
        assert nc == onc and np.array_equal(cmap.cpu().numpy(), ocmap)
        assert (st.lp_moves, st.lp_subrounds, st.clusters_lp) == (ost.lp_moves, ost.lp_subrounds, ost.clusters_lp)


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("k", [2, 255, 256, 1024, 1025])
def test_refinement_with_hubs(ctx, name, k):
    import torch
    import paper_2504_17615_gb300 as gp
    g = GRAPHS[name]
    blk = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    lmax = int(np.bincount(blk, weights=g.vwgt, minlength=k).max()) + 2
    t = torch.from_numpy(blk.copy()).cuda()
    moves = ctx.gp_refine(gp.DeviceGraph.from_host(g), k, lmax, 1, 3, t, gp.default_config(**HOST_PATH))
    oblk, omoves = orc.refine(g, k, lmax, 1, 3, blk)
    assert moves == omoves and np.array_equal(t.cpu().numpy(), oblk)


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("nc", [1, 2, 7, 1500])
def test_contraction_of_long_segments(ctx, name, nc):
    import torch
    import paper_2504_17615_gb300 as gp
    g = GRAPHS[name]
    cmap = np.concatenate([np.arange(nc), np.random.default_rng(nc).integers(0, nc, g.n - nc)]).astype(np.int32)
    got = ctx.gp_contract(gp.DeviceGraph.from_host(g), torch.from_numpy(cmap).cuda(), nc).to_host()
    for a, b in zip(canon(got), canon(orc.contract(g, cmap, nc))):
        assert np.array_equal(a, b)
