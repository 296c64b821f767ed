"""Graphs of 2^30 entries made on the device: counts that twice over no longer fit 32 bits."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def ring():
    """2^25 nodes, each joined to the 16 before and the 16 after it, the weight of an edge its distance."""
    import torch
    import paper_2504_17615_gb300 as gp
    n, d = 1 << 25, 16
    off = torch.cat([torch.arange(-d, 0), torch.arange(1, d + 1)]).cuda()
    adj = (torch.arange(n, device="cuda")[:, None] + off[None, :]) & (n - 1)
    adj = adj.to(torch.int32).reshape(-1).contiguous()
    w = off.abs().to(torch.int32).repeat(n).contiguous()
    xadj = (torch.arange(n + 1, device="cuda") * (2 * d)).to(torch.int32)
    torch.cuda.empty_cache()
    return gp.DeviceGraph(n, n * 2 * d, xadj, adj, torch.ones(n, dtype=torch.int32, device="cuda"), w)


# segments of 2^30, of 3/4 and of 1/2 of 2^30 entries; the arcs meet at two or three places, where
# 16 + 2 * 15 + .. of the ring's edges cross: sum d * d over the distances
@pytest.mark.parametrize("parts", [(1,), (3, 1), (2, 1, 1)])
def test_contraction_to_few_nodes(ctx, ring, parts):
    import torch
    total, nc = sum(parts), len(parts)
    cmap = torch.cat([torch.full((ring.n * p // total,), i, dtype=torch.int32) for i, p in enumerate(parts)]).cuda()
    got = ctx.gp_contract(ring, cmap, nc).to_host()
    cross = sum(x * x for x in range(1, 17))
    assert got.vwgt.tolist() == [ring.n * p // total for p in parts]
    assert got.xadj.tolist() == [0] + [(nc - 1) * (i + 1) for i in range(nc)]
    rows = [i for i in range(nc) for _ in range(nc - 1)]
    assert sorted(zip(rows, got.adjncy.tolist())) == [(i, j) for i in range(nc) for j in range(nc) if i != j]
    assert got.adjwgt.tolist() == [2 * cross if nc == 2 else cross] * len(rows)


# the centre's row, 2^29 + 2 entries, is rated within the eight sub-rounds; a cluster holds two nodes
def test_clustering_of_a_wide_star(ctx):
    import torch
    import paper_2504_17615_gb300 as gp
    leaves = (1 << 29) + 2
    n = leaves + 1
    adj = torch.zeros(2 * leaves, dtype=torch.int32, device="cuda")
    adj[:leaves] = torch.arange(1, n, dtype=torch.int32, device="cuda")
    xadj = torch.arange(leaves - 1, leaves + n, dtype=torch.int32, device="cuda")
    xadj[0] = 0
    one = torch.ones(2 * leaves, dtype=torch.int32, device="cuda")
    g = gp.DeviceGraph(n, 2 * leaves, xadj, adj, one[:n], one)
    cmap, nc, st = ctx.gp_coarsen(g, 2, 1, 5, gp.default_config(dbg_max_subrounds=8, two_hop=0))
    size = torch.zeros(nc, dtype=torch.int32, device="cuda").scatter_add_(0, cmap.long(), one[:n])
    assert st.lp_subrounds == 8 and 0 < st.lp_moves <= 16  # each sub-round: a leaf to the centre, the centre to a leaf
    assert int(size.min()) >= 1 and int(size.max()) == 2
    assert st.clusters_lp == st.clusters_final == nc and n - 9 <= nc < n
