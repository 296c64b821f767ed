"""GPU vs CPU oracle, exact: whole partitions whose hierarchies end in the one-CTA tail, on both sides of
its size limits and started at the input or below it, and configurations that leave it out."""
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


def _check(ctx, g, k, **kw):
    import paper_2504_17615_gb300 as gp
    blocks, cut, st = ctx.gp_partition(gp.DeviceGraph.from_host(g), k, 0.03, 3, gp.default_config(**kw))
    r = orc.partition(g, k, 0.03, 3, orc.Config.default(**{a: b for a, b in kw.items() if a != "small_lp_nodes"}))
    assert cut == r.cut and np.array_equal(blocks.cpu().numpy(), r.blocks)
    assert st.levels == r.stats.levels and st.ip_cut == r.stats.ip_cut
    for i in range(st.levels):
        assert st.lv[i].clusters_final == r.stats.lv[i].clusters_final and st.lv[i].m_next == r.stats.lv[i].m_next


# 4608 nodes and 49152 entries are the limits
@pytest.mark.parametrize("n,m", [(321, 500), (4608, 24576), (4609, 20000), (4600, 24577), (30000, 90000)])
@pytest.mark.parametrize("w", [1, 30])
def test_sizes(ctx, n, m, w):
    g = gg.er(n, m, 6)
    if w > 1:
        g = gg.with_node_weights(gg.with_edge_weights(g, w), 4)
    for k in (2, 5):
        _check(ctx, g, k)


@pytest.mark.parametrize("kw", [{"sparsifier": 0}, {"sparsifier": 2}, {"sparsifier": 3}, {"ref_rounds": 0},
                                {"max_levels": 2}, {"max_levels": 0}, {"lp_subrounds": 3}, {"two_hop": 0, "isolated": 0},
                                {"dbg_max_subrounds": 5}, {"small_lp_nodes": 1000}], ids=str)
def test_configurations(ctx, kw):
    _check(ctx, gg.with_edge_weights(gg.er(4000, 20000, 2), 3), 3, **kw)


@pytest.mark.parametrize("name", ["star", "grid", "iso", "rmat"])
def test_shapes(ctx, name):
    g = {"star": lambda: star(4000), "grid": lambda: gg.grid2d(61, 67), "rmat": lambda: gg.rmat(12, 5, seed=9),
         "iso": lambda: gg.with_isolated(gg.er(2500, 6000, 4), 1500)}[name]()
    for k in (2, 7):
        _check(ctx, g, k)
