"""GPU vs CPU oracle, exact: paths that only very large graphs take, reached on small ones by lowering the sizes
at which a context takes them."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import graphgen as gg
import oracle as orc
from tests.test_gpu_hubs import GRAPHS
from tests.test_gpu_parity import HOST_PATH, canon

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


def limits(ctx, hash_collect=16384, table_slack=16 << 20, tail_slack=4 << 20, few_nodes=72):
    ctx.lib.gp_test_limits(ctypes.c_void_p(ctx.ptr), ctypes.c_int32(hash_collect), ctypes.c_int64(table_slack),
                           ctypes.c_int64(tail_slack), ctypes.c_int32(few_nodes))


# edges of one weight that share a hash prefix: with a limit of 16384 one digit is read, with 64 or 1 one or two,
# with 0 all six
@pytest.mark.parametrize("limit", [0, 1, 3, 64])
@pytest.mark.parametrize("name", ["one_weight", "weights", "rmat"])
def test_exact_sampler_digits(ctx, limit, name):
    import paper_2504_17615_gb300 as gp
    g = {"one_weight": lambda: gg.er(20000, 300000, 5), "weights": lambda: gg.with_edge_weights(gg.er(9000, 90000, 6), 4),
         "rmat": lambda: gg.rmat(13, 16, seed=4)}[name]()
    dg = gp.DeviceGraph.from_host(g)
    limits(ctx, hash_collect=limit)
    for m_hat in (1, 2, g.m // 20 + 1, g.m // 2, g.m * 2 // 3, g.m - 1):
        out, st = ctx.gp_sparsify(dg, m_hat, 3, 9, 3)
        exp, ost = orc.sparsify(g, m_hat, 3, 9, 3)
        got = out.to_host()
        assert got.m == m_hat and st.threshold == ost.threshold
        assert np.array_equal(got.xadj, np.asarray(exp.xadj)) and np.array_equal(got.adjncy, np.asarray(exp.adjncy))
        assert np.array_equal(got.adjwgt, np.asarray(exp.adjwgt))


def _slack(m2, keys, tables, q4):
    """Bytes that let `tables` tables of `keys` keys in all have q4 quarters of a slot a key, and not more; q4 = 0:
    no such tables."""
    return -8 * m2 if q4 == 0 else 8 * (keys * q4 // 4 + tables) - 8 * m2


# hub tables of 3, 2.5, 2 and 1.5 slots a neighbour, and none: the hubs of more than 18432 neighbours then take a
# block each (refinement with few labels counts them per label unless even that is too much)
@pytest.mark.parametrize("q4", [12, 10, 8, 6, 0])
def test_hub_tables(ctx, q4):
    import torch
    import paper_2504_17615_gb300 as gp
    g = GRAPHS["weighted"]
    deg = np.diff(np.asarray(g.xadj))
    hubs = deg[deg > 18432]
    assert len(hubs) >= 2
    limits(ctx, table_slack=_slack(2 * g.m, int(hubs.sum()), len(hubs), q4))
    dg = gp.DeviceGraph.from_host(g)
    cmap, nc, st = ctx.gp_coarsen(dg, 400, 1, 5, gp.default_config(**HOST_PATH))
    ocmap, onc, ost = orc.coarsen(g, 400, 1, 5)
    assert nc == onc and np.array_equal(cmap.cpu().numpy(), ocmap)
    for k in (2, 300, 1025):
        blk = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
        lmax = int(np.bincount(blk, weights=g.vwgt, minlength=k).max()) + 2
        for cfg in (HOST_PATH, {}):
            t = torch.from_numpy(blk.copy()).cuda()
            moves = ctx.gp_refine(dg, k, lmax, 1, 3, t, gp.default_config(**cfg))
            oblk, omoves = orc.refine(g, k, lmax, 1, 3, blk)
            assert moves == omoves and np.array_equal(t.cpu().numpy(), oblk)


# segments above 2048 entries: tables of 2, 1.75, 1.5 and 1.25 slots a key, and a block a segment
@pytest.mark.parametrize("q4", [8, 7, 6, 5, 0])
@pytest.mark.parametrize("name,nc", [("weighted", 7), ("weighted", 5000), ("clique", 1500)])
def test_segment_tables(ctx, name, nc, q4):
    import torch
    import paper_2504_17615_gb300 as gp
    g = GRAPHS[name]
    cmap = np.concatenate([np.arange(nc), np.random.default_rng(nc).integers(0, nc, g.n - nc)]).astype(np.int32)
    seg = np.bincount(cmap, weights=np.diff(np.asarray(g.xadj)), minlength=nc).astype(np.int64)
    long = np.minimum(seg[seg > 2048], nc)
    assert len(long) > 0
    limits(ctx, table_slack=_slack(2 * g.m, int(long.sum()), len(long), q4))
    got = ctx.gp_contract(gp.DeviceGraph.from_host(g), torch.from_numpy(cmap).cuda(), nc).to_host()
    for a, b in zip(canon(got), canon(orc.contract(g, cmap, nc))):
        assert np.array_equal(a, b)


def _levels(ctx, g, k, **kw):
    """Levels of a partition (checked against the oracle) and how many of them were contracted on their own, not
    among the one-CTA levels."""
    import paper_2504_17615_gb300 as gp
    dg = gp.DeviceGraph.from_host(g)
    ctx.profile_reset()
    ctx.profile(True)
    blocks, cut, st = ctx.gp_partition(dg, k, 0.03, 3, gp.default_config(**kw))
    ctx.profile(False)
    r = orc.partition(g, k, 0.03, 3, orc.Config.default(**{a: b for a, b in kw.items() if a != "small_lp_nodes"}))
    assert cut == r.cut and np.array_equal(blocks.cpu().numpy(), r.blocks) and st.levels == r.stats.levels
    return st.levels, ctx.profile_read()["contract"]["launches"]


# 4608 nodes and 49152 entries are the limits; persistent launches switched off take the one-CTA levels with them.
# 321 nodes have a cluster bound of 1: nothing merges, and the level is discarded where it was tried
@pytest.mark.parametrize("n,m,kw,tail", [(321, 500, {}, True), (4608, 24576, {}, True), (4609, 20000, {}, False),
                                         (4600, 24577, {}, False), (4600, 20000, {"small_lp_nodes": 1000}, False)])
def test_one_cta_levels_run(ctx, n, m, kw, tail):
    levels, alone = _levels(ctx, gg.er(n, m, 6), 2, max_levels=1, **kw)
    assert levels == (0 if n == 321 else 1) and alone == (0 if tail else 1)


def test_one_cta_levels_below_the_limits(ctx):
    levels, alone = _levels(ctx, gg.er(30000, 90000, 6), 2)
    assert 0 < alone < levels


# the arena for the way down, and for the way down but not for the way up
@pytest.mark.parametrize("slack", [-10 ** 9, -1500000, -1000000, -700000, -500000, -250000, 0])
def test_one_cta_levels_without_room(ctx, slack):
    limits(ctx, tail_slack=slack)
    levels, alone = _levels(ctx, gg.with_edge_weights(gg.er(4000, 20000, 2), 3), 3)
    assert levels > 0 and (alone > 0 if slack < -10 ** 8 else alone <= levels)
