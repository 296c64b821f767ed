"""GPU vs exact recomputation: the kernels that split the CSR entries evenly over warps, on graphs
whose rows are far longer than a warp's share, with long runs of empty rows, and of sizes around the
edges of windows and shares."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle as orc
from tests._util import star
from tests.test_gpu_parity import canon

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


def _hubs_and_gaps():
    """Two hubs of 30000 and 5000 neighbours, a path, and thousands of empty rows in between."""
    n = 90001
    u = [np.zeros(30000, np.int64), np.full(5000, n - 1), np.arange(70000, 70500)]
    v = [np.arange(20000, 50000), np.arange(15000, 20000), np.arange(70001, 70501)]
    return gg.with_edge_weights(gg.from_pairs(n, np.concatenate(u), np.concatenate(v)), 9)


GRAPHS = {"one_edge": gg.from_pairs(2, [0], [1]), "path33": gg.grid2d(33, 1), "star": star(40000),
          "gaps": _hubs_and_gaps(), "er": gg.with_edge_weights(gg.er(2049, 16385, 3), 6),
          "rmat": gg.rmat(13, 16, seed=4)}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_walks(ctx, name):
    import torch
    import paper_2504_17615_gb300 as gp
    g = GRAPHS[name]
    dg = gp.DeviceGraph.from_host(g)
    rng = np.random.default_rng(5)
    for k in (2, 40, 300, 3000):  # one-byte and wide blocks, volumes in shared and in global memory
        blk = rng.integers(0, k, g.n).astype(np.int32)
        t = torch.from_numpy(blk).cuda()
        assert ctx.gp_cut(dg, t, k)[0] == orc.cut(g, blk)
        st, M = ctx.gp_modularity(dg, t, k), orc.modularity(g, blk, k)
        assert (st.w_internal, st.w_total, st.vol_max, st.vol_sq) == (M.w_internal, M.w_total, M.vol_max, M.vol_sq)
    nc = max(1, g.n // 3)
    cmap = rng.permutation(np.concatenate([np.arange(nc), rng.integers(0, nc, g.n - nc)])).astype(np.int32)
    got, exp = ctx.gp_contract(dg, torch.from_numpy(cmap).cuda(), nc).to_host(), orc.contract(g, cmap, nc)
    for a, b in zip(canon(got), canon(exp)):
        assert np.array_equal(a, b)
    for mode in (1, 2, 3):
        got, exp = ctx.gp_sparsify(dg, g.m // 2, 2, 7, mode)[0].to_host(), orc.sparsify(g, g.m // 2, 2, 7, mode)
        exp = exp[0] if isinstance(exp, tuple) else exp
        # kept entries stay in the order of the input's rows
        assert np.array_equal(got.xadj, np.asarray(exp.xadj)) and np.array_equal(got.adjncy, np.asarray(exp.adjncy))
        assert np.array_equal(got.adjwgt, np.asarray(exp.adjwgt))
