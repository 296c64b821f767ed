"""GPU vs exact recomputation: the kernels that walk all CSR entries, on graphs with far more nodes than entries and with
rows around the size up to which a warp's share takes them whole."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle as orc
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


def _rows(n, degs, gap, far):
    """Node i * gap has degs[i] neighbours from node `far` on."""
    u = np.concatenate([np.full(d, i * gap) for i, d in enumerate(degs)])
    v = np.concatenate([far + np.arange(d) for d in degs])
    return gg.with_edge_weights(gg.from_pairs(n, u, v), 5)


GRAPHS = {
    "few": gg.with_edge_weights(gg.er(300001, 40, 3), 4),
    "ends": gg.from_pairs(500000, [0, 1, 499998], [499999, 2, 499999]),
    "rows": _rows(70000, [127, 128, 129, 130, 500, 1, 128, 129], 33, 60000),
    "long": _rows(200000, [60000, 1, 129, 5000, 40000, 128, 3], 1, 100000),
    "late": _rows(120001, [129] * 300, 7, 119000),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_walks(ctx, name):
    import torch
    import paper_2504_17615_gb300 as gp
    g = GRAPHS[name]
    dg = gp.DeviceGraph.from_host(g)
    for mode in (1, 2, 3):
        for m_hat in (1, g.m // 2, g.m - 1):
            got, (exp, _) = ctx.gp_sparsify(dg, m_hat, 2, 7, mode)[0].to_host(), orc.sparsify(g, m_hat, 2, 7, mode)
            assert np.array_equal(got.xadj, np.asarray(exp.xadj)) and np.array_equal(got.adjncy, np.asarray(exp.adjncy))
            assert np.array_equal(got.adjwgt, np.asarray(exp.adjwgt))
    rng = np.random.default_rng(3)
    for k in (2, 300):
        blk = rng.integers(0, k, g.n).astype(np.int32)
        t = torch.from_numpy(blk).cuda()
        assert ctx.gp_cut(dg, t, k)[0] == orc.cut(g, blk)
        st, M = ctx.gp_modularity(dg, t, k), orc.modularity(g, blk, k)
        assert (st.w_internal, st.w_total, st.vol_max, st.vol_sq) == (M.w_internal, M.w_total, M.vol_max, M.vol_sq)
        t[g.n // 2] = k  # a label out of range on any node, with neighbours or not
        with pytest.raises(gp.GpError):
            ctx.gp_modularity(dg, t, k)
    nc = g.n // 3
    cmap = rng.permutation(np.concatenate([np.arange(nc), rng.integers(0, nc, g.n - nc)])).astype(np.int32)
    got, exp = ctx.gp_contract(dg, torch.from_numpy(cmap).cuda(), nc).to_host(), orc.contract(g, cmap, nc)
    for a, b in zip(canon(got), canon(exp)):
        assert np.array_equal(a, b)


# two passes and one prefix sum (three launches), also when rows lie in several shares
@pytest.mark.parametrize("name", ["few", "long"])
def test_launches_of_a_sparsification(ctx, name):
    import paper_2504_17615_gb300 as gp
    g = GRAPHS[name]
    dg = gp.DeviceGraph.from_host(g)
    before = gp.launch_count()
    ctx.gp_sparsify(dg, g.m // 2, 2, 7, 2)
    assert gp.launch_count() - before <= 5
