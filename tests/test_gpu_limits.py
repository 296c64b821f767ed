"""GPU vs CPU oracle, exact: paths that only very large graphs take, reached on small ones by lowering the sizes
at which a context takes them."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import graphgen as gg
import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


def limits(ctx, hash_collect=16384):
    ctx.lib.gp_test_limits(ctypes.c_void_p(ctx.ptr), ctypes.c_int32(hash_collect))


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
