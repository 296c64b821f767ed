"""GPU vs CPU oracle (the per-graph path above 10,000 nodes), exact: the batched engine's initial partition in every form its growing trials take --
32-bit and 64-bit node words, words and chunk maxima in shared memory or in the arena, one and several nodes
a step, and fallbacks found by scans and from the hash order.  Nothing is coarsened, so every graph goes to
the bisection as it is."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle as orc

pytestmark = pytest.mark.gpu

COARSEST = {"coarsest_factor": 40000}


@pytest.fixture(scope="module")
def ctx():
    import paper_2504_17615_gb300 as gp
    from paper_2504_17615_gb300 import build
    build.build()
    c = gp.Context(0)
    yield c
    c.close()


def _check(ctx, graphs, threads):
    import paper_2504_17615_gb300 as gp
    ctx.batch_set_tuning(engine=1, threads=threads, max_entries=1 << 26, max_nodes=1 << 24, arena_bytes=128 << 20)
    res = ctx.gp_partition_batch([(gp.DeviceGraph.from_host(g), k, 0.03, s) for g, k, s in graphs],
                                 cfg=gp.default_config(**COARSEST), details=True)
    for (g, k, s), (blocks, cut, eng, st) in zip(graphs, res):
        if g.n <= 10000:
            r = orc.partition(g, k, 0.03, s, orc.Config.default(**COARSEST))
            want, want_cut = r.blocks, r.cut
        else:
            b, want_cut, _ = ctx.gp_partition(gp.DeviceGraph.from_host(g), k, 0.03, s, gp.default_config(**COARSEST))
            want = b.cpu().numpy()
        assert eng and st.levels == 0
        assert cut == want_cut, (g.name, k)
        assert np.array_equal(blocks.cpu().numpy(), want), (g.name, k)


# edge weights to 9 keep weighted degrees below 2^15, to 20000 they pass it; 50000 wide nodes: the chunk
# maxima of 64-bit words outgrow a warp's share of the 256-thread engine's shared memory
@pytest.mark.parametrize("wmax", [9, 20000])
@pytest.mark.parametrize("threads", [256, 512, 1024])
def test_words_and_steps(ctx, threads, wmax):
    graphs = []
    for n in (2, 63, 64, 65, 1023, 1024, 1025, 2100, 8200, 32767, 32768, 50000):
        g = gg.with_edge_weights(gg.er(n, min(3 * n, n * (n - 1) // 2), 3), wmax, n)
        graphs.append((gg.with_node_weights(g, 5), 5 if 2 < n < 5000 else 2, n))
    _check(ctx, graphs, threads)


# many components: most steps find no frontier node (the hash order is made at the ninth fallback of a trial)
@pytest.mark.parametrize("cmax", [1, 70000])
def test_fallbacks(ctx, cmax):
    graphs = []
    for n, m in ((40, 5), (900, 150), (6000, 900)):
        g = gg.er(n, m, 8)
        if cmax > 1:  # nodes that stop fitting
            g = gg.with_node_weights(g, cmax)
        graphs += [(g, k, k) for k in (2, 3, 7)]
    _check(ctx, graphs, 512)


# without a tuning: small items on the engine, large ones by the predicted time in a CTA, results as single calls
def test_untuned_split():
    import paper_2504_17615_gb300 as gp
    c = gp.Context(0)
    graphs = [(gp.DeviceGraph.from_host(gg.er(n, 10 * n, n)), k, 0.03, n)
              for n in (1000, 1638, 1639, 4000, 30000, 60000) for k in (2, 64)]
    graphs.append((gp.DeviceGraph.from_host(gg.rmat(16, 16, seed=2)), 8, 0.03, 1))
    res = c.gp_partition_batch(graphs, details=True)
    assert all(r[2] for r, j in zip(res, graphs) if j[0].m2 <= 1 << 15)
    assert not all(r[2] for r in res)
    for (blocks, cut, _, _), (g, k, eps, seed) in zip(res, graphs):
        want, want_cut, _ = c.gp_partition(g, k, eps, seed)
        assert cut == want_cut and np.array_equal(blocks.cpu().numpy(), want.cpu().numpy())
    c.close()
