"""GPU vs CPU oracle, exact: the initial partition in every form its growing kernel takes -- 32-bit and
64-bit node words, one-warp and four-warp steps, words in shared and in global memory, rows and row
bounds in shared memory or not, and fallbacks found by scans and from the hash order."""
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


def _check(ctx, g, k, seed):
    import paper_2504_17615_gb300 as gp
    got = ctx.gp_initial_partition(gp.DeviceGraph.from_host(g), k, 0.03, seed).cpu().numpy()
    assert np.array_equal(got, orc.initial_partition(g, k, 30000, seed))


# 1, 4 | 5, 9 nodes a step (one warp | four), the last 32-bit and the first 64-bit size, global memory;
# edge weights to 9 keep weighted degrees below 2^15, to 20000 they pass it
@pytest.mark.parametrize("n", [2, 63, 64, 65, 1023, 1024, 4095, 4096, 8200, 32767, 32768, 33000])
@pytest.mark.parametrize("wmax", [9, 20000])
def test_words_and_steps(ctx, n, wmax):
    g = gg.with_edge_weights(gg.er(n, min(4 * n, n * (n - 1) // 2), 3), wmax, n)
    _check(ctx, gg.with_node_weights(g, 5), 2 if n > 5000 else 5, n)


# many components: most steps find no frontier node (the hash order is made at the ninth fallback of a trial)
@pytest.mark.parametrize("n,m", [(40, 5), (900, 150), (6000, 900)])
@pytest.mark.parametrize("cmax", [1, 70000])
def test_fallbacks(ctx, n, m, cmax):
    g = gg.er(n, m, 8)
    if cmax > 1:  # weights beyond 16 bits, and nodes that stop fitting
        g = gg.with_node_weights(g, cmax if n < 20000 else 5)
    for k in (2, 3, 7):
        _check(ctx, g, k, k)
