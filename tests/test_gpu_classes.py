"""GPU vs CPU oracle, exact: the tests of the per-phase driver once more with a launch per degree class in every
sub-round, as on large graphs, instead of the classes of few nodes together."""
from __future__ import annotations

import pytest

from tests.test_gpu_hubs import test_clustering_with_hubs, test_refinement_with_hubs  # noqa: F401
from tests.test_gpu_limits import limits
from tests.test_gpu_parity import (test_coarsen_per_phase_driver_matches_oracle,  # noqa: F401
                                   test_lp_state_per_phase_driver, test_refine_per_phase_driver_matches_oracle)
from tests.test_gpu_rows import test_clustering_rows, test_refinement_rows  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gp():
    import paper_2504_17615_gb300 as gpmod
    from paper_2504_17615_gb300 import build
    build.build()
    return gpmod


@pytest.fixture(scope="module")
def ctx(gp):
    c = gp.Context(0)
    limits(c, few_nodes=0)
    yield c
    c.close()


def test_together_and_apart(gp, ctx):
    """The switch does what these tests rely on: apart takes more launches, and the result is the same."""
    import numpy as np
    import graphgen as gg
    g = gp.DeviceGraph.from_host(gg.rmat(12, 12, seed=3))
    got = []
    for few in (0, 72):
        limits(ctx, few_nodes=few)
        before = gp.launch_count()
        cmap, nc, st = ctx.gp_coarsen(g, 40, 1, 5, gp.default_config(small_lp_nodes=0))
        got.append((gp.launch_count() - before, nc, cmap.cpu().numpy()))
    limits(ctx, few_nodes=0)
    assert got[0][0] > got[1][0] and got[0][1] == got[1][1] and np.array_equal(got[0][2], got[1][2])
