"""Shards whose plans hold only their own sources' hub records, through both record kernels,
every hub strategy and with and without the dense core, against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

N = 1 << 13
GRAPHS = {"rmat": (N, *graphgen.rmat(13, 24 * N, seed=6)), "er": (N + 1, *graphgen.er(N + 1, 10 * N, seed=7))}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("strategy", ["auto", "probe", "bitmap"])
@pytest.mark.parametrize("core,max_hubs,nshards", [(0, 131072, 3), (300, 131072, 4), (8192, 131072, 5), (0, 200, 3),
                                                   (0, 200, N + 2)])
def test_shards_of_every_plan(tc, name, strategy, core, max_hubs, nshards):
    n, s, d = GRAPHS[name]
    ref = oracle.triangles(n, s, d)
    with tc.Graph.from_edges(n, s, d) as g:
        g.set_tuning({**g.tuning(), "hub_core": core, "hub_max": max_hubs, "hub_min_degree": 1})
        g.set_strategy("hub", strategy)
        shards = range(nshards) if nshards < 10 else range(0, nshards, nshards // 9)
        parts = [g.count_shard(k, nshards) for k in shards]
        assert all(int(t.sum()) == 3 * T for T, t in parts)
        if nshards < 10:
            assert sum(T for T, _ in parts) == ref["T"]
            np.testing.assert_array_equal(sum(t for _, t in parts), ref["t"])
        assert g.count() == ref["T"]  # planned anew for all sources
        np.testing.assert_array_equal(g.lcc()[0], ref["t"])
