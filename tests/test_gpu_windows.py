"""The hub kernels' windows of ranks at their edges, against the oracle (exact).

Window 1 holds the 16,383 highest ranks, the two below it 65,535 each; a hub's in-edges
are cut into slices of 2,048; hubs of few in-edges take one warp, the others a block.
"""
from __future__ import annotations

from math import comb

import numpy as np
import pytest

import graphgen
import oracle
from tests.gpu_util import assert_matches_oracle

pytestmark = pytest.mark.gpu

HUBS = [(1, 1), (1, 64), (1, 1 << 30), (32, 128)]  # (degree of a hub, in-edges of a block's hub)


def _graph(n):
    """Uniform pairs with some heavy vertices: every rank can be a hub, rows reach every window."""
    s, d = graphgen.er_replace(n, 12 * n, seed=31, stream=n)
    hs = np.repeat(np.arange(0, n, max(1, n // 12), dtype=np.int32), n // 16 + 1)
    hd = (np.arange(hs.size, dtype=np.int64) * 7919 % n).astype(np.int32)
    return np.concatenate([s, hs]), np.concatenate([d, hd])


# around the end of window 1, of window 2, and past it (a third window below every hub)
@pytest.mark.parametrize("n", [33, 16382, 16383, 16384, 81917, 81919, 120_000])
def test_windows_match_the_oracle(tc, n):
    s, d = _graph(n)
    ref = oracle.triangles(n, s, d)
    for min_degree, big_in in HUBS:
        for core in (0, 8192):
            tuning = {"hub_min_degree": min_degree, "hub_big_in": big_in, "hub_core": core}
            assert_matches_oracle(tc, n, s, d, ref=ref, device_io=True, tuning=tuning)


@pytest.mark.parametrize("n", [16384, 100_000])
def test_support_in_every_window(tc, n):
    s, d = _graph(n)
    ru, rv, rs = oracle.edge_support(n, s, d)
    order = np.lexsort((rv, ru))
    with tc.Graph.from_edges(n, s, d) as g:
        for min_degree, big_in in HUBS:
            g.set_tuning({**g.tuning(), "hub_min_degree": min_degree, "hub_big_in": big_in})
            u, v, sup = g.edge_support()
            np.testing.assert_array_equal(u, ru[order])
            np.testing.assert_array_equal(v, rv[order])
            np.testing.assert_array_equal(sup, rs[order])
        assert g.count() == int(rs.sum()) // 3  # the support's plan serves the count


@pytest.mark.parametrize("k", [2047, 2049, 2300])
def test_in_edges_of_one_and_two_slices(tc, k):
    """A complete graph, whose highest hub has k - 1 in-edges and whose rows are long."""
    s, d = np.triu_indices(k, 1)
    with tc.Graph.from_edges(k, s.astype(np.int32), d.astype(np.int32)) as g:
        for core in (0, 1000):
            g.set_tuning({**g.tuning(), "hub_core": core})
            assert g.count() == comb(k, 3)
            t, lcc = g.lcc()
            assert (t == comb(k - 1, 2)).all() and (lcc == 1.0).all()
        assert (g.edge_support()[2] == k - 2).all()
