"""The dense core's bit rows at the edges of words, lanes and blocks, against the oracle
(exact): every vertex a hub, the core the highest hub_core ranks of them."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle
from tests.gpu_util import assert_matches_oracle

pytestmark = pytest.mark.gpu

N = 9000


@pytest.fixture(scope="module")
def graph():
    s, d = graphgen.rmat(14, 20 * N, seed=12, n=N)
    k = np.arange(40, dtype=np.int32)  # a clique among low ids, so that rows are dense somewhere
    s, d = np.concatenate([s, np.repeat(k, 40)]), np.concatenate([d, np.tile(k, 40)])
    return s, d, oracle.triangles(N, s, d), oracle.edge_support(N, s, d)


@pytest.mark.parametrize("core", [2, 31, 32, 33, 127, 128, 129, 255, 256, 257, 4095, 4097, 8191, 8192])
def test_core_sizes_match_the_oracle(tc, graph, core):
    s, d, ref, (ru, rv, rs) = graph
    tuning = {"hub_min_degree": 0, "hub_core": core}
    assert_matches_oracle(tc, N, s, d, ref=ref, device_io=True, tuning=tuning)
    with tc.Graph.from_edges(N, s, d) as g:
        g.set_tuning({**g.tuning(), **tuning})
        u, v, sup = g.edge_support()
    order = np.lexsort((rv, ru))
    np.testing.assert_array_equal(u, ru[order])
    np.testing.assert_array_equal(v, rv[order])
    np.testing.assert_array_equal(sup, rs[order])
