"""The hash-set kernels of the small bucket at the edges of their classes (sources of 2..8,
9..16, 17..32 and 33..256 entries below the hubs), against the oracle (exact)."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle
from tests.gpu_util import assert_matches_oracle

pytestmark = pytest.mark.gpu

BASE = 800


def _clique(k):
    i, j = np.triu_indices(k + 1, 1)  # rows of k, k - 1, ..., 0 entries
    return k + 1, i.astype(np.int32), j.astype(np.int32)


def _fringe(k):
    """Sources of k entries over a dense part whose rows are far longer: the edges a lane
    searches by itself, next to those that are probed."""
    rng = np.random.default_rng(k)
    s, d = np.nonzero(np.triu(rng.random((BASE, BASE)) < 0.5, 1))
    fs = np.repeat(np.arange(300), k) + BASE
    fd = np.concatenate([rng.choice(BASE, k, replace=False) for _ in range(300)])
    return BASE + 300, np.concatenate([s, fs]).astype(np.int32), np.concatenate([d, fd]).astype(np.int32)


GRAPHS = {f"clique {k}": _clique(k) for k in (2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 64, 255, 256, 257)}
GRAPHS |= {f"fringe {k}": _fringe(k) for k in (2, 8, 9, 16, 17, 32, 33, 256)}
GRAPHS["uniform"] = (20000, *graphgen.er(20000, 500000, seed=3))


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("max_hubs", [0, 40])
def test_classes_match_the_oracle(tc, name, max_hubs):
    n, s, d = GRAPHS[name]
    assert_matches_oracle(tc, n, s, d, device_io=True, hubs=(0, max_hubs))
    ru, rv, rs = oracle.edge_support(n, s, d)
    with tc.Graph.from_edges(n, s, d) as g:
        g.set_hubs(0, max_hubs)
        u, v, sup = g.edge_support()
    order = np.lexsort((rv, ru))
    np.testing.assert_array_equal(u, ru[order])
    np.testing.assert_array_equal(v, rv[order])
    np.testing.assert_array_equal(sup, rs[order])


def test_a_plan_is_counted_again(tc):
    """The kernels' work counters start anew with each count."""
    n, s, d = GRAPHS["uniform"]
    T = oracle.triangles(n, s, d)["T"]
    with tc.Graph.from_edges(n, s, d) as g:
        for strategy in ("hash", "merge", "hash"):
            g.set_strategy("small", strategy, 1.0)
            assert g.count() == T
