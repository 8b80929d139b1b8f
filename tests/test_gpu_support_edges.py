"""Per-edge support where the hub kernels share their work out: big hubs with lists below the
highest 16,383 ranks of about 64 and of more than 256 entries, vectors that start anywhere in
a row, and core rows whose ranges do not overlap; exact, by closed forms and the vertex counts."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from tests.test_gpu_communities import _cliques

pytestmark = pytest.mark.gpu


def _support(tc, n, s, d):
    with tc.Graph.from_edges(n, s, d) as g:
        return g.edge_support()


@pytest.mark.parametrize("sizes", [[36] * 420 + [k] * 12 for k in (63, 64, 65, 66, 128, 131, 200, 300)])
@pytest.mark.parametrize("order", [None, 2])
def test_cliques(tc, sizes, order):
    """Every edge of a clique of k lies in k - 2 triangles."""
    n, s, d = _cliques(sizes, order)
    u, v, sup = _support(tc, n, s, d)
    lo, hi = np.minimum(s, d), np.maximum(s, d)
    o = np.lexsort((hi, lo))
    np.testing.assert_array_equal(u, lo[o])
    np.testing.assert_array_equal(v, hi[o])
    want = np.concatenate([np.full(k * (k - 1) // 2, k - 2) for k in sizes])
    np.testing.assert_array_equal(sup, want[o])


def _sums(n, u, v, sup):
    return (np.bincount(u, sup, n) + np.bincount(v, sup, n)).astype(np.uint64) // 2


@pytest.mark.parametrize("n,m", [(20_000, 2_000_000), (17_000, 600_000)])
def test_dense_uniform(tc, n, m):
    """Half the support over a vertex's edges is its t."""
    rng = np.random.default_rng(n)
    s, d = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    with tc.Graph.from_edges(n, s, d) as g:
        T = g.count()
        t, _ = g.lcc()
        u, v, sup = g.edge_support()
    assert int(sup.sum(dtype=np.uint64)) == 3 * T
    np.testing.assert_array_equal(_sums(n, u, v, sup), t)
    if m < 10**6:
        assert T == oracle.triangles(n, s, d)["T"]


@pytest.mark.parametrize("a,b", [(1, 40), (40, 40), (33, 700), (1000, 3000)])
@pytest.mark.parametrize("shuffled", [0, 1])
def test_bipartite_with_a_few_triangles(tc, a, b, shuffled):
    n = a + b
    s, d = np.repeat(np.arange(a), b), np.tile(np.arange(a, n), a)
    s, d = np.append(s, [a, 0]), np.append(d, [n - 1, a - 1])  # one edge within each side
    if shuffled:
        p = np.random.default_rng(a).permutation(n)
        s, d = p[s], p[d]
    s, d = s.astype(np.int32), d.astype(np.int32)
    ref = oracle.triangles(n, s, d)
    u, v, sup = _support(tc, n, s, d)
    assert int(sup.sum(dtype=np.uint64)) == 3 * ref["T"]
    np.testing.assert_array_equal(_sums(n, u, v, sup), ref["t"])
