"""Graphs of communities, in which most probes of the hub kernels match: their counts go
through sets in shared memory below the highest 16,383 ranks.  Around that many vertices and
around the longest list that a set takes (1,024 entries); exact."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from tests.gpu_util import assert_matches_oracle, gpu_run

pytestmark = pytest.mark.gpu
WINDOW = 16383


def _cliques(sizes, order=None, extra=0, seed=1):
    """Disjoint cliques, ids shuffled unless order is None, and a few random pairs."""
    rng = np.random.default_rng(seed)
    src, dst, base = [], [], 0
    for k in sizes:
        a, b = np.triu_indices(k, 1)
        src.append(a + base)
        dst.append(b + base)
        base += k
    src, dst = np.concatenate(src), np.concatenate(dst)
    if order is not None:
        p = np.random.default_rng(order).permutation(base)
        src, dst = p[src], p[dst]
    src = np.concatenate([src, rng.integers(0, base, extra)]).astype(np.int32)
    dst = np.concatenate([dst, rng.integers(0, base, extra)]).astype(np.int32)
    return base, src, dst


def _ring(n, k):
    a = np.repeat(np.arange(n, dtype=np.int64), k)
    return n, a.astype(np.int32), ((a + np.tile(np.arange(1, k + 1), n)) % n).astype(np.int32)


@pytest.mark.parametrize("n", [WINDOW - 1, WINDOW, WINDOW + 1, WINDOW + 9, 20_000])
@pytest.mark.parametrize("order", [None, 5])
def test_cliques_around_the_window(tc, n, order):
    k = 40
    sizes = [k] * (n // k) + ([n % k] if n % k else [])
    assert_matches_oracle(tc, *_cliques(sizes, order, extra=3000), device_io=True)


@pytest.mark.parametrize("sizes", [[1100] * 2 + [36] * 420, [36] * 420 + [1024, 1025, 1026], [300] * 20 + [33] * 350])
def test_long_lists(tc, sizes):
    """t(v) = C(k - 1, 2) in a clique of k; lists of more entries than a set takes."""
    n, s, d = _cliques(sizes)
    T, t, lcc, _ = gpu_run(tc, n, s, d, device_io=True)
    want = np.concatenate([np.full(k, (k - 1) * (k - 2) // 2, np.uint64) for k in sizes])
    np.testing.assert_array_equal(t, want)
    assert T == int(want.sum()) // 3
    assert (lcc == 1.0).all()


@pytest.mark.parametrize("kw", [{"strategies": {"hub": ("probe", 1.0)}}, {"tuning": {"hub_core": 0}},
                                {"tuning": {"hub_big_in": 1}}, {"tuning": {"hub_big_in": 4096}},
                                {"tuning": {"hub_min_degree": 1}}, {"tuning": {"hub_max": 9000}}])
def test_settings(tc, kw):
    n, s, d = _ring(24_000, 24)
    ref = oracle.triangles(n, s, d)
    assert_matches_oracle(tc, n, s, d, ref=ref, **kw)


def test_below_three_windows(tc):
    """Hubs in all three windows: 150,000 vertices, all of degree 40."""
    assert_matches_oracle(tc, *_ring(150_000, 20), device_io=True)


@pytest.mark.parametrize("nshards", [1, 3])
def test_shards_and_counts_anew(tc, nshards):
    n, s, d = _cliques([60] * 330, 9, extra=2000)
    ref = oracle.triangles(n, s, d)
    with tc.Graph.from_edges(n, s, d) as g:
        for _ in range(2):
            parts = [g.count_shard(k, nshards) for k in range(nshards)]
            assert sum(p[0] for p in parts) == ref["T"]
            np.testing.assert_array_equal(sum(p[1] for p in parts), ref["t"])
            assert g.count() == ref["T"]
            np.testing.assert_array_equal(g.lcc()[0], ref["t"])


def test_batch(tc):
    from tests.test_gpu_batch import _check
    _check(tc, [_cliques([70] * 60, k, extra=100, seed=k) for k in range(5)], True)
