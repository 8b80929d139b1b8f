"""The build's one-block scans and ranks at their largest sizes, and its table of dropped
repeats, against the oracle (exact)."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle
from tests.gpu_util import assert_matches_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1023, 1024, 1025, 8191, 8192, 8193, 16383, 16384, 16385])
def test_one_block_sizes(tc, n):
    s, d = graphgen.er(n, 6 * n, seed=n)
    hub = np.arange(1, min(n, 1500), dtype=np.int32)  # a degree past every narrow count
    s, d = np.concatenate([s, np.zeros_like(hub)]), np.concatenate([d, hub])
    assert_matches_oracle(tc, n, s, d, device_io=True)


@pytest.mark.parametrize("n", [(1 << 21) - 1, 1 << 21, (1 << 21) + 1])
def test_scan_over_a_thousand_tiles(tc, n):
    s, d = graphgen.er(n, 1 << 20, seed=8)
    assert_matches_oracle(tc, n, s, d, device_io=True)


@pytest.mark.parametrize("n,hubs,per", [(4000, 1, 3), (4000, 1500, 6), (3000, 3, 300)])
def test_repeats_at_hubs(tc, n, hubs, per):
    """A symmetric CSR drops each pair once, at hubs more often than a block's table has
    slots for; one row repeats its entries."""
    rng = np.random.default_rng(n + hubs)
    s = np.repeat(np.arange(n), per)
    d = np.where(rng.random(n * per) < 0.7, rng.integers(0, hubs, n * per), rng.integers(0, n, n * per))
    s, d = np.concatenate([s, d, np.full(400, 5)]), np.concatenate([d, s, np.full(400, 9)])
    order = np.lexsort((d, s))
    s, d = s[order].astype(np.int32), d[order].astype(np.int32)
    off = np.zeros(n + 1, np.int64)
    off[1:] = np.cumsum(np.bincount(s, minlength=n))
    ref = oracle.triangles(n, s, d)
    for device_io in (False, True):
        assert_matches_oracle(tc, n, s, d, ref=ref, csr=(off, d), device_io=device_io)


@pytest.mark.parametrize("m", [8191, 8192, 8193, 40000])
@pytest.mark.parametrize("n", [2, 300, 4097, 70001])
def test_bucket_fill_over_batches(tc, n, m):
    """Batches fill their rows by buckets: tiles of 8192 pairs that end anywhere, buckets of
    one row and more, every pair of a tile in one bucket."""
    s, d = graphgen.er_replace(n, m, seed=m)
    one = np.zeros(m, np.int32)
    sizes = np.array([n, 2, n], np.int32)
    off = np.array([0, m, 2 * m, 3 * m], np.int64)
    with tc.Graph.batch(sizes, off, np.concatenate([s, one, d]), np.concatenate([d, one + 1, s])) as g:
        T = g.batch_count()
        t, _ = g.lcc()
    ref = oracle.triangles(n, s, d)
    assert [int(x) for x in T] == [ref["T"], 0, ref["T"]]
    np.testing.assert_array_equal(t, np.concatenate([ref["t"], [0, 0], ref["t"]]))


@pytest.mark.parametrize("n,skewed", [(2000, False), (257, True), (300, True), (4097, True), ((1 << 20) - 1, True),
                                      (1 << 20, True), ((1 << 20) + 1, True), ((1 << 20) + 8193, True)])
def test_bucket_fill_of_large_graphs(tc, n, skewed):
    """Rows filled by buckets, even ones and those for skewed degrees at the edges of their
    sizes: half of the pairs at one vertex, some of them repeated."""
    m = 1 << 20
    s, d = graphgen.er_replace(n, m, seed=n)
    if skewed:
        s[::2] = 0
        s[1:4000:2], d[1:4000:2] = n - 1, n - 2
    assert_matches_oracle(tc, n, s, d, device_io=True)


@pytest.mark.parametrize("k", [2, 8, 9, 16, 17, 32, 33, 256, 257, 1025])
@pytest.mark.parametrize("hubs", [(32, 131072), (1, 0)])
def test_lists_filled_to_their_bound(tc, k, hubs):
    """Every source has exactly k entries, so that the planner's list of its class, and the
    sorters' lists, hold as many rows as the pairs allow."""
    sources, heavy = 300, k + 40
    rng = np.random.default_rng(k)
    s = np.repeat(np.arange(sources), k)
    d = sources + np.concatenate([rng.permutation(heavy)[:k] for _ in range(sources)])
    assert_matches_oracle(tc, sources + heavy, s.astype(np.int32), d.astype(np.int32), hubs=hubs, device_io=True)
