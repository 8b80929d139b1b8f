"""The directed count's queue of pushed entries and its hub kernel at the edges of their
groups, against the oracle (exact)."""
from __future__ import annotations

import numpy as np
import pytest

from tests.test_gpu_directed import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 31, 32, 33, 63, 64, 65, 127, 1000])
def test_pushed_entries(tc, m):
    """Few vertices of few in-edges: nothing is pulled."""
    rng = np.random.default_rng(m)
    n = max(4, m // 4)
    _check(tc, n, rng.integers(0, n, m), rng.integers(0, n, m), device_io=True)


@pytest.mark.parametrize("k", [33, 34, 40, 63, 64, 65, 72, 73, 128, 129, 300])
def test_cliques_with_hubs(tc, k):
    """Suffixes of every length up to k against hubs, each pair in one or both directions,
    next to sparse vertices whose entries are pushed."""
    rng = np.random.default_rng(k)
    i, j = np.triu_indices(k, 1)
    way = rng.integers(0, 3, len(i))
    s = np.concatenate([i[way != 1], j[way != 0], rng.integers(k, k + 500, 2000)])
    d = np.concatenate([j[way != 1], i[way != 0], rng.integers(0, k + 500, 2000)])
    _check(tc, k + 500, s, d)
