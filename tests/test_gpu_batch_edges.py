"""Batches whose graphs begin and end anywhere in a warp's share of the pairs, and the rule
that leaves out hubs, against the oracle graph by graph (exact)."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
from tests import families as F
from tests.test_gpu_batch import _check, _pack

pytestmark = pytest.mark.gpu


def _er(n, m, seed):
    return (n, *graphgen.er_replace(n, m, seed=seed))


EMPTY = (0, np.array([], np.int32), np.array([], np.int32))


@pytest.mark.parametrize("sizes", [[1], [255], [256], [257], [0, 0, 256, 0, 255, 1, 0], [31, 33, 192, 257, 0, 0, 2047],
                                   [1] * 700, [0] * 300 + [5000] + [0] * 300])
def test_boundaries_inside_a_warps_pairs(tc, sizes):
    _check(tc, [_er(40, m, i) if m else EMPTY for i, m in enumerate(sizes)], True)


@pytest.mark.parametrize("at", [0, 254, 255, 256, 511, 512, 799])
def test_an_id_of_the_next_graph_is_refused(tc, at):
    import torch
    n, off, s, d = _pack([_er(30, 255, 1), EMPTY, _er(30, 257, 2), _er(30, 288, 3)])
    s[at] = 30
    with tc.Graph.batch(n, off, torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()) as g:
        with pytest.raises(tc.TCError) as err:
            g.batch_count()
        assert err.value.status == tc.TC_EINVAL


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("hubs", [None, (8, 131072)])
def test_hubs_out_of_reach(tc, order, hubs):
    """A dense graph before (order 0: hubs left out unless set) or after a large sparse one."""
    import oracle
    graphs = [_er(1500, 60000, 5), (140000, *F.wheel(3000)[1])]
    if order:
        graphs.reverse()
    n, off, s, d = _pack(graphs)
    with tc.Graph.batch(n, off, s, d) as g:
        if hubs:
            g.set_hubs(*hubs)
        T = g.batch_count()
        t, _ = g.lcc()
    refs = [oracle.triangles(*x) for x in graphs]
    assert [int(x) for x in T] == [r["T"] for r in refs]
    np.testing.assert_array_equal(t, np.concatenate([r["t"] for r in refs]))
