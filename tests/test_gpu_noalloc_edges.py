"""tc_count_noalloc at the edges of its kernels, against the oracle (exact): rows of 32
and 33 entries (the sorting network and the bitmap), rows full of repeats, degrees at and
past the last bin of the rank sort, sizes at the limits."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def _stars(n, degrees):
    """Vertex i of the first ones joined to `degrees[i]` others, and a path through all."""
    s = [np.full(k, i) for i, k in enumerate(degrees)]
    d = [(i + 1 + np.arange(k)) % n for i, k in enumerate(degrees)]
    p = np.arange(n - 1)
    return np.concatenate(s + [p]).astype(np.int32), np.concatenate(d + [p + 1]).astype(np.int32)


def _cases():
    out = []
    rng = np.random.default_rng(5)
    for k in (31, 32, 33, 34, 65):  # dense blocks: rows of up to k - 1 entries
        s, d = np.triu_indices(k, 1)
        out.append((f"clique{k}", k + 3, s.astype(np.int32), d.astype(np.int32)))
    s, d = rng.integers(0, 40, (2, 5000)).astype(np.int32)
    out.append(("repeats", 41, s, d))
    out.append(("one_pair_often", 2, np.zeros(262144, np.int32), np.ones(262144, np.int32)))
    out.append(("bins", 4096, *_stars(4096, [1021, 1022, 1023, 1024, 1025, 2000, 4000, 1023])))
    out.append(("most_in_the_last_bin", 1300, *(x.astype(np.int32) for x in rng.integers(0, 256, (2, 262144)))))
    out.append(("n_limit", 16384, *graphgen.er_replace(16384, 262144, seed=3)))
    out.append(("n_limit_sparse", 16384, *graphgen.er_replace(16384, 100, seed=3)))
    out.append(("rmat_ragged", 3001, *graphgen.rmat(12, 30011, seed=9, n=3001)))
    out.append(("one_vertex", 1, np.zeros(3, np.int32), np.zeros(3, np.int32)))
    return out


@pytest.mark.parametrize("name,n,s,d", _cases(), ids=[c[0] for c in _cases()])
def test_noalloc_matches_the_oracle(tc, name, n, s, d):
    import torch
    ref = oracle.triangles(n, s, d)
    t = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    lcc = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    T = tc.tc_count_noalloc(n, torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda(), t, lcc)
    assert T == ref["T"]
    np.testing.assert_array_equal(t.cpu().numpy().view(np.uint64), ref["t"])
    np.testing.assert_array_equal(lcc.cpu().numpy().view(np.uint64), ref["lcc"].view(np.uint64))


def test_noalloc_leaves_the_outputs_when_an_id_is_bad(tc):
    import torch
    s = torch.tensor([0, 1, 4], dtype=torch.int32, device="cuda")
    t = torch.full((4,), -1, dtype=torch.int64, device="cuda")
    with pytest.raises(tc.TCError) as err:
        tc.tc_count_noalloc(4, s, s.roll(1), t)
    assert err.value.status == tc.TC_EINVAL
    assert (t == -1).all()


@pytest.mark.parametrize("n", [0, 1, 512, 513, 16384])
@pytest.mark.parametrize("outputs", [0, 1])
def test_noalloc_without_pairs_launches_nothing(tc, n, outputs):
    import torch
    none = torch.empty(0, dtype=torch.int32, device="cuda")
    t = torch.full((n,), -1, dtype=torch.int64, device="cuda") if outputs else None
    lcc = torch.full((n,), -1.0, dtype=torch.float64, device="cuda") if outputs else None
    before = tc.tc_launch_count()
    assert tc.tc_count_noalloc(n, none, none, t, lcc) == 0
    assert tc.tc_launch_count() == before
    if outputs:
        assert (t == 0).all() and (lcc.view(torch.int64) == 0).all()
