"""Streams and events handed from destroyed graphs to new ones: several threads create,
count and destroy graphs of different sizes on streams of their own, before and after the
kept sets are given back."""
from __future__ import annotations

import threading

import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def test_threads_reuse_the_sets_of_destroyed_graphs(tc):
    import torch
    cases = []
    for i, n in enumerate((1, 700, 3000, 20_000)):
        s, d = graphgen.rmat(max(1, (n - 1).bit_length()), 9 * n, seed=40 + i, n=n)
        cases.append((n, s, d, oracle.triangles(n, s, d)))
    failures = []

    def work(k):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for j in range(12):
                    n, s, d, ref = cases[(j + k) % len(cases)]
                    host = (j + k) % 3 == 0
                    ss, dd = (s, d) if host else (torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda())
                    with tc.Graph.from_edges(n, ss, dd, stream) as g:
                        t, lcc = g.lcc()
                        assert g.count() == ref["T"]
                    np.testing.assert_array_equal(t, ref["t"])
                    np.testing.assert_array_equal(lcc, ref["lcc"])
        except BaseException as e:  # reported by the test's own thread
            failures.append(e)

    for _ in range(2):
        threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not failures, failures[0]
        torch.cuda.synchronize()
        tc.tc_release_cached_graphs()


def test_graph_destroyed_with_work_in_flight(tc):
    """The next graph takes the streams while the destroyed one's count still runs."""
    import torch
    n = 1 << 16
    s, d = graphgen.rmat(16, 16 * n, seed=8)
    ref = oracle.triangles(n, s, d)
    src, dst = torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()
    outs = []
    for _ in range(6):
        t = torch.empty(n, dtype=torch.int64, device="cuda")
        with tc.Graph.from_edges(n, src, dst) as g:
            g.lcc(t, torch.empty(n, dtype=torch.float64, device="cuda"))
        outs.append(t)
    torch.cuda.synchronize()
    for t in outs:
        np.testing.assert_array_equal(t.cpu().numpy().view(np.uint64), ref["t"])
