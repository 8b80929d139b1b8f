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
    """The same graph in turn on one stream; each is destroyed before its outputs are done."""
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


def _lcc_without_waiting(tc, g, t, lcc):
    """lcc_compute itself: the binding's lcc() reads the graph's size, which waits."""
    assert tc.lib().lcc_compute(g.handle, t.data_ptr(), lcc.data_ptr(), tc.TC_MEM_DEVICE) == tc.TC_OK


def test_graphs_on_two_streams_destroyed_with_work_in_flight(tc):
    """Different graphs on two streams in turn; each is destroyed while its count runs, so the
    next one may find its streams and events busy, its memory free."""
    import torch
    cases = []
    for scale, seed in ((16, 8), (13, 9), (15, 10)):
        n = 1 << scale
        s, d = graphgen.rmat(scale, 16 * n, seed=seed)
        cases.append((n, torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda(), oracle.triangles(n, s, d)))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = []
    for k in range(12):
        n, src, dst, ref = cases[k % len(cases)]
        t = torch.empty(n, dtype=torch.int64, device="cuda")
        lcc = torch.empty(n, dtype=torch.float64, device="cuda")
        with tc.Graph.from_edges(n, src, dst, streams[k % 2]) as g:
            _lcc_without_waiting(tc, g, t, lcc)
        outs.append((t, lcc, ref))
    torch.cuda.synchronize()
    for t, lcc, ref in outs:
        np.testing.assert_array_equal(t.cpu().numpy().view(np.uint64), ref["t"])
        np.testing.assert_array_equal(lcc.cpu().numpy().view(np.uint64), ref["lcc"].view(np.uint64))


def test_a_graph_does_not_wait_for_a_destroyed_ones_stream(tc):
    import torch
    n = 1 << 13
    s, d = graphgen.rmat(13, 16 * n, seed=3)
    ref = oracle.triangles(n, s, d)
    src, dst = torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()
    t = torch.empty(n, dtype=torch.int64, device="cuda")
    lcc = torch.empty(n, dtype=torch.float64, device="cuda")
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    tc.tc_release_cached_graphs()
    with tc.Graph.from_edges(n, src, dst, two) as g:  # loads what a first call loads
        assert g.count() == ref["T"]
    torch.cuda.synchronize()
    tc.tc_release_cached_graphs()
    with tc.Graph.from_edges(n, src, dst, one) as g:
        with torch.cuda.stream(one):
            torch.cuda._sleep(1_500_000_000)  # most of a second
        _lcc_without_waiting(tc, g, t, lcc)
    with tc.Graph.from_edges(n, src, dst, two) as g:
        assert g.count() == ref["T"]
    assert not one.query()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(t.cpu().numpy().view(np.uint64), ref["t"])
