"""The host code of the library (tc_api.cu) against a fake CUDA runtime: what it answers when
the device code raises a flag or a call of the runtime fails."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

from tests import fake_cuda

OK, EINVAL, ENOMEM, ECUDA, ETIMEOUT, EBUSY, EINTERNAL = range(7)
HOST, DEVICE = 0, 1
OVERFLOW = 4  # ERR_OVERFLOW: a guard of the build or of the plan has fired


@pytest.fixture(scope="session")
def fake_lib(tmp_path_factory):
    return fake_cuda.load(str(tmp_path_factory.mktemp("fake_cuda")))


@pytest.fixture
def fake(fake_lib):
    fake_lib.fake_reset()
    yield fake_lib
    fake_lib.fake_reset()


def _ptr(a):
    return a.ctypes.data if a is not None else None


def _pairs(m):
    return np.zeros(m, np.int32), np.ones(m, np.int32)


def _graph(fake, n=50, m=60, kind=DEVICE, stream=None):
    s, d = _pairs(m)
    g = ctypes.c_void_p()
    st = fake.tc_graph_create_from_edges(n, m, _ptr(s), _ptr(d), kind, stream, ctypes.byref(g))
    assert st == OK
    return g


def _batch(fake):
    n, off = np.array([30, 20], np.int32), np.array([0, 25, 60], np.int64)
    s, d = _pairs(60)
    g = ctypes.c_void_p()
    assert fake.tc_batch_create(2, _ptr(n), _ptr(off), _ptr(s), _ptr(d), DEVICE, None, ctypes.byref(g)) == OK
    return g


def _calls(fake, g, kind):
    """The calls that read a graph's results or statistics back, by name."""
    T, t, lcc = ctypes.c_uint64(), np.zeros(50, np.uint64), np.zeros(50)
    m = ctypes.c_int64()
    e = [np.zeros(60, np.int32) for _ in range(3)]
    cap = np.array([16], np.uint64)
    return {
        "tc_count": lambda: fake.tc_count(g, ctypes.byref(T)),
        "lcc_compute": lambda: fake.lcc_compute(g, ctypes.c_void_p(_ptr(t)), ctypes.c_void_p(_ptr(lcc)), HOST),
        "tc_count_shard": lambda: fake.tc_count_shard(g, 0, 2, None, HOST, ctypes.byref(T)),
        "tc_lcc_from_counts": lambda: fake.tc_lcc_from_counts(g, ctypes.c_void_p(_ptr(t)),
                                                              ctypes.c_void_p(_ptr(lcc)), HOST),
        "tc_count_vertex_formula": lambda: fake.tc_count_vertex_formula(g, ctypes.c_void_p(_ptr(t)), kind,
                                                                        ctypes.byref(T)),
        "tc_edge_support": lambda: fake.tc_edge_support(g, *(ctypes.c_void_p(_ptr(a)) for a in e), kind),
        "tc_remote_cache": lambda: fake.tc_remote_cache(g, 2, 1, ctypes.c_void_p(_ptr(cap)), None, None, None),
        "tc_graph_info": lambda: fake.tc_graph_info(g, ctypes.byref(m), None, None),
        "tc_graph_size": lambda: fake.tc_graph_size(g, None, ctypes.byref(m)),
    }


CALLS = ["tc_count", "lcc_compute", "tc_count_shard", "tc_lcc_from_counts", "tc_count_vertex_formula",
         "tc_edge_support", "tc_remote_cache", "tc_graph_info", "tc_graph_size"]


@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("flag", [0, OVERFLOW])
def test_a_guard_of_the_build_is_reported(fake, call, flag):
    """Rows that the partition could not fill are empty: every call that reads the graph back
    says so instead of answering from them."""
    fake.fake_flags(flag, 0)
    g = _graph(fake)
    try:
        f = _calls(fake, g, DEVICE)[call]
        for _ in range(2):
            assert f() == (EINTERNAL if flag else OK)
    finally:
        fake.tc_graph_destroy(g)


@pytest.mark.parametrize("flag", [0, OVERFLOW])
@pytest.mark.parametrize("during_build", [0, 1])
def test_a_guard_in_a_batch_is_reported(fake, flag, during_build):
    fake.fake_flags(flag if during_build else 0, 0 if during_build else flag)
    g = _batch(fake)
    try:
        T = np.zeros(2, np.uint64)
        for kind in (HOST, DEVICE):
            assert fake.tc_batch_count(g, ctypes.c_void_p(_ptr(T)), kind) == (EINTERNAL if flag else OK)
    finally:
        fake.tc_graph_destroy(g)


@pytest.mark.parametrize("flag", [0, OVERFLOW])
@pytest.mark.parametrize("dir_bits", [0, 1])
def test_a_guard_reaches_the_directed_count(fake, flag, dir_bits):
    fake.fake_flags(flag, 0)
    s, d = _pairs(60)
    assert fake.fake_undirected_rows(50, 60, _ptr(s), _ptr(d), dir_bits) == (EINTERNAL if flag else OK)


@pytest.mark.parametrize("call", ["tc_count", "lcc_compute"])
def test_a_guard_of_the_count_is_reported(fake, call):
    fake.fake_flags(0, OVERFLOW)
    g = _graph(fake)
    try:
        f = _calls(fake, g, DEVICE)[call]
        assert f() == EINTERNAL and f() == EINTERNAL
        T = ctypes.c_uint64()
        assert fake.tc_count(g, ctypes.byref(T)) == EINTERNAL
    finally:
        fake.tc_graph_destroy(g)


@pytest.mark.parametrize("n", [0, 50])
def test_timings_are_the_graphs_own(fake, n):
    """A graph without vertices runs no phases: no timing, whatever the events that it took
    over from a destroyed graph hold."""
    ms = (ctypes.c_float * 8)()
    T = ctypes.c_uint64()
    for size in (50, n):
        g = _graph(fake, n=size, m=60 if size else 0)
        assert fake.tc_count(g, ctypes.byref(T)) == OK
        for timing in (fake.tc_graph_last_timing, fake.tc_graph_build_timing):
            assert timing(g, ms, 8) == (OK if size else EINVAL)
        fake.tc_graph_destroy(g)


def _count(fake, g):
    T = ctypes.c_uint64()
    assert fake.tc_count(g, ctypes.byref(T)) == OK


def test_streams_are_handed_on_once_they_are_idle(fake):
    """A graph that is destroyed with work in flight leaves a busy second stream: the next one
    takes another, so that its work does not wait for the first graph's."""
    def side(k):
        g = _graph(fake)
        assert fake.lcc_compute(g, ctypes.c_void_p(_ptr(t)), None, DEVICE) == OK  # does not wait
        fake.tc_graph_destroy(g)
        return fake.fake_plan_side(k)

    t = np.zeros(50, np.uint64)

    first = side(0)
    assert first > 0 and side(1) == first
    fake.fake_busy(first, 1)
    second = side(2)
    assert second not in (0, first) and side(3) == second
    fake.fake_busy(second, 1)
    third = side(4)
    assert third not in (0, first, second)
    fake.fake_busy(first, 0)
    fake.fake_busy(third, 1)
    assert side(5) == first
    fake.tc_release_cached_graphs()
    assert fake.fake_live_streams() == 0 and fake.fake_live_events() == 0


def test_the_sets_kept_are_bounded(fake):
    streams, t = 0, np.zeros(50, np.uint64)
    for k in range(80):
        g = _graph(fake)
        assert fake.lcc_compute(g, ctypes.c_void_p(_ptr(t)), None, DEVICE) == OK
        fake.fake_busy(fake.fake_plan_side(k), 1)
        fake.tc_graph_destroy(g)
        streams = max(streams, fake.fake_live_streams())
    assert streams <= 2 * 65


@pytest.mark.parametrize("kind", [HOST, DEVICE])
@pytest.mark.parametrize("kth", [1, 2])
def test_one_stream_is_enough(fake, kind, kth):
    """Where a second stream cannot be created the work stays on the graph's own."""
    fake.fake_fail(b"stream", kth)
    g = _graph(fake, kind=kind)
    _count(fake, g)
    assert (fake.fake_plan_side(0) == 0) == (kth == 1)
    fake.tc_graph_destroy(g)
    g = _graph(fake, kind=kind)
    _count(fake, g)
    assert fake.fake_plan_side(1) != 0
    fake.tc_graph_destroy(g)


@pytest.mark.parametrize("kth", range(1, 20))
def test_nothing_is_lost_when_an_event_cannot_be_created(fake, kth):
    s, d = _pairs(60)
    g = ctypes.c_void_p()
    fake.fake_fail(b"event", kth)
    st = fake.tc_graph_create_from_edges(50, 60, _ptr(s), _ptr(d), HOST, None, ctypes.byref(g))
    assert st in (OK, ECUDA) and bool(g.value) == (st == OK)
    if st == OK:
        fake.tc_graph_destroy(g)
    fake.tc_release_cached_graphs()
    assert fake.fake_live_streams() == 0 and fake.fake_live_events() == 0 and fake.fake_bytes() == 0


MIB = 1 << 20


@pytest.mark.parametrize("n,m", [(1 << 20, 16 << 20), (1 << 23, 8 << 23), (1 << 23, 60_000_000), (1 << 22, 1 << 22),
                                 (100_000_000, 30_000_000), (400_000_000, 1 << 30), (1_500_000_000, (1 << 31) - 1),
                                 ((1 << 31) - 1, 1000), ((1 << 31) - 1, 500_000_000), (1000, (1 << 31) - 1)])
@pytest.mark.parametrize("directed", [0, 1])
def test_memory_of_a_build(fake, n, m, directed):
    """What a graph can have in pairs and vertices depends on the memory of its build: at most
    40 bytes a pair beside the input and 100 a vertex, and the arrays of a fixed size."""
    one = ctypes.c_void_p(64)  # never read here
    fake.fake_max_deg(100)
    if directed:
        assert fake.fake_undirected_rows(n, m, one, one, 0) == OK
    else:
        g = ctypes.c_void_p()
        assert fake.tc_graph_create_from_edges(n, m, one, one, DEVICE, None, ctypes.byref(g)) == OK
        # and what stays: the arrays of the count
        assert fake.fake_bytes() <= 32 * m + 130 * n + 64 * MIB
        fake.tc_graph_destroy(g)
    assert fake.fake_peak() <= 40 * m + 100 * n + 64 * MIB
