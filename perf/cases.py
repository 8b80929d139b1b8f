"""Performance cases of the triangle-count and LCC library.

Each case is one call sequence that a program makes through the package's public
entry points, on seeded synthetic graphs: R-MAT with (0.57, 0.19, 0.19, 0.05) and
uniform pairs with replacement, the two families of the benchmark and of the tests.

Kinds:
  edges    a device edge list to T, t[] and LCC[] (create, count, LCC, release)
  csr      the same from device CSR arrays that hold both directions of every edge
  host     the same from and to pinned host buffers
  batch    many small graphs in one call, per-graph T, t[] and LCC[]
  serve    a burst of requests through the serving loop
  noalloc  the no-allocation entry point for small graphs
  directed Eq. 1 on a directed edge list
  support  triangles per edge of a graph that the program keeps
  shard    one shard of the count of a graph that the program keeps

Every output is a whole number, or one correctly rounded IEEE division of two whole
numbers, so the results are unique and the tolerance is exact everywhere.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2202_13976_gb300 as tc

GAMMA = -0x61c8864680b583eb  # 0x9e3779b97f4a7c15 as a signed 64-bit number
MIX1 = -0x40a7b892e31b1a47   # 0xbf58476d1ce4e5b9
MIX2 = -0x6b2fb644ecceee15   # 0x94d049bb133111eb
MASK64 = (1 << 64) - 1
RMAT_CUTS = tuple(int(math.floor(p * 2 ** 32)) for p in (0.57, 0.57 + 0.19, 0.57 + 0.19 + 0.19))
MAX_PAIRS = 8 << 23          # pairs of the largest listed graph
SLOTS, BUDGET = 8, 120 << 30  # the serving loop as the benchmark runs it


def listed():
    return [
        # the smallest configuration of the benchmark: latency, launches and host work count
        {"name": "edges_er4096", "kind": "edges", "gen": "er", "n": 4096, "m": 32768},
        # real-time code that must not allocate: a graph of a few thousand vertices, ragged sizes
        {"name": "noalloc_rmat_3k", "kind": "noalloc", "gen": "rmat", "n": 3001, "m": 30011},
        # a graph of the middle of the serving range (log-uniform in [1,000, 4,000,000]),
        # given as the symmetric CSR that most graph programs hold; n is no power of two
        {"name": "csr_rmat_60k", "kind": "csr", "gen": "rmat", "n": 60001, "m": 600011},
        # the benchmark's medium scale-free graph
        {"name": "edges_rmat20", "kind": "edges", "gen": "rmat", "n": 1 << 20, "m": 16 << 20},
        # the benchmark's default workload, the largest single graph
        {"name": "edges_rmat23", "kind": "edges", "gen": "rmat", "n": 1 << 23, "m": 8 << 23},
        # the uniform graph of the same size: no hubs, no reuse of lists
        {"name": "edges_er23", "kind": "edges", "gen": "er", "n": 1 << 23, "m": 60_000_000},
        # data that lives on the host: edge list in, t[] and LCC[] out over the host link
        {"name": "host_rmat_2m", "kind": "host", "gen": "rmat", "n": 2_000_003, "m": 20_000_003},
        # the benchmark's batch (n log-uniform in [32, 65,536], half R-MAT, half uniform), 1,000 graphs of it
        {"name": "batch_1000", "kind": "batch", "graphs": 1000, "n_max": 65536},
        # a burst of requests of mixed sizes through the serving loop (70 % R-MAT)
        {"name": "serve_48", "kind": "serve", "requests": 48, "n_max": 1_000_000},
        # directed graphs, Eq. 1
        {"name": "directed_rmat_1m", "kind": "directed", "gen": "rmat", "n": 1_000_000, "m": 16_000_000},
        # triangles per edge (the k-truss input) of a kept graph
        {"name": "support_rmat20", "kind": "support", "gen": "rmat", "n": 1 << 20, "m": 16 << 20},
        # one rank's share of the count of a replicated graph, planned and counted anew
        {"name": "shard_rmat_3m", "kind": "shard", "gen": "rmat", "n": 3_000_000, "m": 24_000_000,
         "shard": 1, "nshards": 4},
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["edges", "edges", "edges", "csr", "host", "batch", "serve", "noalloc", "directed", "support",
                       "shard"])
    if kind == "batch":
        return {"kind": kind, "graphs": log_int(20, 1000), "n_max": log_int(4096, 65536)}
    if kind == "serve":
        return {"kind": kind, "requests": log_int(4, 48), "n_max": log_int(20_000, 1_000_000)}
    gen = "rmat" if rng.random() < 0.7 else "er"
    if kind == "noalloc":
        n = log_int(100, 16384)
        return {"kind": kind, "gen": gen, "n": n, "m": min(262144, int(rng.uniform(4, 16) * n))}
    top = {"edges": 1 << 23, "csr": 2_000_000, "host": 2_000_003, "directed": 1_000_000, "support": 1 << 20,
           "shard": 3_000_000}[kind]
    n = log_int(1000, top)
    cap = {"edges": MAX_PAIRS, "csr": 16 << 20, "host": 20_000_003, "directed": 16_000_000, "support": 16 << 20,
           "shard": 24_000_000}[kind]
    case = {"kind": kind, "gen": gen, "n": n, "m": min(cap, int(rng.uniform(4, 16) * n))}
    if kind == "shard":
        case["nshards"] = rng.choice([2, 3, 4, 8])
        case["shard"] = rng.randrange(case["nshards"])
    return case


# ---- inputs ----------------------------------------------------------------------
# Counter-based SplitMix64 in 64-bit integer tensors: the definition that the serving
# loop's requests are generated by, so that every kind of case takes its graphs from
# one generator.

def _mix_int(z):
    z = ((z ^ (z >> 30)) * 0xbf58476d1ce4e5b9) & MASK64
    z = ((z ^ (z >> 27)) * 0x94d049bb133111eb) & MASK64
    return z ^ (z >> 31)


def _stream_key(seed, stream):
    g = 0x9e3779b97f4a7c15
    key = _mix_int(_mix_int((seed + g) & MASK64) ^ (((stream + 1) * g) & MASK64))
    return key - (1 << 64) if key >> 63 else key


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _mix(z):
    z = (z ^ _shr(z, 30)) * MIX1
    z = (z ^ _shr(z, 27)) * MIX2
    return z ^ _shr(z, 31)


def _rmat_attempt(key, e, attempt, scale):
    row = torch.zeros_like(e)
    col = torch.zeros_like(e)
    base = (e * 64 + attempt) * 16
    x = None
    for level in range(scale):
        if level % 2 == 0:
            x = _mix((base + (level // 2 + 1)) * GAMMA + key)
            u = _shr(x, 32)
        else:
            u = x & 0xffffffff
        bit = 1 << (scale - 1 - level)
        a, ab, abc = RMAT_CUTS
        row += (u >= ab) * bit
        col += (((u >= a) & (u < ab)) | (u >= abc)) * bit
    return row, col


def _pairs(gen, n, m, seed, stream=0):
    """m pairs over n vertices as two int32 CUDA tensors."""
    src = torch.empty(m, dtype=torch.int32, device="cuda")
    dst = torch.empty(m, dtype=torch.int32, device="cuda")
    key = _stream_key(seed, stream)
    scale = max(1, (n - 1).bit_length())
    step = 1 << 23
    for first in range(0, m, step):
        e = torch.arange(first, min(m, first + step), dtype=torch.int64, device="cuda")
        if gen == "er":
            x = _mix((e + 1) * GAMMA + key)
            row, col = (_shr(x, 32) * n) >> 32, ((x & 0xffffffff) * n) >> 32
        else:
            row, col = _rmat_attempt(key, e, 0, scale)
            for attempt in range(1, 64):
                bad = ((row >= n) | (col >= n)).nonzero().squeeze(1)
                if bad.numel() == 0:
                    break
                row[bad], col[bad] = _rmat_attempt(key, e[bad], attempt, scale)
            row, col = row % n, col % n
        src[first:first + e.numel()] = row
        dst[first:first + e.numel()] = col
    return src, dst


def _batch_specs(case):
    """(n, edge offsets) of a batch: n log-uniform in [32, n_max], average degree U(4, 32)."""
    rng = np.random.RandomState(case["graphs"] * 65537 + case["n_max"])
    G = case["graphs"]
    n = np.floor(np.exp(rng.uniform(math.log(32), math.log(case["n_max"] + 1), G))).astype(np.int32)
    m = np.rint(n * rng.uniform(4, 32, G) / 2).astype(np.int64)
    off = np.concatenate([[0], np.cumsum(m)])
    while off[-1] > MAX_PAIRS:  # a draw of large graphs: the batch ends before the limit
        n, m, off = n[:-1], m[:-1], off[:-1]
    return n, off


def _batch_pairs(n, off, seed):
    """Local ids of all graphs: even graphs R-MAT, odd ones uniform, every level drawn for all pairs at once."""
    G, m = len(n), int(off[-1])
    g = torch.repeat_interleave(torch.arange(G, device="cuda"), torch.from_numpy(np.diff(off)).cuda(), output_size=m)
    nn = torch.from_numpy(n).cuda().long()
    scale = torch.tensor([max(1, (int(x) - 1).bit_length()) for x in n], device="cuda")
    src = torch.empty(m, dtype=torch.int32, device="cuda")
    dst = torch.empty(m, dtype=torch.int32, device="cuda")
    key = _stream_key(seed, 0)
    step = 1 << 23
    for first in range(0, m, step):
        e = torch.arange(first, min(m, first + step), dtype=torch.int64, device="cuda")
        gi = g[first:first + e.numel()]
        n_e, s_e = nn[gi], scale[gi]
        top = int(s_e.max())
        x = _mix((e + 1) * GAMMA + _stream_key(seed, 1))
        er_row, er_col = (_shr(x, 32) * n_e) >> 32, ((x & 0xffffffff) * n_e) >> 32
        row, col = _rmat_attempt(key, e, 0, top)
        # a graph of fewer levels takes the last ones; ids past n are folded back
        row, col = (row & ((1 << s_e) - 1)) % n_e, (col & ((1 << s_e) - 1)) % n_e
        even = gi % 2 == 0
        src[first:first + e.numel()] = torch.where(even, row, er_row)
        dst[first:first + e.numel()] = torch.where(even, col, er_col)
    return src, dst


class _Request:
    """What tc.Server.submit reads of a workload."""

    def __init__(self, kind, n, m, seed, stream):
        self.kind, self.n, self.m, self.seed, self.stream = kind, n, m, seed, stream


def _requests(case, seed):
    """The requests' sizes belong to the case, their graphs to the seed."""
    rng = np.random.RandomState(case["requests"] * 1000003 + case["n_max"])
    out = []
    for q in range(case["requests"]):
        n = int(math.exp(rng.uniform(math.log(1000), math.log(case["n_max"]))))
        m = int(round(rng.uniform(4, 16) * n))
        out.append(_Request("rmat" if rng.uniform() < 0.7 else "er_replace", n, m, seed, q + 1))
    return out


class _Server:
    """A serving loop that lives as long as the program that holds it."""

    def __init__(self):
        self.srv, self.done = tc.Server(BUDGET, SLOTS), 0

    def __del__(self):
        self.srv.stop()


class _Kept:
    """A graph handle that the program keeps."""

    def __init__(self, n, src, dst):
        self.g = tc.Graph.from_edges(n, src, dst, torch.cuda.current_stream())


def _symmetric_csr(n, src, dst):
    """Sorted symmetric rows without loops: (int64 offsets[n + 1], int32 adj)."""
    s, d = src.long(), dst.long()
    keep = s != d
    s, d = s[keep], d[keep]
    key = torch.unique(torch.cat([s * n + d, d * n + s]))
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return off, (key % n).int()


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "serve":
        st["requests"], st["server"] = _requests(case, seed), _Server()
        return st
    if kind == "batch":
        n, off = _batch_specs(case)
        st["n"], st["off"] = n, off
        st["src"], st["dst"] = _batch_pairs(n, off, seed)
        total = int(n.sum())
        st["T"] = torch.empty(len(n), dtype=torch.int64, device="cuda")
        st["t"] = torch.empty(total, dtype=torch.int64, device="cuda")
        st["lcc"] = torch.empty(total, dtype=torch.float64, device="cuda")
        return st
    n = st["n"] = case["n"]
    src, dst = _pairs(case["gen"], n, case["m"], seed)
    if kind == "csr":
        st["off"], st["adj"] = _symmetric_csr(n, src, dst)
    elif kind == "host":
        st["pinned"] = [src.cpu().pin_memory(), dst.cpu().pin_memory(),
                        torch.empty(n, dtype=torch.int64).pin_memory(), torch.empty(n, dtype=torch.float64).pin_memory()]
        st["src"], st["dst"], st["t"], st["lcc"] = [x.numpy() for x in st["pinned"]]
        return st
    elif kind in ("support", "shard"):
        st["kept"] = _Kept(n, src, dst)
        if kind == "support":
            # room for every pair, as a program has that did not count the repeats
            st["out"] = [torch.zeros(case["m"], dtype=torch.int32, device="cuda") for _ in range(3)]
            return st
        st["shard"], st["nshards"] = case["shard"], case["nshards"]
    else:
        st["src"], st["dst"] = src, dst
    st["t"] = torch.empty(n, dtype=torch.int64, device="cuda")
    st["lcc"] = torch.empty(n, dtype=torch.float64, device="cuda")
    return st


# ---- one pass ----------------------------------------------------------------------

def _count(g, st):
    try:
        T = g.count()
        g.lcc(st["t"], st["lcc"])
    finally:
        g.close()
    return {"T": T, "t": st["t"], "lcc": st["lcc"]}


def run(state):
    st, kind = state, state["kind"]
    stream = torch.cuda.current_stream()
    if kind == "edges" or kind == "host":
        return _count(tc.Graph.from_edges(st["n"], st["src"], st["dst"], stream), st)
    if kind == "csr":
        return _count(tc.Graph.from_csr(st["n"], st["off"], st["adj"], stream), st)
    if kind == "noalloc":
        T = tc.tc_count_noalloc(st["n"], st["src"], st["dst"], st["t"], st["lcc"], stream)
        return {"T": T, "t": st["t"], "lcc": st["lcc"]}
    if kind == "batch":
        tc.tc_batch_run(st["n"], st["off"], st["src"], st["dst"], st["T"], st["t"], st["lcc"], stream=stream)
        return {"T": st["T"], "t": st["t"], "lcc": st["lcc"]}
    if kind == "directed":
        c, lcc, stats = tc.tc_directed_lcc(st["n"], st["src"], st["dst"], st["t"], st["lcc"], stream)
        return {"c": c, "lcc": lcc, "m_directed": stats["m_directed"], "total": stats["total"]}
    if kind == "support":
        u, v, s = st["kept"].g.edge_support(*st["out"])
        return {"u": u, "v": v, "support": s}
    if kind == "shard":
        T, t = st["kept"].g.count_shard(st["shard"], st["nshards"], st["t"])
        return {"T": T, "t": t}
    server = st["server"]
    for q, r in enumerate(st["requests"]):
        server.srv.submit(q, r)
    server.done += len(st["requests"])
    if not server.srv.wait(server.done, 120.0):
        raise RuntimeError("the serving loop did not finish its requests")
    res = sorted(server.srv.poll(), key=lambda r: r["id"])
    if any(r["status"] != 0 for r in res):
        raise RuntimeError("a request failed")
    return {k: np.array([r[k] for r in res], dtype=np.uint64).view(np.int64)
            for k in ("T", "m_simple", "t_hash", "lcc_hash")}


# ---- the work and the reference ----------------------------------------------------

def work(case):
    """The pairs read once, t[] and LCC[] written once; one multiplication and one division per LCC."""
    kind = case["kind"]
    if kind == "serve":
        reqs = _requests(case, 1)
        n, m = sum(r.n for r in reqs), sum(r.m for r in reqs)
        return {"bytes": 8 * m + 16 * n, "flops": 2 * n}
    if kind == "batch":
        n, off = _batch_specs(case)
        return {"bytes": 8 * int(off[-1]) + 16 * int(n.sum()), "flops": 2 * int(n.sum())}
    n, m = case["n"], case["m"]
    if kind == "csr":
        return {"bytes": 8 * m + 24 * n, "flops": 2 * n}
    if kind == "support":  # the kept rows read, three words per edge written
        return {"bytes": 16 * m, "flops": 0}
    if kind == "shard":
        return {"bytes": 4 * m + 8 * n, "flops": 0}
    return {"bytes": 8 * m + 16 * n, "flops": 2 * n}


def tolerance(case):
    return "exact"


def _orient(n, src, dst):
    """Distinct edges oriented by (pairs at the vertex, id): dict of rank-space arrays."""
    s, d = src.long(), dst.long()
    keep = s != d
    s, d = s[keep], d[keep]
    pairs = torch.bincount(s, minlength=n) + torch.bincount(d, minlength=n)
    id_of = torch.argsort(pairs, stable=True)
    rank = torch.empty_like(id_of)
    rank[id_of] = torch.arange(n, device=rank.device)
    rs, rd = rank[s], rank[d]
    lo, hi = torch.minimum(rs, rd), torch.maximum(rs, rd)
    key = torch.unique(lo * n + hi)
    return {"n": n, "rank": rank, "id_of": id_of, "key": key, "u": key // n, "v": key % n,
            "forward": torch.unique((lo * n + hi)[rs < rd]), "back": torch.unique((lo * n + hi)[rs > rd])}


def _triangles(o, sources=None):
    """Chunks of triangles u < v < w (ranks) as the positions of their edges (uv, uw, vw) in the key list."""
    n, key = o["n"], o["key"]
    m = key.numel()
    if m == 0:
        return
    ends = torch.searchsorted(key, (o["u"] + 1) * n)
    suffix = ends - torch.arange(m, device=key.device) - 1
    if sources is not None:
        suffix = torch.where((o["u"] >= sources[0]) & (o["u"] < sources[1]), suffix, torch.zeros_like(suffix))
    total = suffix.cumsum(0)
    cuts, done = [0], 0
    while cuts[-1] < m:
        at = int(torch.searchsorted(total, torch.tensor(done + (1 << 25), device=key.device), right=True))
        at = max(at, cuts[-1] + 1)
        done = int(total[at - 1])
        cuts.append(at)
    for a, b in zip(cuts, cuts[1:]):
        cnt = suffix[a:b]
        size = int(cnt.sum())
        if size == 0:
            continue
        uv = torch.repeat_interleave(torch.arange(a, b, device=key.device), cnt, output_size=size)
        first = cnt.cumsum(0) - cnt
        uw = uv + 1 + torch.arange(size, device=key.device) - first[uv - a]
        want = o["v"][uv] * n + o["v"][uw]
        vw = torch.searchsorted(key, want).clamp_(max=m - 1)
        hit = (key[vw] == want).nonzero().squeeze(1)
        yield uv[hit], uw[hit], vw[hit]


def _counts(o, sources=None):
    t = torch.zeros(o["n"], dtype=torch.int64, device="cuda")
    for uv, uw, _ in _triangles(o, sources):
        for r in (o["u"][uv], o["v"][uv], o["v"][uw]):
            t += torch.bincount(r, minlength=o["n"])
    return t[o["rank"]]


def _lcc(t, d):
    return torch.where((d < 2) | (t == 0), 0.0, (2 * t).double() / (d * (d - 1)).clamp(min=1).double())


def _degrees(o):
    d = torch.bincount(o["u"], minlength=o["n"]) + torch.bincount(o["v"], minlength=o["n"])
    return d[o["rank"]]


def _t_and_lcc(n, src, dst):
    o = _orient(n, src, dst)
    t = _counts(o)
    return o, t, _lcc(t, _degrees(o))


def _hash(x):
    return int(_mix((torch.arange(x.numel(), device="cuda") * GAMMA) ^ x).sum())


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        rows = []
        for r in _requests(case, seed):
            o, t, lcc = _t_and_lcc(r.n, *_pairs("rmat" if r.kind == "rmat" else "er", r.n, r.m, r.seed, r.stream))
            rows.append((int(t.sum()) // 3, o["key"].numel(), _hash(t), _hash(lcc.view(torch.int64))))
        cols = list(zip(*rows))
        return {k: np.array(cols[i], dtype=np.int64) for i, k in enumerate(("T", "m_simple", "t_hash", "lcc_hash"))}
    if kind == "batch":
        n, off = _batch_specs(case)
        src, dst = _batch_pairs(n, off, seed)
        nn = torch.from_numpy(n).cuda().long()
        G, total = len(n), int(n.sum())
        base = nn.cumsum(0) - nn
        shift = torch.repeat_interleave(base, torch.from_numpy(np.diff(off)).cuda(), output_size=src.numel())
        _, t, lcc = _t_and_lcc(total, src + shift, dst + shift)
        of = torch.repeat_interleave(torch.arange(G, device="cuda"), nn, output_size=total)
        T = torch.zeros(G, dtype=torch.int64, device="cuda").index_add_(0, of, t) // 3
        return {"T": T, "t": t, "lcc": lcc}
    n = case["n"]
    src, dst = _pairs(case["gen"], n, case["m"], seed)
    if kind == "directed":
        o = _orient(n, src, dst)
        m = o["key"].numel()
        bit = torch.zeros(m, 2, dtype=torch.int64, device="cuda")
        for k, name in enumerate(("forward", "back")):
            bit[torch.searchsorted(o["key"], o[name]), k] = 1
        c = torch.zeros(n, dtype=torch.int64, device="cuda")
        for uv, uw, vw in _triangles(o):
            f, g, h = bit[uv], bit[uw], bit[vw]  # u -> v / v -> u, u -> w / w -> u, v -> w / w -> v
            for r, x in ((o["u"][uv], f[:, 0] * g[:, 0] * h.sum(1)), (o["v"][uv], f[:, 1] * h[:, 0] * g.sum(1)),
                         (o["v"][uw], g[:, 1] * h[:, 1] * f.sum(1))):
                c.index_add_(0, r, x)
        out = torch.bincount(o["u"], bit[:, 0].double(), n) + torch.bincount(o["v"], bit[:, 1].double(), n)
        out, c = out.long()[o["rank"]], c[o["rank"]]
        lcc = torch.where((out < 2) | (c == 0), 0.0, c.double() / (out * (out - 1)).clamp(min=1).double())
        return {"c": c, "lcc": lcc, "m_directed": int(bit.sum()), "total": int(c.sum())}
    if kind == "support":
        o = _orient(n, src, dst)
        s = torch.zeros(o["key"].numel(), dtype=torch.int64, device="cuda")
        for edges in _triangles(o):
            for e in edges:
                s += torch.bincount(e, minlength=s.numel())
        u, v = o["id_of"][o["u"]], o["id_of"][o["v"]]
        rest = case["m"] - s.numel()  # the entries after the distinct edges stay zero
        u, v, s = [torch.nn.functional.pad(x, (0, rest)).int() for x in (torch.minimum(u, v), torch.maximum(u, v), s)]
        return {"u": u, "v": v, "support": s}
    if kind == "shard":
        o = _orient(n, src, dst)
        d = torch.bincount(o["u"], minlength=n)
        prefix = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), (d * (d + 1) // 2 + 1).cumsum(0)])
        total, k, N = int(prefix[-1]), case["shard"], case["nshards"]
        lo, hi = [int(torch.searchsorted(prefix[:n], torch.tensor(total * x // N, device="cuda"))) for x in (k, k + 1)]
        t = _counts(o, (lo, n if k + 1 == N else hi))
        return {"T": int(t.sum()) // 3, "t": t}
    if kind == "csr":
        off, adj = _symmetric_csr(n, src, dst)
        src = torch.repeat_interleave(torch.arange(n, device="cuda"), off.diff(), output_size=adj.numel())
        dst = adj
    _, t, lcc = _t_and_lcc(n, src, dst)
    T = int(t.sum()) // 3
    if kind == "host":
        t, lcc = t.cpu().numpy(), lcc.cpu().numpy()
    return {"T": T, "t": t, "lcc": lcc}
