"""What a slab has room for, against the CPU oracle: queries that use most of the lists of a
small slab end on it with the oracle's result, and those whose tiles exceed the load limit
(3/4 of the slab's) are handed to the next tier."""
import numpy as np
import pytest

import oracle
import paper_2206_13574_gb300 as gw
from paper_2206_13574_gb300 import _build, synth

pytestmark = pytest.mark.gpu
FIELDS = [("edit_distance", "distance"), ("n_scores", "n_scores"), ("cells", "cells"),
          ("peak_frontier", "peak"), ("visited", "visited"), ("spills", "spills"),
          ("pruned", "pruned"), ("is_upper_bound", "is_upper_bound")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    _build.build()
    oracle.build()


def same(r, w, ctx):
    assert int(r["status"]) == 0, (ctx, r, w)
    for a, b in FIELDS:
        assert int(r[a]) == w[b], (ctx, a, int(r[a]), w[b])


def engine(graph, threads, log2, prune=False):
    """One tier (or two) of four CTAs of `threads` threads."""
    cfg = gw.default_config(graph, prune=prune)
    log2 = (log2,) if isinstance(log2, int) else log2
    cfg.n_tiers = len(log2)
    for t, lg in enumerate(log2):
        cfg.tiers[t].ctas, cfg.tiers[t].log2_tiles, cfg.tiers[t].threads = 4, lg, threads
    return gw.Engine(graph, prune=prune, config=cfg)


def batch(queries):
    off = np.concatenate([[0], np.cumsum([len(q) for q in queries])]).astype(np.uint64)
    return np.frombuffer(b"".join(queries), np.uint8), off


# Score 0 fills 4 n diagonals, and at score 1 all of C, G and T reach the end of their vertex
# at once: 3 n spill requests, over the 256 kept in shared memory, the 512 kept whole and the
# 1,024 that half of the slab's diagonals make; 192 tiles are the load limit (n = 383)
@pytest.mark.parametrize("threads", [64, 256, 1024])
def test_every_diagonal_spills_in_one_score(threads):
    g = synth.Graph.from_lists(["A", "C", "G", "T"], [(0, 0), (0, 1), (0, 2), (0, 3), (1, 2), (2, 3), (3, 0)])
    graph = gw.Graph.from_synth(g)
    lens = [84, 85, 86, 87, 170, 171, 172, 340, 341, 342, 343, 360, 383, 384, 500]
    qs = [b"A" * n for n in lens]
    seq, off = batch(qs)
    zero, one = [0] * len(qs), [1] * len(qs)
    want = [oracle.gwfa(g, q, 0, 1) for q in qs]
    res = engine(graph, threads, 8).align_batch(seq, off, zero, one)
    for n, r, w in zip(lens, res, want):
        if n < 384:
            same(r, w, n)
        else:
            assert int(r["status"]) == gw.GWFA_ERR_CAPACITY, n
    for n, r, w in zip(lens, engine(graph, threads, (8, 11)).align_batch(seq, off, zero, one), want):
        same(r, w, n)


# A free start puts all diagonals of a run of one base on the wavefront at score 0, and every
# one of them reaches the end of its vertex; 1,528 diagonals are what the load limit admits
@pytest.mark.parametrize("threads", [64, 1024])
@pytest.mark.parametrize("size", [255, 257, 511, 513, 1023, 1025, 1300, 1528, 1529])
def test_free_start_on_a_run_of_one_base(threads, size):
    g = synth.Graph.from_lists(["A" * size, "GC"], [])
    graph = gw.Graph.from_synth(g)
    qs = [b"A" * size, b"A" * size + b"T"]
    seq, off = batch(qs)
    res = engine(graph, threads, 8).align_batch(seq, off, [0, 0], [0, 0], ends=1)
    wide = engine(graph, threads, (8, 11)).align_batch(seq, off, [0, 0], [0, 0], ends=1)
    for q, a, b in zip(qs, res, wide):
        w = oracle.gwfa(g, q, 0, 0, ends=1)
        same(b, w, q[size:])
        if size <= 1528:
            same(a, w, q[size:])
        else:
            assert int(a["status"]) == gw.GWFA_ERR_CAPACITY


def bubble_chain(rng, sites, seg):
    """Segments of `seg` bases with a bubble of two single bases after each, and a walk through."""
    labels, arcs, walk = [], [], []
    for _ in range(sites):
        at = len(labels)
        labels.append("".join("ACGT"[c] for c in rng.integers(0, 4, seg)))
        a, b = rng.permutation(4)[:2]
        labels += ["ACGT"[a], "ACGT"[b]]
        arcs += [(at, at + 1), (at, at + 2), (at + 1, at + 3), (at + 2, at + 3)]
        walk += [at, at + 1 + int(rng.integers(2))]
    labels.append("ACGTTGCA")
    return synth.Graph.from_lists(labels, arcs), walk + [len(labels) - 1]


def noisy(rng, text, rate):
    q = np.searchsorted(np.frombuffer(b"ACGT", np.uint8), np.frombuffer(text, np.uint8))
    q = np.where(rng.random(len(q)) < rate, rng.integers(0, 4, len(q)), q)
    q = np.repeat(q, rng.choice([0, 1, 2], len(q), p=[rate / 2, 1 - rate, rate / 2]))
    return bytes(np.frombuffer(b"ACGT", np.uint8)[q])


# The eight diagonals of a tile of the run spill into one tile each, many at once: a tile uses
# up one record however many threads meet there (192 are the load limit)
@pytest.mark.parametrize("threads", [64, 256, 1024])
@pytest.mark.parametrize("size", [255, 257, 511, 513, 755])
def test_spills_that_meet_at_one_tile(threads, size):
    g = synth.Graph.from_lists(["A" * size, "GC"], [(0, 1)])
    qs = [b"A" * size + t for t in (b"GC", b"TC", b"C")]
    seq, off = batch(qs)
    res = engine(gw.Graph.from_synth(g), threads, 8).align_batch(seq, off, [0] * 3, [1] * 3, ends=1)
    for q, r in zip(qs, res):
        same(r, oracle.gwfa(g, q, 0, 1, ends=1), q[size:])


# Behind a bubble both of its vertices spill into the same tiles in the same round.  Under the
# memory bound a long query passes thousands of bubbles on a slab of 256 tiles.
@pytest.mark.parametrize("threads", [32, 256])
def test_bubbles_under_the_memory_bound(threads):
    rng = np.random.default_rng(threads)
    g, walk = bubble_chain(rng, 1500, 12)
    text = b"".join(g.label(v) for v in walk)
    qs = [noisy(rng, text, e) for e in (0.01, 0.02, 0.03, 0.03)]
    seq, off = batch(qs)
    opts = dict(evict_lag=60, evict_every=4)
    res = engine(gw.Graph.from_synth(g), threads, 8, prune=True).align_batch(
        seq, off, [0] * 4, [walk[-1]] * 4, max_lag=60, **opts)
    for i, (q, r) in enumerate(zip(qs, res)):
        w = oracle.gwfa(g, q, 0, walk[-1], a_diff=60, **opts)
        same(r, w, i)
        assert int(r["evicted"]) == w["evicted"]


# A round of spills into a vertex with many arcs inserts more diagonals than it has requests:
# over the 64 kept in shared memory, and over twice the tiles of the slab (traceback runs on
# the pruning kernel).  160 bases make 1,288 insertions into 189 tiles.
@pytest.mark.parametrize("threads", [32, 256, 1024])
@pytest.mark.parametrize("size", [1, 7, 8, 31, 32, 63, 64, 65, 120, 160])
def test_insertions_of_a_vertex_with_many_arcs(threads, size):
    import torch
    ends = ["ACG", "CAT", "CGT", "GCA", "GTT", "TAC", "TCC", "TGA"]
    g = synth.Graph.from_lists(["A" * size] + ends, [(0, 1 + i) for i in range(8)])
    qs = [b"A" * size + t for t in ((b"CGT", b"CT", b"CAGT") if size < 64 else (b"CGT",))]   # (T holds 512 requests)
    n = len(qs)
    seq, off = batch(qs)
    vs, ve = np.zeros(n, np.uint32), np.full(n, 3, np.uint32)
    b = gw.DeviceBatch(synth.Queries(seq.copy(), off, vs, ve, np.zeros(n, np.int64), np.zeros(n)))
    eng = engine(gw.Graph.from_synth(g), threads, 8, prune=True)
    paths = torch.zeros(n * 8, dtype=torch.int32, device="cuda")
    plen = torch.zeros(n, dtype=torch.int32, device="cuda")
    eng.set_paths(paths.data_ptr(), 8, plen.data_ptr())
    b.run(eng, traceback=True, ends=1)
    torch.cuda.synchronize()
    for i, (q, r) in enumerate(zip(qs, b.results())):
        same(r, oracle.gwfa(g, q, 0, 3, ends=1), q[size:])
        assert plen[i].item() == 2 and paths[8 * i:8 * i + 2].tolist() == [0, 3]


# Which lag-pruned reads a slab has room for is the same on CTAs of every width
@pytest.mark.parametrize("lag", [400, 1000])
def test_the_load_limit_with_pruning_does_not_depend_on_timing(lag):
    rng = np.random.default_rng(lag)
    g, walk = bubble_chain(rng, 300, 12)
    graph = gw.Graph.from_synth(g)
    text = b"".join(g.label(v) for v in walk)
    qs = [noisy(rng, text, e) for e in rng.uniform(0, 0.1, 200)]
    seq, off = batch(qs)
    first = None
    for threads in (32, 256, 512, 1024):
        eng = engine(graph, threads, 11, prune=True)
        for _ in range(2):
            res = eng.align_batch(seq, off, [0] * len(qs), [walk[-1]] * len(qs), max_lag=lag)
            first = res if first is None else first
            assert np.array_equal(res["status"], first["status"]), threads
    fit = np.nonzero(first["status"] == 0)[0]
    assert 0 < len(fit) < len(qs)
    for i in fit[:8]:
        same(first[i], oracle.gwfa(g, qs[i], 0, walk[-1], a_diff=lag), i)


# The tiles of the statistics are those that hold a diagonal when the query ends: with the
# spills of its last score, without the neighbours that only a next score would need
@pytest.mark.parametrize("lag", [0, 500])
def test_tiles_in_the_statistics(lag):
    import torch
    g = synth.Graph.from_lists(["A", "C", "G", "T"], [(0, 0), (0, 1), (0, 2), (0, 3), (1, 2), (2, 3), (3, 0)])
    lens = [0, 1, 6, 7, 8, 100, 343, 1000]
    seq, off = batch([b"A" * n for n in lens])
    stats = torch.zeros(len(lens) * 8, dtype=torch.int64, device="cuda")
    eng = engine(gw.Graph.from_synth(g), 64, 11, prune=lag > 0)
    eng.set_stats(stats.data_ptr())
    for ve in (0, 1):   # distance 0 and 1; diagonals 0..n of A, 1..n of the others
        res = eng.align_batch(seq, off, [0] * len(lens), [ve] * len(lens), max_lag=lag)
        for n, r, t in zip(lens, res, stats.view(-1, 8)[:, 6].tolist()):
            w = oracle.gwfa(g, b"A" * n, 0, ve, a_diff=lag)
            if n > 0:
                assert (int(r["edit_distance"]), int(r["visited"])) == (w["distance"], w["visited"])
                assert w["visited"] not in (4 * n + 1, 4 * n + 4) or t == 4 * (n // 8 + 1), (n, t)
    rng = np.random.default_rng(3)
    ends = ["".join("ACGT"[c] for c in rng.integers(0, 4, 12)) for _ in range(50)]
    eng = engine(gw.Graph.from_synth(synth.Graph.from_lists(["ACGTTGCA"] + ends, [(0, 1 + i) for i in range(50)])), 64, 11, prune=lag > 0)
    eng.set_stats(stats.data_ptr())
    seq, off = batch([("ACGTTGCA" + ends[20]).encode()])
    assert eng.align_batch(seq, off, [0], [21], max_lag=lag)[0]["edit_distance"] == 0
    assert stats[6].item() == 51   # the first vertex and its successors, (u, 8) each


# A score whose spills bring the tiles to most of the slab may leave border words for as many
# tiles again (here each of 5,000 diagonals for the tile on its left).  They belong to the
# next score: a query that ends in this one does not need them, and has room.
@pytest.mark.parametrize("threads", [64, 256, 1024])
@pytest.mark.parametrize("mode", ["exact", "lag", "traceback"])
def test_tiles_of_the_next_score_leave_room_for_spills(threads, mode):
    import torch
    rng = np.random.default_rng(threads)
    ends = ["".join("ACGT"[c] for c in rng.integers(0, 4, 12)) for _ in range(5000)]
    g = synth.Graph.from_lists(["ACGTTGCA"] + ends, [(0, 1 + i) for i in range(5000)])
    qs = [("ACGTTGCA" + ends[i]).encode() for i in (0, 2500, 4999)] + [("ACGTTGCT" + ends[7]).encode()]
    ve = np.array([1, 2501, 5000, 8], np.uint32)
    n, vs = len(qs), np.zeros(4, np.uint32)
    seq, off = batch(qs)
    prune, lag = mode != "exact", 500 if mode == "lag" else 0
    b = gw.DeviceBatch(synth.Queries(seq.copy(), off, vs, ve, np.zeros(n, np.int64), np.zeros(n)))
    graph = gw.Graph.from_synth(g)
    for log2, fit in ((13, 3), (15, 4)):   # 6,144 tiles are the load limit; the last query needs 10,000
        eng = engine(graph, threads, log2, prune=prune)
        for _ in range(3):
            b.run(eng, traceback=mode == "traceback", max_lag=lag)
            torch.cuda.synchronize()
            res = b.results()
            for i in range(n):
                if i < fit:
                    same(res[i], oracle.gwfa(g, qs[i], 0, int(ve[i]), a_diff=lag), i)
                else:
                    assert int(res[i]["status"]) == gw.GWFA_ERR_CAPACITY


# With pruning a border word's candidate may be dropped, its tile staying empty: such tiles
# give way to those that hold a diagonal.  Reads with few errors leave many.
@pytest.mark.parametrize("threads", [64, 256, 1024])
def test_empty_tiles_give_way(threads):
    import torch
    rng = np.random.default_rng(11)
    g, walk = bubble_chain(rng, 1500, 3)
    graph = gw.Graph.from_synth(g)
    text = b"".join(g.label(v) for v in walk)
    qs = [noisy(rng, text, e) for e in rng.uniform(0.0005, 0.012, 120)]
    seq, off = batch(qs)
    n, end = len(qs), [walk[-1]] * len(qs)
    held = torch.zeros(n * 8, dtype=torch.int64, device="cuda")
    eng = engine(graph, threads, 17, prune=True)
    eng.set_stats(held.data_ptr())
    want = eng.align_batch(seq, off, [0] * n, end, max_lag=200)
    held = held.view(n, 8)[:, 6].cpu().numpy()
    res = engine(graph, threads, 13, prune=True).align_batch(seq, off, [0] * n, end, max_lag=200)
    assert (want["status"] == 0).all() and ((held > 5000) & (held <= 6144)).sum() > 5 and (held > 6144).any()
    for i in range(n):
        if held[i] <= 6144:
            assert int(res[i]["status"]) == 0, (i, held[i])
            for f in ("edit_distance", "cells", "visited", "pruned", "spills"):
                assert res[i][f] == want[i][f], (i, f)
        else:
            assert int(res[i]["status"]) == gw.GWFA_ERR_CAPACITY
