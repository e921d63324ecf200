"""The alignment kernel's tile records against the CPU oracle, where they can go wrong:
vertex lengths around the 8-diagonal tile and the 16-base window, self arcs, batches on
CTAs of every width, queries whose tiles outgrow the listed-flags in shared memory, and
records freed by the memory bound and used again.  Distances and work counters are
integers fixed by the method, so they are compared for equality."""
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
    if w["distance"] < 0:
        assert int(r["status"]) == w["distance"], (ctx, r, w)
        return
    assert int(r["status"]) == 0, (ctx, r, w)
    for a, b in FIELDS:
        assert int(r[a]) == w[b], (ctx, a, int(r[a]), w[b])


def chain_graph(rng, lengths, loops):
    """Bubbles of two parallel vertices between single ones, some with self arcs."""
    labels, arcs, prev = [], [], []
    for i, n in enumerate(lengths):
        here = []
        for _ in range(1 + i % 2):
            labels.append("".join("ACGT"[c] for c in rng.integers(0, 4, n)))
            here.append(len(labels) - 1)
            if loops and rng.random() < 0.3:
                arcs.append((here[-1], here[-1]))
        arcs += [(u, v) for u in prev for v in here]
        prev = here
    labels.append("ACGTTGCA")
    arcs += [(u, len(labels) - 1) for u in prev]
    return synth.Graph.from_lists(labels, arcs)


@pytest.mark.parametrize("threads", [32, 512, 1024])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 33])
def test_vertex_lengths_around_tile_and_window(n, threads):
    rng = np.random.default_rng(1000 * n + threads)
    g = chain_graph(rng, [max(1, n + int(x)) for x in rng.integers(-1, 2, 24)], loops=n < 16)
    graph = gw.Graph.from_synth(g)
    qs, ends = [], []
    for i in range(24):   # walks with errors, unrelated bases, and very short queries
        if i % 3 == 2:
            q = rng.integers(0, 4, int(rng.integers(0, 3 * n + 2)))
        else:
            q = np.frombuffer(b"".join(g.label(v) for v in range(0, g.n_vertices, 2)), np.uint8)
            q = np.searchsorted(np.frombuffer(b"ACGT", np.uint8), q)
            err = rng.random(len(q)) < 0.12
            q = np.delete(np.where(err, rng.integers(0, 4, len(q)), q), np.nonzero(rng.random(len(q)) < 0.03)[0])
        qs.append(bytes(np.frombuffer(b"ACGT", np.uint8)[q]))
        ends.append(g.n_vertices - 1 if i % 4 else int(rng.integers(0, g.n_vertices)))
    off = np.concatenate([[0], np.cumsum([len(q) for q in qs])]).astype(np.uint64)
    seq = np.frombuffer(b"".join(qs), np.uint8)
    for lag in (0, 9, 40):
        cfg = gw.default_config(graph, prune=lag > 0)
        cfg.threads = threads
        res = gw.Engine(graph, prune=lag > 0, config=cfg).align_batch(seq, off, [0] * len(qs), ends, max_lag=lag)
        for i, q in enumerate(qs):
            same(res[i], oracle.gwfa(g, q, 0, ends[i], a_diff=lag), (n, lag, i))


def test_more_tiles_than_flags_in_shared_memory():
    """25 kb at 5%: about 45,000 tiles, beyond the 32,768 whose flags are in shared memory."""
    import torch
    g, _ = synth.make_config(2, n_queries=1)
    c = synth.CONFIGS[2]
    qs = synth.make_queries(g, 3, 91, synth._const(25_000), synth._const(0.05), c["weights"], c["loops"])
    graph = gw.Graph.from_synth(g)
    eng = gw.Engine(graph)
    stats = torch.zeros(3 * 8, dtype=torch.int64, device="cuda")
    eng.set_stats(stats.data_ptr())
    res = eng.align_batch(qs.seq, qs.off, qs.v_s, qs.v_e)
    assert stats.view(3, 8)[:, 6].max().item() > 32768
    for i, w in enumerate(oracle.gwfa_many(g, qs, range(3))):
        same(res[i], w, i)


def test_freed_records_are_used_again():
    """Evicting at every score on a slab that holds a fraction of the diagonals ever
    visited: the records handed out must come from the free list."""
    g, qs = synth.make_config(3, n_queries=6, backbone=200_000)
    graph = gw.Graph.from_synth(g)
    cfg = gw.default_config(graph, prune=True)
    cfg.n_tiers = 1
    cfg.tiers[0].ctas, cfg.tiers[0].log2_tiles = 4, 9
    eng = gw.Engine(graph, prune=True, config=cfg)
    res = eng.align_batch(qs.seq, qs.off, qs.v_s, qs.v_e, max_lag=300, evict_lag=300, evict_every=1)
    want = oracle.gwfa_many(g, qs, range(len(qs)), a_diff=300, evict_lag=300, evict_every=1)
    for i, w in enumerate(want):
        same(res[i], w, i)
        assert int(res[i]["evicted"]) == w["evicted"] and w["visited"] > 8 * 384


@pytest.mark.parametrize("prune", [False, True])
def test_the_load_limit_does_not_depend_on_timing(prune):
    """Which queries a slab has room for is the same on CTAs of every width, also for those
    that end in the very score that brings the tiles to the limit."""
    g, _ = synth.make_config(2, n_queries=1)
    graph = gw.Graph.from_synth(g)
    for seed in range(3):
        qs = synth.make_queries(g, 600, seed, synth._const(3000), synth._uniform(0.0, 0.08), (1, 1, 1), (1, 1))
        first = None
        for threads in (64, 256, 512 if prune else 1024):
            cfg = gw.default_config(graph, prune=prune)
            cfg.n_tiers, cfg.threads = 1, threads
            cfg.tiers[0].log2_tiles = 10
            eng = gw.Engine(graph, prune=prune, config=cfg)
            for _ in range(2):
                status = eng.align_batch(qs.seq, qs.off, qs.v_s, qs.v_e)["status"].copy()
                first = status if first is None else first
                assert np.array_equal(status, first), (seed, threads)
            eng.close()
        assert 0 < (first == 0).sum() < 600
