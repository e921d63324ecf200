"""Cost-model features on the GPU against a plain Python form of their definition: queries
whose co-reachable subgraph fits the searches' shared-memory tables and queries that
outgrow them (more than 768 vertices), cyclic graphs, vertices with more than four arcs,
queries shorter than a k-mer and a vertex that cannot reach v_e."""
import math

import numpy as np
import pytest

import paper_2206_13574_gb300 as gw
from paper_2206_13574_gb300 import _build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    _build.build()


def reach(src, arcs, lens, budget):
    far, todo = {src: 0}, [src]
    while todo:
        nxt = []
        for v in todo:
            c = far[v] + lens[v]
            if c <= budget:
                for u in arcs[v]:
                    if c < far.get(u, budget + 1):
                        far[u] = c
                        nxt.append(u)
        todo = nxt
    return far


def cycle_arcs(arcs):
    """Arcs inside a strongly connected component (Kosaraju, iterative)."""
    n = len(arcs)
    back = [[] for _ in arcs]
    for u, vs in enumerate(arcs):
        for v in vs:
            back[v].append(u)
    seen, order = [False] * n, []
    for r in range(n):
        if seen[r]:
            continue
        stack, seen[r] = [(r, iter(arcs[r]))], True
        while stack:
            v, it = stack[-1]
            w = next((x for x in it if not seen[x]), None)
            if w is None:
                order.append(v)
                stack.pop()
            else:
                seen[w] = True
                stack.append((w, iter(arcs[w])))
    comp = [-1] * n
    for r in reversed(order):
        if comp[r] < 0:
            todo, comp[r] = [r], r
            while todo:
                v = todo.pop()
                for u in back[v]:
                    if comp[u] < 0:
                        comp[u] = r
                        todo.append(u)
    return {(u, v) for u in range(n) for v in arcs[u] if comp[u] == comp[v]}


def reference(g, qs):
    lens = g.lengths().tolist()
    out = [sorted({int(v) for v in g.arc_dst[g.arc_src == u]}) for u in range(g.n_vertices)] if g.n_vertices < 3000 else None
    if out is None:
        out = [[] for _ in lens]
        for u, v in sorted(set(zip(g.arc_src.tolist(), g.arc_dst.tolist()))):
            out[u].append(v)
    back = [[] for _ in lens]
    for u, vs in enumerate(out):
        for v in vs:
            back[v].append(u)
    cyc = cycle_arcs(out)
    kmers = {g.label(v)[p:p + 16] for v in range(g.n_vertices) for p in range(lens[v] - 15)}
    feat, most = [], 0
    for i in range(len(qs)):
        q = qs.query(i)
        n = len(q)
        miss = sum(q[p:p + 16] not in kmers for p in (t * (n - 16) // 63 for t in range(64))) / 64 if n >= 16 else 0.0
        budget = (5 * n + 3) // 4 + 64
        f, b = reach(int(qs.v_s[i]), out, lens, budget), reach(int(qs.v_e[i]), back, lens, budget)
        most = max(most, len(f), len(b))
        s = {v for v in f if v in b and f[v] + lens[v] + b[v] <= budget}
        arcs = [(v, u) for v in s for u in out[v] if u in s]
        deg = {}
        for v, _ in arcs:
            deg[v] = deg.get(v, 0) + 1
        feat.append([math.log1p(n), miss, math.log1p(len(s)), math.log1p(len(arcs)),
                     sum(d > 1 for d in deg.values()) * 1000 / max(n, 1), math.log1p(sum(a in cyc for a in arcs))])
    return np.array(feat), most


def check(g, qs):
    import torch
    graph = gw.Graph.from_synth(g)
    model = gw.CostModel(graph)
    got = model.features(gw.DeviceBatch(qs))
    torch.cuda.synchronize()
    want, most = reference(g, qs)
    # log1pf of an integer below 2^24: an ulp of float32 or two
    assert np.allclose(got.cpu().numpy(), want, rtol=5e-7, atol=1e-7)
    return most


@pytest.mark.parametrize("length,n,fits", [(12, 20, True), (2000, 60, True), (20000, 20, True), (100_000, 3, False)])
def test_benchmark_graph(length, n, fits):
    g, _ = synth.make_config(2, n_queries=1)
    qs = synth.make_queries(g, n, 71, synth._const(length), synth._const(0.03), (1, 1, 1), (1, 1))
    if length == 12:   # shorter than a k-mer once cut
        qs = synth.Queries(qs.seq[:12 * n].copy(), np.arange(n + 1, dtype=np.uint64) * 12, qs.v_s, qs.v_e, qs.edits, qs.divergence)
    assert (check(g, qs) <= 768) == fits


# up to 608 queries get tables for 1,536 vertices a search, more than that 768; searches on
# both sides of what fits, and some beyond what the mean vertex length says will fit
@pytest.mark.parametrize("length,n", [(85_000, 12), (118_000, 12), (3000, 609), (52_000, 609)])
def test_table_sizes(length, n):
    g, _ = synth.make_config(2, n_queries=1)
    qs = synth.make_queries(g, n, 77, synth._const(length), synth._const(0.03), (1, 1, 1), (1, 1))
    check(g, qs)


def test_cycles_and_many_arcs():
    rng = np.random.default_rng(5)
    labels = ["".join("ACGT"[c] for c in rng.integers(0, 4, int(rng.integers(1, 40)))) for _ in range(120)]
    arcs = [(u, u + 1) for u in range(118)]   # vertex 119 is reached by nothing
    arcs += [(u, int(v)) for u in range(0, 118, 3) for v in rng.integers(0, 119, 6)]
    arcs += [(u, u) for u in range(0, 118, 10)]
    g = synth.Graph.from_lists(labels, arcs)
    m = 40
    seq = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, 100 * m)]
    vs, ve = rng.integers(0, 119, m).astype(np.uint32), rng.integers(0, 120, m).astype(np.uint32)
    ve[0] = 119
    qs = synth.Queries(seq, np.arange(m + 1, dtype=np.uint64) * 100, vs, ve, np.zeros(m, np.int64), np.zeros(m))
    check(g, qs)


# A vertex with more arcs than the 256 frontier slots of a search (forward, backward, both)
# sends it to the global-memory form in the middle of a step; with 1,300 queries some warps
# run two of them, one of each form
@pytest.mark.parametrize("out,back", [(255, 1), (257, 1), (1, 257), (400, 400)])
@pytest.mark.parametrize("n", [5, 1300])
def test_frontier_overflow(out, back, n):
    rng = np.random.default_rng(out + back)
    labels = ["".join("ACGT"[c] for c in rng.integers(0, 4, int(rng.integers(1, 20)))) for _ in range(60 + out + back)]
    arcs = [(v, v + 1) for v in range(59)]
    arcs += [(10, 60 + i) for i in range(out)] + [(60 + i, 11) for i in range(out)]
    arcs += [(40, 60 + out + i) for i in range(back)] + [(60 + out + i, 41) for i in range(back)]
    arcs += [(30, 29)]
    g = synth.Graph.from_lists(labels, arcs)
    lens = rng.integers(20, 400, n)
    seq = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, int(lens.sum()))]
    vs, ve = rng.integers(0, 30, n).astype(np.uint32), rng.integers(20, 60, n).astype(np.uint32)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    check(g, synth.Queries(seq, off, vs, ve, np.zeros(n, np.int64), np.zeros(n)))


# A dense stretch (a bubble every 9 bases) beside long vertices: searches of 1,300 and 3,400
# vertices that begin in shared memory and go on in global memory
@pytest.mark.parametrize("n,length", [(12, 3000), (620, 3000), (12, 8000), (620, 8000)])
def test_search_goes_on_in_global_memory(n, length):
    rng = np.random.default_rng(n + length)
    labels, arcs, walk = [], [], []
    for _ in range(1000):
        at = len(labels)
        labels.append("".join("ACGT"[c] for c in rng.integers(0, 4, 8)))
        a, b = rng.permutation(4)[:2]
        labels += ["ACGT"[a], "ACGT"[b]]
        arcs += [(at, at + 1), (at, at + 2), (at + 1, at + 3), (at + 2, at + 3)]
        walk += [at, at + 1 + int(rng.integers(2))]
    labels += ["ACGTTGCA", "".join("ACGT"[c] for c in rng.integers(0, 4, 300_000))]
    arcs += [(len(labels) - 2, len(labels) - 1), (len(labels) - 2, len(labels) - 3)]
    g = synth.Graph.from_lists(labels, arcs)
    qs, vs, ve = [], [], []
    for i in range(n):
        first = 2 * int(rng.integers(0, 650 if length < 5000 else 100))
        last = min(first + length * 2 // 9, len(walk) - 1)
        qs.append("".join(labels[v] for v in walk[first:last + 1])[:length])
        vs.append(walk[first])
        ve.append(walk[last])
    off = np.concatenate([[0], np.cumsum([len(q) for q in qs])]).astype(np.uint64)
    seq = np.frombuffer("".join(qs).encode(), np.uint8).copy()
    check(g, synth.Queries(seq, off, np.array(vs, np.uint32), np.array(ve, np.uint32), np.zeros(n, np.int64), np.zeros(n)))
