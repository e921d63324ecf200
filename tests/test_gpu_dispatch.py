"""Launch rules do not change results: the CTA width that the engine chooses for a batch
(on the host where it knows the lengths, on the device where it does not), and the two
ways a host-buffer batch and a single call bring their inputs over."""
import numpy as np
import pytest

import oracle
import paper_2206_13574_gb300 as gw
from paper_2206_13574_gb300 import _build, synth

pytestmark = pytest.mark.gpu
FIELDS = [f for f in gw.RESULT_DTYPE.names if f != "device_us"]


@pytest.fixture(scope="module")
def graph():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    _build.build()
    oracle.build()
    g, _ = synth.make_config(2, n_queries=1)
    return g, gw.Graph.from_synth(g)


# 1 query per SM of 600 bases mean, or 180, are where the width changes (152 SMs)
@pytest.mark.parametrize("n,length", [(1, 0), (1, 5000), (152, 599), (152, 601), (152, 179), (152, 181),
                                      (300, 2000), (900, 900), (2000, 150), (2000, 3000)])
@pytest.mark.parametrize("mode", ["exact", "lag", "traceback"])
def test_chosen_width(graph, n, length, mode):
    import torch
    g, gr = graph
    if length:
        qs = synth.make_queries(g, n, 7 + n, synth._const(length), synth._uniform(0.0, 0.04), (1, 1, 1), (1, 1))
    else:   # nothing but empty queries
        qs = synth.Queries(np.zeros(0, np.uint8), np.zeros(n + 1, np.uint64), np.zeros(n, np.uint32),
                           np.zeros(n, np.uint32), np.zeros(n, np.int64), np.zeros(n))
    prune = mode != "exact"
    opts = dict(max_lag=60 if mode == "lag" else 0)
    cfg = gw.default_config(gr, prune=prune)
    cfg.threads = 64
    want = gw.Engine(gr, prune=prune, config=cfg).align_batch(qs.seq, qs.off, qs.v_s, qs.v_e, **opts)
    eng = gw.Engine(gr, prune=prune)
    host = eng.align_batch(qs.seq, qs.off, qs.v_s, qs.v_e, **opts)
    got = [host]
    if length:   # a device batch without a base is refused
        batch = gw.DeviceBatch(qs)
        batch.run(eng, traceback=mode == "traceback", **opts)
        torch.cuda.synchronize()
        got.append(batch.results())
    for res in got:
        for f in FIELDS:
            assert np.array_equal(res[f], want[f]), f
    for i in range(0, n, max(1, n // 5)):
        w = oracle.gwfa(g, qs.query(i), int(qs.v_s[i]), int(qs.v_e[i]), a_diff=opts["max_lag"])
        assert (int(want[i]["edit_distance"]), int(want[i]["cells"])) == (w["distance"], w["cells"])


# a width that the configuration names is the one that runs: one launch a tier, while the
# engine's own choice for a device batch is settled there, among three launches of tier 0
@pytest.mark.parametrize("threads", [0, 128, 256, 512, 1024, None])
def test_configured_width(graph, threads):
    import torch
    g, gr = graph
    qs = synth.make_queries(g, 100, 3, synth._const(900), synth._const(0.02), (1, 1, 1), (1, 1))
    cfg = gw.default_config(gr)
    assert cfg.threads == gw.GWFA_THREADS_AUTO
    if threads is not None:
        cfg.threads = threads
    eng = gw.Engine(gr, config=cfg)
    batch = gw.DeviceBatch(qs)
    batch.run(eng)
    torch.cuda.synchronize()
    assert eng.last_launches == (3 if threads is not None else 5)
    want = gr.align(qs.query(0), int(qs.v_s[0]), int(qs.v_e[0]))
    assert int(batch.results()[0]["cells"]) == want["cells"]


@pytest.mark.parametrize("kb", [2, 250, 260, 700])   # one copy up to 256 KB of inputs
def test_host_batch_inputs(graph, kb):
    g, gr = graph
    qs = synth.make_queries(g, kb, 3, synth._const(1000), synth._const(0.02), (1, 1, 1), (1, 1))
    seq = qs.seq.copy()
    seq[int(qs.off[1])] = ord("N")   # query 1 is not ACGT
    eng = gw.Engine(gr)
    order = np.arange(kb, dtype=np.uint32)[::-1].copy()
    a = eng.align_batch(seq, qs.off, qs.v_s, qs.v_e, order=order)
    b = eng.align_batch(seq, qs.off, qs.v_s, qs.v_e)
    for f in FIELDS:
        assert np.array_equal(a[f], b[f]), f
    assert a["status"][1] == gw.GWFA_ERR_INVALID and (np.delete(a["status"], 1) == 0).all()
    w = oracle.gwfa(g, qs.query(0), int(qs.v_s[0]), int(qs.v_e[0]))
    assert (int(a[0]["edit_distance"]), int(a[0]["cells"])) == (w["distance"], w["cells"])


def test_single_calls(graph):
    """Lengths around the packed word and the plain path's change of width, either case,
    a base outside ACGT, and vertices that cannot be reached."""
    g, gr = graph
    base = synth.make_queries(g, 1, 11, synth._const(3200), synth._const(0.01), (1, 1, 1), (1, 1))
    q, vs, ve = base.query(0), int(base.v_s[0]), int(base.v_e[0])
    for n in (0, 1, 15, 16, 17, 33, 2999, 3000, 3001, len(q)):
        w = oracle.gwfa(g, q[:n], vs, vs)
        for text in (q[:n], q[:n].lower()):
            r = gr.align(text, vs, vs)
            assert (r["edit_distance"], r["cells"], r["visited"]) == (w["distance"], w["cells"], w["visited"]), n
    r, walk = gr.align_path(q, vs, ve)
    assert r["edit_distance"] == oracle.gwfa(g, q, vs, ve)["distance"] and walk[0] == vs and walk[-1] == ve
    bad = gr.align(q[:100] + b"N" + q[100:], vs, ve)
    assert (bad["status"], bad["edit_distance"], bad["cells"]) == (gw.GWFA_ERR_INVALID, -1, 0)
    assert gr.align(q, ve, vs)["status"] == gw.GWFA_ERR_UNREACHABLE
    assert gr.align(q, vs, ve)["edit_distance"] == r["edit_distance"]   # and the path works on


# more queries than SMs run longest first when the batch brings no order: every length
# class from empty on, classes of one query and of many, and one query over 1,024 of them
@pytest.mark.parametrize("n", [153, 305, 1025, 4097])
def test_batch_without_order(graph, n):
    import torch
    g, gr = graph
    rng = np.random.default_rng(n)
    lens = np.where(rng.random(n) < 0.1, rng.integers(0, 4, n), (2.0 ** rng.uniform(2, 11, n)).astype(np.int64))
    qs = synth.make_queries(g, n, n, synth._const(2100), synth._uniform(0.0, 0.02), (1, 1, 1), (1, 1))
    seq = np.concatenate([np.frombuffer(qs.query(i), np.uint8)[:lens[i]] for i in range(n)])
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    cut = synth.Queries(seq, off, qs.v_s, qs.v_s, qs.edits, qs.divergence)
    eng = gw.Engine(gr)
    want = eng.align_batch(seq, off, cut.v_s, cut.v_e, order=np.arange(n, dtype=np.uint32))
    batch = gw.DeviceBatch(cut)
    batch.run(eng)
    torch.cuda.synchronize()
    for res in (batch.results(), eng.align_batch(seq, off, cut.v_s, cut.v_e)):
        for f in FIELDS:
            assert np.array_equal(res[f], want[f]), f


def test_launches_of_a_batch_without_order(graph):
    import torch
    g, gr = graph
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n, sort in ((sms, 0), (sms + 1, 1)):
        qs = synth.make_queries(g, n, 3, synth._const(300), synth._const(0.01), (1, 1, 1), (1, 1))
        cfg = gw.default_config(gr)
        cfg.threads = 128
        eng = gw.Engine(gr, config=cfg)
        batch = gw.DeviceBatch(qs)
        batch.run(eng)
        assert eng.last_launches == 3 + sort                # three tiers
        eng.align_batch(qs.seq, qs.off, qs.v_s, qs.v_e)
        assert eng.last_launches == 3 + 1 + sort            # and the packing
        eng.align_batch(qs.seq, qs.off, qs.v_s, qs.v_e, order=np.arange(n))
        assert eng.last_launches == 3 + 1


@pytest.mark.parametrize("prune", [False, True])
def test_autotuner_knows_the_size_of_a_slab(graph, prune):
    from paper_2206_13574_gb300 import autotune
    g, gr = graph
    size = []
    for ctas in (8, 24):
        cfg = gw.default_config(gr, prune=prune)
        cfg.n_tiers, cfg.tiers[0].ctas, cfg.tiers[0].log2_tiles = 1, ctas, 14
        size.append(gw.Engine(gr, prune=prune, config=cfg).device_bytes)
    estimate = autotune._tier0_bytes(16, 14, prune)
    assert abs(size[1] - size[0] - estimate) < 0.001 * estimate


# up to four queries an SM start on tier 1's slabs: tier 0's would overflow here, and some
# queries leave tier 1's as well (or have no tier to go to)
@pytest.mark.parametrize("n,tiers", [(20, 3), (152, 3), (300, 3), (300, 2), (300, 1)])
def test_few_queries_start_on_tier_1(graph, n, tiers):
    import torch
    g, gr = graph
    qs = synth.make_queries(g, n, 5, synth._const(5000), synth._uniform(0.0, 0.08), (1, 1, 1), (1, 1))
    cfg = gw.default_config(gr)
    cfg.n_tiers = tiers
    cfg.tiers[0].log2_tiles, cfg.tiers[1].log2_tiles, cfg.tiers[2].log2_tiles = 8, 12, 17
    fixed = gw.default_config(gr)
    fixed.threads, fixed.n_tiers = 256, tiers
    for t in range(3):
        fixed.tiers[t].log2_tiles = cfg.tiers[t].log2_tiles
    want = gw.Engine(gr, config=fixed).align_batch(qs.seq, qs.off, qs.v_s, qs.v_e)
    eng = gw.Engine(gr, config=cfg)
    batch = gw.DeviceBatch(qs)
    batch.run(eng)
    torch.cuda.synchronize()
    assert (want["status"] == 0).all() == (tiers == 3)
    for res in (batch.results(), eng.align_batch(qs.seq, qs.off, qs.v_s, qs.v_e)):
        assert np.array_equal(res["status"], want["status"])
        for f in FIELDS:   # a query that ends without room reports what it did until then
            assert np.array_equal(res[f][want["status"] == 0], want[f][want["status"] == 0]), f


@pytest.mark.parametrize("huge,wide", [(0, 700), (300, 400), (160, 0), (3, 2)])
def test_more_class_ctas_than_fit(graph, huge, wide):
    """Classes with more CTAs than the GPU holds beside tier 0 run on fewer."""
    import torch
    g, gr = graph
    qs = synth.make_queries(g, 900, 17, synth._const(1500), synth._uniform(0.0, 0.05), (1, 1, 1), (1, 1))
    order = np.argsort(-qs.edits, kind="stable").astype(np.uint32)
    want = gw.Engine(gr).align_batch(qs.seq, qs.off, qs.v_s, qs.v_e)
    cfg = gw.default_config(gr)
    cfg.wide.ctas, cfg.wide.log2_tiles, cfg.wide.threads = wide, 14, 512
    cfg.huge.ctas, cfg.huge.log2_tiles, cfg.huge.threads = huge, 15, 1024
    eng = gw.Engine(gr, config=cfg)
    batch = gw.DeviceBatch(qs, order=order)
    batch.run(eng, n_wide=wide, n_huge=huge)
    torch.cuda.synchronize()
    res = batch.results()
    for f in FIELDS:
        assert np.array_equal(res[f], want[f]), f
