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
