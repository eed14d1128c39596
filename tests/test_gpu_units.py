"""Chains whose stride divides their array, stepped by the simulator's units all
the same (tune head_streams=2: the plan's set modes, splits, time parts, head
streams and unit loops, and no uniform chains): the whole batched workload at
full length under every plan of test_gpu_full_batch.py, and the chains cut in
time of test_gpu_time_split.py, against the oracle bit for bit."""
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import oracle
from paper_1509_02308_gb300 import workloads as W
from test_gpu_full_batch import _run
from test_gpu_time_split import TUNES, _want, host_traces, lru_geoms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1509_02308_gb300 import api, autotune

UNITS = {"head_streams": 2}


def _fields(description):
    return dict(kv.split("=", 1) for kv in description.split())


def test_whole_batch_in_the_units():
    geoms, runs = W.config2()
    flat, offs = api.pchase_build_batch(runs)
    traces = [(flat[int(offs[i]):int(offs[i + 1])], r.length, r.warmup, r.n_elems, r.stride)
              for i, r in enumerate(runs)]
    pairs = [(i, i) for i in range(len(runs))]
    timed = autotune.lookup(geoms, traces, pairs) or {}
    variants = {"timed": dict(timed, **UNITS), "default": UNITS,
                "scans": {"batch_max_sets": 0xFFFFFFFF, "scan_max_ways": 16, "max_split": 8, **UNITS},
                "splits": {"batch_max_sets": 1 << 30, "split_cost_ns": 2_000_000, **UNITS},
                "shared_loop": dict(timed, kind_affinity=0xFFFFFFFF, **UNITS)}
    results = {k: _run(geoms, traces, pairs, v) for k, v in variants.items()}
    for name, (_, _, _, description) in results.items():
        d = _fields(description)
        assert "uniform" not in d, (name, description)
        if name != "scans":
            assert "streams" in d and int(d["split"]) >= 1 and int(d["time_split"]) >= 1, (name, description)
    del traces, flat
    torch.cuda.empty_cache()

    def one(i):
        g, r = geoms[i], runs[i]
        want = oracle.cache_sim(g.C, g.b, g.ways, g.sets, g.policy,
                                oracle.pchase_trace(r.n_elems, r.stride, r.length), seed=g.seed)
        bad = []
        for name, (bits, counts, woffs, _) in results.items():
            w0 = int(woffs[i])
            got = api.unpack_bits(bits[w0:w0 + (r.length + 31) // 32], r.length)
            if not np.array_equal(got, want):
                bad.append((name, i, "bitmap", int(np.argmax(got != want))))
            elif (int(counts[i, 0]) != int(want.sum())
                  or int(counts[i, 1]) != int(want[r.warmup:].sum())):
                bad.append((name, i, "counts"))
        return bad

    order = sorted(range(len(runs)), key=lambda i: -runs[i].length * max(1, geoms[i].ways))
    with ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as ex:
        bad = [b for r in ex.map(one, order) for b in r]
    assert not bad, bad[:10]


@pytest.mark.parametrize("tune_name", list(TUNES))
def test_time_parts_of_chains_in_the_units(tune_name):
    rng = np.random.Generator(np.random.PCG64(31))
    geoms = lru_geoms()
    host, descs = host_traces(rng)
    plan = api.SimPlan(geoms, descs, tune=dict(TUNES[tune_name] or {}, **UNITS))
    d = _fields(plan.description)
    assert "uniform" not in d, plan.description
    if tune_name != "default":
        assert int(d["time_split"]) >= 10, plan.description
    bitmaps, counts = plan.run()
    torch.cuda.synchronize()
    b = bitmaps.cpu().numpy().view(np.uint32)
    c = counts.view(-1, 2).cpu().numpy()
    for gi, g in enumerate(geoms):
        for ti, (tr, ds) in enumerate(zip(host, descs)):
            i = gi * len(host) + ti
            want = _want(g, tr)
            got = api.unpack_bits(b[int(plan.word_offsets[i]):], tr.size)
            assert np.array_equal(got, want), (tune_name, g, ti, int(np.argmax(got != want)))
            assert c[i, 0] == want.sum() and c[i, 1] == want[ds[2]:].sum(), (tune_name, g, ti)
