"""Uniform chains (uniform.cu) against the oracle and the simulator's units:
strides that divide the array, every policy, set counts that are not powers of
two, strides below and above a line, sets at the edges of the small and the
windowed play (n = a + 1, 31 .. 34 lines, hundreds), arrays that only claim to
be the chain, and the matcher."""
import math

import numpy as np
import pytest

import oracle
from paper_1509_02308_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1509_02308_gb300 import api

UNITS = {"head_streams": 2}  # every item in the simulator's units


def _forms():
    """(geometry, run): per accesses of one pass, n lines per set class."""
    out = []
    seed = 0x51AB
    for a, n in ((1, 2), (1, 5), (2, 3), (3, 4), (4, 5), (4, 4), (5, 9), (8, 9), (16, 19), (16, 32),
                 (16, 33), (30, 31), (31, 32), (31, 33), (32, 34), (33, 34), (40, 100), (512, 674)):
        for T in (1, 2, 3, 12, 48):
            if a * T > 2048:
                continue
            for pol in (W.LRU, W.FIFO, W.RANDOM, W.WEIGHTED):
                if pol == W.WEIGHTED and a < 3:
                    continue
                seed += 1
                b = (4, 32, 128)[seed % 3]
                lines = (n - 1) * T + 1 + seed % T  # the first classes hold n lines
                k = seed % 5
                if k == 0:      # several accesses a line
                    s, per = 1, lines * (b // 4) - seed % max(1, b // 4)
                elif k == 1:    # one access a line
                    s, per = b // 4, lines
                elif k == 2:    # every second line
                    s, per = 2 * (b // 4), lines
                elif k == 3:    # every third line
                    s, per = 3 * (b // 4), lines
                else:           # a stride that is not a power of two, below a line
                    s = max(1, 3 * (b // 4) // 8)
                    per = max(1, lines * (b // 4) // s)
                length = min(20000, 7 * per + seed % 61)
                if seed % 7 == 0:
                    length = per + 1
                if seed % 11 == 0:
                    length = max(1, per - 1)
                out.append((W.Geom(a * T * b, b, a, T, pol, seed * 0x9E3779B97F4A7C15 & (2**64 - 1)),
                            W.Run(per * s, s, length, min(length, per))))
    for m in (1, 2, 3):  # mappings from higher bits, whole and part blocks of lines
        for nb in (96 * 128, 97 * 32 * 4, 12288 + 32 * 5, 12288 + 512):
            for pol in (W.LRU, W.FIFO, W.RANDOM):
                out.append((W.Geom(12288, 32, 96, 4, pol, 77, mapping=m),
                            W.Run(nb // 4, 1, 4 * (nb // 4), nb // 4)))
    out.append((W.Geom(1024, 32, 4, 8, W.RANDOM, 3), W.Run(64, 64, 500, 1)))  # one element
    out.append((W.Geom(1024, 32, 4, 8, W.FIFO, 3), W.Run(4, 1, 500, 4)))      # one line
    return out


def _want(g, r):
    return oracle.cache_sim(g.C, g.b, g.ways, g.sets, g.policy,
                            oracle.pchase_trace(r.n_elems, r.stride, r.length), seed=g.seed,
                            mapping=g.mapping)


@pytest.mark.parametrize("explicit", [False, True])
def test_uniform_chains_match_oracle_and_units(explicit):
    forms = _forms()
    runs = [r for _, r in forms]
    if explicit:
        flat, offs = api.pchase_build_batch(runs)
        traces = [(flat[int(offs[i]):int(offs[i + 1])], r.length, r.warmup, r.n_elems, r.stride)
                  for i, r in enumerate(runs)]
    else:
        traces = [(None, r.length, r.warmup, r.n_elems, r.stride) for r in runs]
    pairs = [(i, i) for i in range(len(runs))]
    geoms = [g for g, _ in forms]
    got = {}
    for name, tune in (("uniform", None), ("units", UNITS)):
        plan = api.SimPlan(geoms, traces, pairs=pairs, tune=tune)
        assert ("uniform=" in plan.description) == (name == "uniform")
        st = api.status_word()
        bits, counts = plan.run(status=st)
        assert int(st.item()) == 0
        got[name] = (bits.cpu().numpy().view(np.uint32), counts.cpu().numpy().reshape(-1, 2))
        off = plan.word_offsets
        # counts alone (no bitmaps)
        _, only = plan.run(want_bitmaps=False)
        assert np.array_equal(only.cpu().numpy().reshape(-1, 2), got[name][1])
    assert np.array_equal(got["uniform"][0], got["units"][0])
    assert np.array_equal(got["uniform"][1], got["units"][1])
    words, counts = got["uniform"]
    for i, (g, r) in enumerate(forms):
        want = _want(g, r)
        have = api.unpack_bits(words[int(off[i]):], r.length)
        assert np.array_equal(have, want), (i, g, r, int(np.argmax(have != want)))
        assert counts[i].tolist() == [int(want.sum()), int(want[r.warmup:].sum())], (i, g, r)


def test_arrays_that_only_claim_to_be_chains():
    """One changed element anywhere sends the item to the units; so does an
    index out of range, which sets the status word as before."""
    rng = np.random.Generator(np.random.PCG64(9))
    geoms, traces, host = [], [], []
    for k, (N, s, L) in enumerate([(640, 32, 900), (4096, 8, 5000), (300, 3, 777), (96, 96, 50)] * 4):
        tr = oracle.pchase_trace(N, s, L)
        at = int(rng.integers(0, L)) if k % 4 else (0, 1, L - 2, L - 1)[k // 4 % 4]
        tr[at] = (int(tr[at]) + 1 + int(rng.integers(0, N))) % N
        host.append(tr)
        geoms.append(W.Geom(2048, 32, (2, 4, 8, 64)[k % 4], (32, 16, 8, 1)[k % 4], k % 3, 11 + k))
        buf = torch.empty(L + 3, dtype=torch.int32, device="cuda")
        t = buf[k % 4:k % 4 + L] if k % 4 + L <= L + 3 else buf[:L]  # every 4-byte alignment
        t.copy_(torch.from_numpy(tr.view(np.int32)))
        traces.append((t, L, L // 3, N, s))
    pairs = [(i, i) for i in range(len(geoms))]
    plan = api.SimPlan(geoms, traces, pairs=pairs)
    st = api.status_word()
    bits, _ = plan.run(status=st)
    assert int(st.item()) == 0
    words = bits.cpu().numpy().view(np.uint32)
    for i, (g, tr) in enumerate(zip(geoms, host)):
        want = oracle.cache_sim(g.C, g.b, g.ways, g.sets, g.policy, tr, seed=g.seed)
        have = api.unpack_bits(words[int(plan.word_offsets[i]):], tr.size)
        assert np.array_equal(have, want), (i, g)
    traces[1][0][17] = 1 << 20
    plan.run(status=st)
    assert int(st.item()) == 1


def test_matcher_over_uniform_chains():
    """Distances of the uniform path equal the units' (one observation and
    several), with traces above the played items' matcher limit among them."""
    runs = [W.Run(n // 4, s // 4, 3 * (n // s) + n % 7, n // s)
            for n, s in ((12288, 128), (16512, 128), (18432, 32), (2048, 4), (24576, 256))]
    runs.append(W.Run(18432 // 4, 1, 40000, 18432 // 4))
    cands = [W.Geom(C, b, a, C // (a * b), p, 5 + a) for C in (2048, 12288, 16384) for b in (32, 128)
             for a in (2, 4, 16) for p in (0, 1, 2)]
    traces = [(None, r.length, r.warmup, r.n_elems, r.stride) for r in runs]
    rng = np.random.Generator(np.random.PCG64(4))
    n = sum(r.length for r in runs)
    lat = torch.from_numpy((100.0 + 300.0 * (rng.random((3, n)) < 0.4)).astype(np.float32)).cuda()
    res = []
    for tune in (None, UNITS):
        plan = api.SimPlan(cands, traces, tune=tune)
        d1, p1 = plan.infer(lat[0])
        d3, p3 = api.infer_batch(plan, lat)
        res.append([x.cpu().numpy() for x in (d1, p1, d3, p3)])
    for x, y in zip(*res):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("n_geom", [15, 16, 70])
def test_matcher_groups_candidates(n_geom):
    """Candidates whose words are the same are matched together: line sizes,
    classes that overflow in part, mappings and unequal sets between them, one
    line to a pass, index arrays of which one is not the chain it claims."""
    runs = [W.Run(n // 4, s // 4, ln, n // s) for n, s, ln in
            ((4096, 128, 31), (8192, 32, 1025), (12416, 128, 300), (64, 64, 77), (20480, 4, 12000),
             (12288, 4096, 64), (16384, 128, 640))]
    flat, offs = api.pchase_build_batch(runs)
    flat[int(offs[6]) + 200] = 0
    traces = [(flat[int(offs[i]):int(offs[i + 1])] if i % 2 == 0 else None, r.length, r.warmup, r.n_elems,
               r.stride) for i, r in enumerate(runs)]
    cands = [W.Geom(C, b, a, C // (a * b), p, 3 * a) for b in (32, 128) for a in (1, 2, 4, 8)
             for C in (4096, 8192, 12288, 16384) for p in (0, 1, 2)]
    cands = cands[::96 // n_geom][:n_geom - 2] + [W.Geom(8192, 32, 4, 64, 0, 1, mapping=2),
                                                  W.Geom((3 * 4 + 5) * 128, 128, 4, 3, 0, 1, extra=5)]
    assert len(cands) == n_geom
    rng = np.random.Generator(np.random.PCG64(n_geom))
    n = sum(r.length for r in runs)
    lat = torch.from_numpy((100.0 + 300.0 * (rng.random((2, n)) < 0.4)).astype(np.float32)).cuda()
    res = []
    for tune in (None, UNITS):
        plan = api.SimPlan(cands, traces, tune=tune)
        d1, p1 = plan.infer(lat[0])
        d2, p2 = api.infer_batch(plan, lat)
        res.append([x.cpu().numpy() for x in (d1, p1, d2, p2)])
    for x, y in zip(*res):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("explicit", [False, True])
def test_long_small_sets_by_segments(explicit):
    """Overflowing sets of at most 32 lines with enough misses to be cut into
    segments: few and many ways, classes of which only the larger ones are cut,
    a line and several accesses to a line, weighted victims, plays that forget
    their start late or (28 lines in 20 ways) perhaps not in time, and traces
    that end anywhere in a segment."""
    forms = []
    for a, nl, T, stride, ln, pol in ((4, 6, 1, 8, 100003, W.RANDOM), (2, 9, 2, 8, 180000, W.RANDOM),
                                      (4, 11, 2, 8, 190001, W.RANDOM), (2, 4, 1, 8, 90000, W.RANDOM),
                                      (16, 23, 1, 8, 120000, W.RANDOM), (20, 28, 1, 16, 130007, W.RANDOM),
                                      (22, 32, 1, 8, 131000, W.RANDOM), (4, 6, 1, 1, 500000, W.RANDOM),
                                      (4, 7, 1, 8, 99999, W.WEIGHTED), (8, 36, 3, 8, 260000, W.RANDOM),
                                      (2, 3, 1, 8, 77777, W.RANDOM), (8, 11, 1, 8, 90000, W.RANDOM),
                                      (12, 16, 1, 8, 110000, W.RANDOM)):
        n = 8 * nl if stride <= 8 else stride * nl
        forms.append((W.Geom(a * T * 32, 32, a, T, pol, 1000 + 7 * len(forms)),
                      W.Run(n, stride, ln, n // stride)))
    runs = [r for _, r in forms]
    flat, offs = api.pchase_build_batch(runs)
    traces = [(flat[int(offs[i]):int(offs[i + 1])] if explicit else None, r.length, r.warmup, r.n_elems,
               r.stride) for i, r in enumerate(runs)]
    pairs = [(i, i) for i in range(len(runs))]
    geoms = [g for g, _ in forms]
    plan = api.SimPlan(geoms, traces, pairs=pairs)
    cut = int(plan.description.split("uniform=")[1].split()[0].split(",")[2])
    assert cut >= 3 * len(forms)  # every item is, into eight segments and more
    for _ in range(2):  # (the second run over the first one's states)
        bits, counts = plan.run()
    words, counts = bits.cpu().numpy().view(np.uint32), counts.cpu().numpy().reshape(-1, 2)
    for i, (g, r) in enumerate(forms):
        want = _want(g, r)
        have = api.unpack_bits(words[int(plan.word_offsets[i]):], r.length)
        assert np.array_equal(have, want), (i, g, r, int(np.argmax(have != want)))
        assert counts[i].tolist() == [int(want.sum()), int(want[r.warmup:].sum())], (i, g, r)


def test_uniform_run_captured_in_a_graph():
    runs = [W.Run(n // 4, 32, 4 * (n // 128), n // 128) for n in (8192, 16512, 20480)]
    flat, offs = api.pchase_build_batch(runs)
    traces = [(flat[int(offs[i]):int(offs[i + 1])], r.length, r.warmup, r.n_elems, r.stride)
              for i, r in enumerate(runs)]
    geoms = [W.Geom(16384, 128, 4, 32, p, 9) for p in (0, 1, 2)]
    plan = api.SimPlan(geoms, traces)
    bits, counts = plan.run()
    want = (bits.clone(), counts.clone())
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.run(bits, counts, stream=torch.cuda.current_stream())
    bits.zero_()
    counts.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(bits, want[0]) and torch.equal(counts, want[1])
    assert math.prod(counts.shape) == 2 * len(geoms) * len(runs)
