"""Performance cases of the fine-grained P-chase framework.

Each case is one call (or the two or three calls that belong together) that a
user of the package makes: replaying P-chase traces through simulated caches,
recovering a geometry from latencies, and the learned inverse.  Sizes are the
ones of the repository's workloads, tests and benchmark, with ragged ones
between them.  Nothing here checks results.
"""
import math

import numpy as np
import torch

from paper_1509_02308_gb300 import api
from paper_1509_02308_gb300 import inverse as INV
from paper_1509_02308_gb300 import workloads as W

DEV = "cuda"
POINTS, CH, TAPS, FLAT, HIDDEN, LOGITS = 512, 64, 5, 2048, 256, 31
HEADS = (17, 4, 7, 3)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one cache under the paper's array-size sweep (Sec. 4.1): the interactive
        # call of somebody who fits one geometry by hand; bound by latency
        {"name": "sweep_one_cache", "kind": "sweep", "passes": 3, "step_bytes": 128},
        # a few hundred short traces: a user's own batch of geometries
        {"name": "sim_short_384", "kind": "sim", "items": 384, "max_len": 16384},
        # the benchmark's batch: 4096 geometries x P-chase traces of 1K-1M accesses
        {"name": "sim_batch_4096", "kind": "sim", "items": 4096, "max_len": 1 << 20},
        # build the traces and simulate them in one-shot form, planning included
        {"name": "oneshot_256", "kind": "oneshot", "items": 256, "max_len": 65536},
        # L1 -> L2 and L1 TLB -> L2 TLB cascades over analytic streams
        {"name": "hierarchy_512", "kind": "hierarchy", "items": 512},
        # texture L1 (bits 7-8 mapping) and Fermi L1 (weighted policy) sweeps
        {"name": "variants", "kind": "variants", "fermi_seeds": 64, "passes": 4},
        # the miss-rate table of some candidates over the 512-point plan, which
        # the learned inverse trains on
        {"name": "rate_table_64", "kind": "rates", "candidates": 64},
        # exhaustive inference of one observation: 1308 candidates x 108 traces
        {"name": "infer_one", "kind": "infer", "observations": 1},
        # latencies of many runs to hit / miss bits
        {"name": "classify_64x64k", "kind": "classify", "observations": 64, "max_len": 65536},
        # the network alone over a large batch of mean-latency traces
        {"name": "network_65536", "kind": "network", "traces": 65536},
        # one training step at the training batch
        {"name": "train_4096", "kind": "train", "batch": 4096},
        # the least-squares judge, also the network's fallback
        {"name": "lsq_8192", "kind": "lsq", "traces": 8192, "candidates": 1308},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("sweep", "sim", "sim", "sim", "oneshot", "hierarchy", "variants", "rates",
                       "infer", "classify", "network", "network", "train", "train", "lsq"))
    if kind == "sweep":
        return {"kind": kind, "passes": rng.randint(2, 8), "step_bytes": 32 * rng.randint(1, 8)}
    if kind == "sim":
        return {"kind": kind, "items": _log_int(rng, 16, 4096), "max_len": _log_int(rng, 2048, 1 << 20)}
    if kind == "oneshot":
        return {"kind": kind, "items": _log_int(rng, 8, 1024), "max_len": _log_int(rng, 2048, 1 << 18)}
    if kind == "hierarchy":
        return {"kind": kind, "items": _log_int(rng, 16, 512)}
    if kind == "variants":
        return {"kind": kind, "fermi_seeds": _log_int(rng, 1, 64), "passes": rng.randint(2, 6)}
    if kind == "rates":
        return {"kind": kind, "candidates": _log_int(rng, 2, 64)}
    if kind == "infer":
        return {"kind": kind, "observations": rng.randint(2, 12)}
    if kind == "classify":
        return {"kind": kind, "observations": _log_int(rng, 1, 256),
                "max_len": _log_int(rng, 1024, 1 << 17)}
    if kind == "network":
        return {"kind": kind, "traces": _log_int(rng, 1, 65536)}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 16, 4096)}
    return {"kind": kind, "traces": _log_int(rng, 16, 8192), "candidates": _log_int(rng, 64, 1308)}


# ------------------------------------------------------- simulator inputs
def _built(runs):
    """The runs' index arrays on the GPU, as trace descriptors."""
    flat, offs = api.pchase_build_batch(runs)
    return [(flat[int(offs[i]):int(offs[i + 1])], r.length, r.warmup, r.n_elems, r.stride)
            for i, r in enumerate(runs)]


def _uniform(n_bytes, stride_bytes, passes):
    """A uniform run of `passes` passes, the first one warm-up."""
    n, s = max(1, n_bytes // 4), max(1, stride_bytes // 4)
    per = n // math.gcd(n, s)
    return W.Run(n, s, passes * per, per)


def _sweep_runs(case):
    """12-24 KB arrays, stride 128 B."""
    return [_uniform(nb, 128, case["passes"]) for nb in range(12288, 24577, case["step_bytes"])]


def _sweep_geom(seed):
    """A 16 KB cache of 128 B lines: its ways and policy differ with the seed."""
    ways = (4, 2, 8, 16)[seed % 4]
    return W.Geom(16384, 128, ways, 128 // ways, (W.LRU, W.FIFO, W.RANDOM)[seed // 4 % 3], seed)


def _with_lengths(runs, lens):
    """The runs, each as long as `lens` says (a case's outputs keep their sizes)."""
    return [W.Run(r.n_elems, r.stride, n, min(n, r.n_elems // math.gcd(r.n_elems, r.stride)))
            for r, n in zip(runs, lens)]


def _batch(case, seed):
    """The batched-simulation workload: geometries, strides and array sizes
    from the seed, lengths from the case alone."""
    _, fixed = W.config2(case["items"], max_len=case["max_len"])
    geoms, runs = W.config2(case["items"], seed_base=0x5EED0002 + 1000003 * (seed + 1),
                            max_len=case["max_len"])
    return geoms, _with_lengths(runs, [r.length for r in fixed])


def _variant_items(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    geoms, runs, pairs = [], [], []

    def add(g, sizes, strides):
        first = len(runs)
        runs.extend(_uniform(nb, sb, case["passes"]) for nb in sizes for sb in strides)
        return first, len(runs)

    for C, ways in ((12288, 96), (24576, 192)):
        geoms.append(W.Geom(C, 32, ways, 4, W.LRU, mapping=2))
        sizes = list(range(C, C + 513, 32)) + list(range(C + 1024, 61441, 1024))
        a, b = add(geoms[-1], sizes, (4, 32))
        pairs += [(len(geoms) - 1, t) for t in range(a, b)]
    a, b = add(None, range(15 * 1024, 24 * 1024 + 1, 128), (4, 128))
    for _ in range(case["fermi_seeds"]):
        geoms.append(W.Geom(16384, 128, 4, 32, W.WEIGHTED, int(rng.integers(1, 1 << 62))))
        pairs += [(len(geoms) - 1, t) for t in range(a, b)]
    return geoms, runs, pairs


def _infer_runs():
    """The one-geometry configuration with stride-4 B runs around its capacity."""
    truth, runs = W.config1()
    for d in (-4, 0, 4, 32, 36, 64, 68, 128, 132, 256, 260):
        runs.append(_uniform(truth.C + d, 4, 3))
    return runs


def _hierarchy(case, seed):
    fixed = W.hierarchy_config(case["items"])[-1]
    *levels, runs = W.hierarchy_config(case["items"], seed_base=0x5EED0005 + 1000003 * (seed + 1))
    return (*levels, _with_lengths(runs, [r.length for r in fixed]))


def _bits_of(words, n):
    """LSB-first packed miss bits (an int32 tensor) as n truth values."""
    sh = torch.arange(32, device=words.device, dtype=torch.int32)
    return ((words.view(-1, 1) >> sh) & 1).reshape(-1)[:n].bool()


# ------------------------------------------------ latencies and mean-latency traces
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _latencies(miss, g):
    """Per-access latencies: two plateaus with 2 % jitter and a few spikes."""
    lat = 100.0 + 300.0 * miss.float()
    lat = lat * (1.0 + 0.02 * torch.randn(lat.shape, device=DEV, generator=g))
    spike = torch.rand(lat.shape, device=DEV, generator=g) < 0.002
    return torch.where(spike, lat * (2.0 + 8.0 * torch.rand(lat.shape, device=DEV, generator=g)), lat)


def _plan_rates(n, g):
    """Miss-rate rows over a 512-point plan for n cache geometries drawn from
    the grid: zero up to the capacity, a ramp as sets overflow one after the
    other, then the stride's plateau; the last points tell the policies apart."""
    def pick(k):
        return torch.randint(0, k, (n, 1), device=DEV, generator=g)

    cap = torch.tensor(W.CAPACITIES, dtype=torch.float32, device=DEV)[pick(17)]
    line = 32.0 * 2.0 ** pick(4).float()
    ways = 2.0 ** pick(4).float()
    policy = pick(3)

    def sizes(lo, hi, k):
        return lo * (hi / lo) ** (torch.arange(k, device=DEV) / (k - 1.0))

    def seg(nb, sb):
        over = (nb.view(1, -1) - cap) * ways / cap
        lru = over.clamp(0.0, 1.0)
        rand = (over / (over.abs() + 0.25 * ways + 0.5)).clamp(0.0, 1.0)
        return torch.where(policy == 2, rand, lru) * (sb / line).clamp(max=1.0)

    rows = [seg(sizes(512, 524288, 176), 4.0), seg(sizes(512, 524288, 176), 32.0),
            seg(sizes(1024, 524288, 61), 128.0)]
    stride = 4.0 * 2.0 ** torch.arange(35, device=DEV).remainder(18).float()
    left = 524288.0 / stride.view(1, -1) * line > cap  # the lines visited do not fit
    rows.append(torch.where(left, (stride.view(1, -1) / line).clamp(max=1.0), torch.zeros_like(cap)))
    fits = (sizes(1024, 262144, 32).view(1, -1) <= cap).float()
    hot = torch.where(policy == 0, 0.5 * torch.ones_like(cap), 0.5625 + 0.0625 * policy.float())
    for step in (32.0, 256.0):
        rows.append((fits * hot + (1.0 - fits)) * (step / line).clamp(max=1.0))
    # a rate is a count over at most 2^15 accesses
    return (torch.round(torch.cat(rows, 1) * 32768.0) / 32768.0).contiguous()


def _mean_traces(rates, n, g):
    """n mean-latency traces t0 + (t1 - t0) r of random rows, 2 % jitter, 0.5 %
    spikes, min-max normalised."""
    r = rates[torch.randint(0, rates.shape[0], (n,), device=DEV, generator=g)]
    u = torch.rand(n, 2, device=DEV, generator=g)
    t0 = 20.0 + 380.0 * u[:, :1]
    rho = torch.exp(math.log(1.5) + math.log(20.0) * u[:, 1:])
    y = (t0 + t0 * (rho - 1.0) * r) * (1.0 + 0.02 * torch.randn(r.shape, device=DEV, generator=g))
    spike = torch.rand(r.shape, device=DEV, generator=g) < 0.005
    y = torch.where(spike, y * (2.0 + 8.0 * torch.rand(r.shape, device=DEV, generator=g)), y)
    lo, hi = y.amin(1, keepdim=True), y.amax(1, keepdim=True)
    return ((y - lo) / (hi - lo)).contiguous()


# ------------------------------------------------------------ network weights
def _layers():
    """(rows, columns) of each weight matrix, first to last; a bias of `rows`
    follows each."""
    return [(CH, TAPS), (CH, TAPS * CH), (CH, TAPS * CH), (CH, TAPS * CH), (HIDDEN, FLAT),
            (LOGITS, HIDDEN)]


def _weights(g):
    parts = []
    for r, c in _layers():
        s = math.sqrt(6.0 / c)
        parts.append(((2.0 * torch.rand(r * c, device=DEV, generator=g) - 1.0) * s))
        parts.append((2.0 * torch.rand(r, device=DEV, generator=g) - 1.0) * 0.1)
    return torch.cat(parts)


def _moments(n, g):
    """Adam moments as some steps of training leave them."""
    m = 1e-4 * torch.randn(n, device=DEV, generator=g)
    v = (1e-3 * (0.5 + torch.rand(n, device=DEV, generator=g))) ** 2
    return m, v


def _network_inputs(case, seed):
    g = _gen(seed)
    w = _weights(g)
    return w, _mean_traces(_plan_rates(512, g), case["traces"], g)


def _train_inputs(case, seed):
    g = _gen(seed)
    w = _weights(g)
    m, v = _moments(w.numel(), g)
    x = _mean_traces(_plan_rates(512, g), case["batch"], g)
    lab = torch.stack([torch.randint(0, k, (case["batch"],), device=DEV, generator=g)
                       for k in HEADS], 1).to(torch.int32).contiguous()
    return w, m, v, x, lab


def _lsq_inputs(case, seed):
    g = _gen(seed)
    rates = _plan_rates(case["candidates"], g)
    return rates, _mean_traces(rates, case["traces"], g)


def _classify_lengths(case):
    rng, top = np.random.Generator(np.random.PCG64(1)), case["max_len"]
    return [top if i == 0 else int(rng.integers(max(1, top // 4), top + 1))
            for i in range(case["observations"])]


def _classify_inputs(case, seed):
    g = _gen(seed)
    rng = np.random.Generator(np.random.PCG64(seed))
    lats = []
    for n in _classify_lengths(case):
        rate = float(rng.uniform(0.02, 0.9))
        lats.append(_latencies(torch.rand(n, device=DEV, generator=g) < rate, g))
    return lats


def _load(net, w):
    net.weights().copy_(w)
    net.param_array(1).copy_(w.bfloat16())


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        runs = _sweep_runs(case)
        return kind, api.SimPlan([_sweep_geom(seed)], _built(runs), pairs=[(0, t) for t in range(len(runs))])
    if kind == "sim":
        geoms, runs = _batch(case, seed)
        return kind, api.SimPlan(geoms, _built(runs), pairs=[(i, i) for i in range(len(runs))])
    if kind == "oneshot":
        return kind, _batch(case, seed)
    if kind == "hierarchy":
        l1, l2, t1, t2, runs = _hierarchy(case, seed)
        traces = [(None, r.length, r.warmup, r.n_elems, r.stride) for r in runs]
        pairs = [(i, i) for i in range(len(runs))]
        return kind, (api.HierarchyPlan([l1, l2], traces, pairs=pairs),
                      api.HierarchyPlan([t1, t2], traces, pairs=pairs))
    if kind == "variants":
        geoms, runs, pairs = _variant_items(case, seed)
        return kind, api.SimPlan(geoms, _built(runs), pairs=pairs)
    if kind == "rates":
        rng = np.random.Generator(np.random.PCG64(seed))
        every = INV.candidate_table(seed_base=0x5EED + 7919 * seed)
        cands = [every[int(i)] for i in rng.choice(len(every), case["candidates"], replace=False)]
        pts, traces, keep = INV.plan_traces()
        return kind, (api.SimPlan(cands, traces), keep)
    if kind == "infer":
        runs = _infer_runs()
        traces = _built(runs)
        cands = [W.Geom(C, b, a, T, p, 0x5EED + i)
                 for i, (C, b, a, T) in enumerate(W.geometry_grid()) for p in (0, 1, 2)]
        near = [c for c in cands if 8192 <= c.C <= 32768]
        truth = near[seed % len(near)]
        words, _, offs = api.cache_sim_batch([truth], traces, pairs=[(0, t) for t in range(len(traces))])
        miss = torch.cat([_bits_of(words[int(offs[t]):int(offs[t + 1])], r.length)
                          for t, r in enumerate(runs)])
        g = _gen(seed)
        lats = torch.stack([_latencies(miss, g) for _ in range(case["observations"])])
        return kind, (api.SimPlan(cands, traces), lats)
    if kind == "classify":
        return kind, _classify_inputs(case, seed)
    if kind == "network":
        w, x = _network_inputs(case, seed)
        net = INV.LearnedInverse(max_batch=case["traces"], infer_only=True)
        _load(net, w)
        return kind, (net, x)
    if kind == "train":
        w, m, v, x, lab = _train_inputs(case, seed)
        net = INV.LearnedInverse(max_batch=case["batch"])
        net.init(1)
        _load(net, w)
        net.param_array(3).copy_(m)
        net.param_array(4).copy_(v)
        return kind, (net, x, lab, torch.zeros(1, device=DEV))
    return kind, _lsq_inputs(case, seed)


TRAIN_STEP, TRAIN_LR = 100, 1e-3


def run(state):
    kind, s = state
    if kind in ("sweep", "sim", "variants"):
        return s.run()
    if kind == "oneshot":
        geoms, runs = s
        traces = _built(runs)
        bitmaps, counts, _ = api.cache_sim_batch(geoms, traces, pairs=[(i, i) for i in range(len(runs))])
        return bitmaps, counts
    if kind == "hierarchy":
        return s[0].run() + s[1].run()
    if kind == "rates":
        return s[0].run(want_bitmaps=False)[1]
    if kind == "infer":
        plan, lats = s
        return plan.infer(lats[0]) if lats.shape[0] == 1 else api.infer_batch(plan, lats)
    if kind == "classify":
        bits, _, thr = api.pchase_classify(s)
        return bits, thr
    if kind == "network":
        net, x = s
        pred, conf, logits = net.infer(x, want_logits=True)
        return {"pred": pred, "conf": conf, "logits": logits}
    if kind == "train":
        net, x, lab, loss = s
        loss.zero_()
        INV._check(net.L.pchase_inverse_train_step(
            net.h, net._p, net._w, x.data_ptr(), lab.data_ptr(), x.shape[0], TRAIN_LR, TRAIN_STEP,
            loss.data_ptr(), torch.cuda.current_stream().cuda_stream))
        return {"loss": loss, "grad": net.param_array(2), "w": net.weights(),
                "m": net.param_array(3), "v": net.param_array(4)}
    rates, y = s
    return INV.lsq_match(rates, y)


# ------------------------------------------------------------------- the work
def _sim_bytes(runs, pairs=None, analytic=False):
    """Index arrays read once, one bit per simulated access and two 64-bit
    counts per item written."""
    lens = [r.length for r in runs] if pairs is None else [runs[t].length for _, t in pairs]
    read = 0 if analytic else 4 * sum(r.length for r in runs)
    return read + sum(4 * ((n + 31) // 32) + 16 for n in lens)


def work(case):
    kind = case["kind"]
    macs = sum(r * c for r, c in _layers()[4:])
    macs += sum(CH * TAPS * cin * out for cin, out in ((1, 256), (CH, 128), (CH, 64), (CH, 32)))
    n_par = sum(r * c + r for r, c in _layers())
    if kind == "sweep":
        return {"bytes": _sim_bytes(_sweep_runs(case)), "flops": 0}
    if kind in ("sim", "oneshot"):
        _, runs = _batch(case, 0)
        built = 4 * sum(r.length for r in runs) if kind == "oneshot" else 0
        return {"bytes": _sim_bytes(runs) + built, "flops": 0}
    if kind == "hierarchy":
        runs = _hierarchy(case, 0)[-1]
        return {"bytes": 4 * _sim_bytes(runs, analytic=True), "flops": 0}
    if kind == "variants":
        _, runs, pairs = _variant_items(case, 0)
        return {"bytes": _sim_bytes(runs, pairs), "flops": 0}
    if kind == "rates":
        chains = 4 * sum(r.length for r, tr in W.p512_plan() if tr is not None)
        return {"bytes": chains + 16 * POINTS * case["candidates"], "flops": 0}
    if kind == "infer":
        n = sum(r.length for r in _infer_runs())
        return {"bytes": 4 * n * (1 + case["observations"]) + 8 * 1308 * case["observations"], "flops": 0}
    if kind == "classify":
        lens = _classify_lengths(case)
        return {"bytes": sum(4 * n + 4 * ((n + 31) // 32) + 4 for n in lens), "flops": 0}
    if kind == "network":
        return {"bytes": case["traces"] * (4 * POINTS + 4 * LOGITS + 20) + 4 * n_par,
                "flops": 2 * macs * case["traces"]}
    if kind == "train":
        return {"bytes": case["batch"] * (4 * POINTS + 16) + 4 * n_par * 8,
                "flops": 6 * macs * case["batch"]}
    n, g = case["traces"], case["candidates"]
    return {"bytes": 4 * POINTS * (n + g) + 8 * n, "flops": 2 * POINTS * n * g}


# ------------------------------------------------------- the answers in 64 bits
def _gelu(z):
    return 0.5 * z * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (z + 0.044715 * z ** 3)))


def _unpacked(w):
    out, o = [], 0
    for r, c in _layers():
        out.append((w[o:o + r * c].view(r, c), w[o + r * c:o + r * c + r]))
        o += r * c + r
    return out


def _forward(w, x):
    """Logits in 64 bits: activations [B, position, channel], stride 2, zero
    padding of 2; column kk * cin + ci of a weight row is tap kk, channel ci."""
    L = _unpacked(w)
    h = x.unsqueeze(-1)
    for W_, b in L[:4]:
        B, n, cin = h.shape
        p = torch.nn.functional.pad(h, (0, 0, 2, 2))
        cols = torch.cat([p[:, k:k + n:2] for k in range(TAPS)], 2)
        h = _gelu(cols @ W_.t() + b)
    h = _gelu(h.reshape(h.shape[0], -1) @ L[4][0].t() + L[4][1])
    return h @ L[5][0].t() + L[5][1]


def exact(case, seed):
    kind = case["kind"]
    if kind == "classify":
        thr = []
        for lat in _classify_inputs(case, seed):
            v = lat.double().sort().values[:lat.numel() - lat.numel() // 200]
            gap = v[1:] - v[:-1]
            if gap.numel() == 0 or float(gap.max()) <= 0.0:
                thr.append(v[-1:])
            else:
                k = int(gap.argmax())
                thr.append(((v[k] + v[k + 1]) * 0.5).view(1))
        return [None, torch.cat(thr)]
    if kind == "network":
        w, x = _network_inputs(case, seed)
        w = w.double()
        lg = torch.cat([_forward(w, x[i:i + 2048].double()) for i in range(0, x.shape[0], 2048)])
        conf, o = torch.ones(lg.shape[0], dtype=torch.float64, device=DEV), 0
        for k in HEADS:
            conf = conf * torch.softmax(lg[:, o:o + k], 1).amax(1)
            o += k
        return {"pred": None, "conf": conf, "logits": lg}
    if kind == "train":
        w, m, v, x, lab = _train_inputs(case, seed)
        w, m, v = w.double().requires_grad_(True), m.double(), v.double()
        total, B = 0.0, x.shape[0]
        for i in range(0, B, 512):
            lg = _forward(w, x[i:i + 512].double())
            o, loss = 0, 0.0
            for h, k in enumerate(HEADS):
                loss = loss + torch.nn.functional.cross_entropy(
                    lg[:, o:o + k], lab[i:i + 512, h].long(), reduction="sum")
                o += k
            loss = loss / (4.0 * B)
            loss.backward()
            total += float(loss.detach())
        g = w.grad
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        c1, c2 = 1.0 - 0.9 ** (TRAIN_STEP + 1), 1.0 - 0.999 ** (TRAIN_STEP + 1)
        new = w.detach() - TRAIN_LR * (m / c1) / ((v / c2).sqrt() + 1e-8)
        return {"loss": torch.tensor([total], dtype=torch.float64), "grad": g, "w": new, "m": m, "v": v}
    if kind == "lsq":
        rates, y = _lsq_inputs(case, seed)
        R = rates.double()
        res = []
        for i in range(0, y.shape[0], 4096):
            t = y[i:i + 4096].double()
            keep = (t <= t.sort(1).values[:, POINTS - 6:POINTS - 5]).double()
            cnt = keep.sum(1, keepdim=True)
            sy, syy = (keep * t).sum(1, keepdim=True), (keep * t * t).sum(1, keepdim=True)
            var_y = syy - sy * sy / cnt
            r1, r2 = keep @ R.t(), keep @ (R * R).t()
            cov = (keep * t) @ R.t() - sy * r1 / cnt
            var_r = r2 - r1 * r1 / cnt
            fit = var_y - cov * cov / var_r.clamp(min=1e-12)
            best = torch.where((var_r > 1e-12) & (cov > 0.0), fit, var_y.expand_as(fit))
            res.append(best.clamp(min=0.0).amin(1))
        return [None, torch.cat(res)]
    return None
