"""A plan whose launches fan out (played sets, segments, jumbo and pool units)
captured into CUDA graphs while it also runs outside of the capture and in a
second one: workspaces and streams of their own, one plan."""
import ctypes
import glob
import os

import numpy as np
import pytest

import oracle
from paper_1509_02308_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1509_02308_gb300 import api
    from paper_1509_02308_gb300 import capi as C

# played sets: in segments, in windows, in the larger tables; units of the slot
# mix, of the one-warp launch, with their state in global memory
FORMS = [(W.Geom(4 * 32, 32, 4, 1, W.RANDOM, 5), W.Run(48, 8, 100003, 6)),
         (W.Geom(40 * 32, 32, 40, 1, W.RANDOM, 6), W.Run(800, 8, 9001, 100)),
         (W.Geom(1000 * 32, 32, 1000, 1, W.RANDOM, 6), W.Run(1400 * 8, 8, 9001, 1400)),
         (W.Geom(2048, 32, 8, 8, W.FIFO, 8), W.Run(1000, 7, 5000, 10)),
         (W.Geom(4 * 20000, 4, 4, 5000, W.RANDOM, 8), W.Run(30001, 7, 4000, 10)),
         (W.Geom(128 << 20, 128, 16, 65536, W.LRU, 9), W.Run(40000001, 33, 3000, 10))]


def _runtime():
    """The CUDA runtime that this process has loaded already."""
    paths = [l.split()[-1] for l in open("/proc/self/maps") if "libcudart.so" in l]
    paths += glob.glob("/usr/local/cuda/lib64/libcudart.so*")
    assert paths
    return ctypes.CDLL(os.path.realpath(paths[0]))


class _Graph:
    """A capture on a stream of its own, apart from torch's."""

    def __init__(self, rt):
        self.rt, self.stream = rt, torch.cuda.Stream()
        self.graph, self.exec, self.open = ctypes.c_void_p(), ctypes.c_void_p(), True
        self._ok(rt.cudaStreamBeginCapture(self._st(), 2))  # cudaStreamCaptureModeRelaxed

    def _st(self):
        return ctypes.c_void_p(self.stream.cuda_stream)

    def _ok(self, rc):
        assert rc == 0, rc

    def end(self):
        self.open = False
        self._ok(self.rt.cudaStreamEndCapture(self._st(), ctypes.byref(self.graph)))
        self._ok(self.rt.cudaGraphInstantiateWithFlags(ctypes.byref(self.exec), self.graph,
                                                       ctypes.c_ulonglong(0)))

    def kernels(self):
        n = ctypes.c_size_t(0)
        self._ok(self.rt.cudaGraphGetNodes(self.graph, None, ctypes.byref(n)))
        nodes = (ctypes.c_void_p * n.value)()
        self._ok(self.rt.cudaGraphGetNodes(self.graph, nodes, ctypes.byref(n)))
        count = 0
        for v in nodes:
            t = ctypes.c_int(-1)
            self._ok(self.rt.cudaGraphNodeGetType(ctypes.c_void_p(v), ctypes.byref(t)))
            count += t.value == 0  # cudaGraphNodeTypeKernel
        return count

    def launch(self):
        self._ok(self.rt.cudaGraphLaunch(self.exec, self._st()))
        self.stream.synchronize()

    def close(self):
        if self.open:  # (a failed test leaves no capture behind)
            self.rt.cudaStreamEndCapture(self._st(), ctypes.byref(self.graph))
        if self.exec:
            self.rt.cudaGraphExecDestroy(self.exec)
        if self.graph:
            self.rt.cudaGraphDestroy(self.graph)


class _Place:
    """A workspace and outputs of a plan's run."""

    def __init__(self, plan):
        self.plan = plan
        self.ws = torch.empty(plan.ws_bytes + 256, dtype=torch.uint8, device="cuda")
        self.at = (self.ws.data_ptr() + 255) & ~255
        self.bits = torch.zeros(plan.bitmap_words, dtype=torch.int32, device="cuda")
        self.counts = torch.zeros(2 * plan.n_items, dtype=torch.int64, device="cuda")
        C.check(plan.L.pchase_sim_plan_upload(plan.h, self.at, plan.ws_bytes, C.stream_handle()))

    def run(self, stream):
        C.check(self.plan.L.pchase_sim_run(self.plan.h, self.at, C.ptr(self.bits), None,
                                           C.ptr(self.counts), None, C.stream_handle(stream)))

    def take(self):
        torch.cuda.synchronize()
        out = self.bits.cpu().numpy().view(np.uint32).copy(), self.counts.cpu().numpy().copy()
        self.bits.zero_()
        self.counts.zero_()
        torch.cuda.synchronize()
        return out


def _plan(explicit):
    runs = [r for _, r in FORMS]
    flat, offs = api.pchase_build_batch(runs)
    traces = [(flat[int(offs[i]):int(offs[i + 1])] if explicit else None, r.length, r.warmup, r.n_elems,
               r.stride) for i, r in enumerate(runs)]
    plan = api.SimPlan([g for g, _ in FORMS], traces, pairs=[(i, i) for i in range(len(runs))])
    plan._flat = flat
    return plan


@pytest.mark.parametrize("first_captured", [False, True])
@pytest.mark.parametrize("explicit", [False, True])
def test_a_plan_runs_while_it_is_captured_twice(explicit, first_captured):
    rt = _runtime()
    plan = _plan(explicit)
    d = dict(kv.split("=", 1) for kv in plan.description.split())
    assert int(d["jumbo"]) >= 1 and int(d["global_state"]) >= 1, plan.description
    assert int(d["uniform"].split(",")[1]) >= 2 and int(d["uniform"].split(",")[2]) >= 1, plan.description
    places = [_Place(plan) for _ in range(3)]
    torch.cuda.synchronize()
    if not first_captured:  # the plan has its own streams by then
        places[0].run(torch.cuda.current_stream())
        places[0].take()
    other, graphs = torch.cuda.Stream(), []
    try:
        graphs.append(_Graph(rt))
        places[0].run(graphs[0].stream)
        places[2].run(other)  # beside the capture
        graphs.append(_Graph(rt))
        places[1].run(graphs[1].stream)
        places[2].run(other)
        graphs[0].end()
        places[2].run(other)
        graphs[1].end()
        assert [g.kernels() for g in graphs] == [plan.launches] * 2
        want = places[2].take()
        for i, (g, r) in enumerate(FORMS):
            miss = oracle.cache_sim(g.C, g.b, g.ways, g.sets, g.policy,
                                    oracle.pchase_trace(r.n_elems, r.stride, r.length), seed=g.seed)
            assert np.array_equal(api.unpack_bits(want[0][int(plan.word_offsets[i]):], r.length), miss), i
        for _ in range(2):
            for g in graphs:
                g.launch()
            for p in places[:2]:
                got = p.take()
                assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    finally:
        for g in graphs:
            g.close()


@pytest.mark.parametrize("n_geom", [3, 16])
def test_a_match_launches_no_segments(n_geom):
    """Sets long enough for segments are in items that the matcher leaves to the
    units: a match queues the check, the words (of groups too, from 16
    candidates on), the played sets and the units, and nothing for segments."""
    runs = [W.Run(48, 8, 100003, 6), W.Run(800, 8, 9001, 100)]
    traces = [(None, r.length, r.warmup, r.n_elems, r.stride) for r in runs]
    cands = [W.Geom(4 * 32 * (1 + k % 4), 32, 4 * (1 + k % 4), 1, (W.RANDOM, W.LRU, W.FIFO)[k % 3], 5 + k)
             for k in range(n_geom)]
    rng = np.random.Generator(np.random.PCG64(n_geom))
    words = [(r.length + 31) // 32 for r in runs]
    obs = torch.from_numpy(rng.integers(-2**31, 2**31, sum(words)).astype(np.int32)).cuda()
    owo = torch.tensor([0, words[0]], dtype=torch.int64, device="cuda")
    plan = api.SimPlan(cands, traces)
    assert int(plan.description.split("uniform=")[1].split()[0].split(",")[2]) >= 1, plan.description
    dist = torch.zeros(n_geom, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    g = _Graph(_runtime())
    try:
        C.check(plan.L.pchase_match_run(plan.h, plan._ws, C.ptr(obs), C.ptr(owo), 2**64 - 1, C.ptr(dist),
                                        None, C.stream_handle(g.stream)))
        g.end()
        assert g.kernels() == 4 + (n_geom >= 16)
        g.launch()
    finally:
        g.close()
    want = api.SimPlan(cands, traces, tune={"head_streams": 2}).match(obs, owo)
    assert torch.equal(dist, want) and torch.equal(plan.match(obs, owo), want)
