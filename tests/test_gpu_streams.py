"""Calls on a stream that has work queued, not the current one: the memory of
their temporaries is not given out again while they wait."""
import types

import numpy as np
import pytest

from paper_1509_02308_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1509_02308_gb300 import api


def _scribble(nbytes):
    """Fills what the current stream's pool gives out for the sizes up to nbytes."""
    keep = []
    for n in [1 << k for k in range(9, nbytes.bit_length() + 1)]:
        for _ in range(4):
            keep.append(torch.full((n,), 0x7E, dtype=torch.uint8, device="cuda"))
    torch.cuda.current_stream().synchronize()


@pytest.mark.parametrize("handle_only", [False, True])
def test_classify_and_infer_on_a_busy_stream(handle_only):
    rng = np.random.Generator(np.random.PCG64(3))
    lats = [torch.from_numpy(rng.choice([100.0, 400.0], n).astype(np.float32)).cuda()
            for n in (70000, 33, 1, 20001)]
    bits, words, thr = api.pchase_classify(lats)
    runs = [W.Run(n // 4, 8, 2 * (n // 32), n // 32) for n in (4096, 8192, 12320)]
    traces = [(None, r.length, r.warmup, r.n_elems, r.stride) for r in runs]
    plan = api.SimPlan([W.Geom(8192, 32, 4, 64, p, 3) for p in (0, 1, 2)], traces)
    obs = torch.from_numpy(rng.choice([100.0, 400.0], (5, sum(r.length for r in runs))).astype(np.float32)).cuda()
    want = api.infer_batch(plan, obs) + plan.infer(obs[0])
    stream = torch.cuda.Stream()
    arg = types.SimpleNamespace(cuda_stream=stream.cuda_stream) if handle_only else stream
    _scribble(1 << 22)  # (the pool has the blocks by then)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        torch.cuda._sleep(1_000_000_000)  # half a second
    got_bits, _, got_thr = api.pchase_classify(lats, stream=arg)
    _scribble(1 << 22)
    got = api.infer_batch(plan, obs, stream=arg) + plan.infer(obs[0], stream=arg)
    _scribble(1 << 22)
    assert not stream.query()  # (the calls were still waiting)
    torch.cuda.synchronize()
    assert torch.equal(got_thr, thr) and len(words) == 4
    used = sum((x.numel() + 31) // 32 for x in lats)
    assert torch.equal(got_bits[:used], bits[:used])
    for a, b in zip(got, want):
        assert torch.equal(a, b)
