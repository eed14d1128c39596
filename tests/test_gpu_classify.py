"""Classification (classify.cu) against the oracle's sort: sizes around a
cluster's slices and its limits, and values for which the coarse buckets do not
settle the largest gap."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1509_02308_gb300 import api


def _values(kind, n, rng):
    if kind == "plateaus":
        v = np.where(rng.random(n) < 0.3, 400.0, 100.0) * (1 + 0.02 * rng.standard_normal(n))
        v[rng.random(n) < 0.003] *= 8.0
    elif kind == "smooth":      # no gap wider than a coarse bucket
        v = rng.random(n) * 300.0
    elif kind == "ladder":      # equal gaps: the lowest one counts
        v = 100.0 + 0.5 * rng.integers(0, 3000, n)
    elif kind == "same":
        v = np.full(n, 37.0)
    elif kind == "tiny":        # buckets narrower than the smallest normal number
        v = rng.integers(0, 50, n) * 1e-42
    elif kind == "wide":        # a range that overflows
        v = np.where(rng.random(n) < 0.5, -3e38, 3e38)
    elif kind == "signed":
        v = rng.standard_normal(n) * 10.0
        v[rng.random(n) < 0.2] += 90.0
        v[: n // 50] = -0.0
    else:                       # infinite values among the kept ones
        v = np.where(rng.random(n) < 0.2, np.inf, 100.0 + rng.random(n))
    return v.astype(np.float32)


SIZES = (1, 2, 31, 33, 199, 200, 1000, 8191, 8192, 8193, 16385, 32769, 65537, 131071)


@pytest.mark.parametrize("kind", ["plateaus", "smooth", "ladder", "same", "signed"])
@pytest.mark.parametrize("sizes", [SIZES[:7], SIZES[7:10], SIZES[10:], (393000,), (500000,)])
def test_classify_matches_oracle(kind, sizes):
    if sizes[0] > 390000 and kind in ("ladder", "same"):
        sizes = (sizes[0] // 4,)
    rng = np.random.Generator(np.random.PCG64(len(kind) + sizes[0]))
    obs = [_values(kind, n, rng) for n in sizes]
    bits, w, thr = api.pchase_classify([torch.from_numpy(v).cuda() for v in obs])
    bits, thr = bits.cpu().numpy().view(np.uint32), thr.cpu().numpy()
    for i, v in enumerate(obs):
        want, cut = oracle.classify(v)
        assert np.float32(cut) == thr[i], (kind, v.size, cut, thr[i])
        assert np.array_equal(api.unpack_bits(bits[int(w[i]):], v.size), want), (kind, v.size)


@pytest.mark.parametrize("kind", ["tiny", "wide", "inf"])
def test_irregular_values_agree_with_long_observations(kind):
    """Where the bucket arithmetic over- or underflows the answer is what the
    buckets give; the one-launch path gives the same as the launches over
    global memory (observations too long for a cluster), here the same values
    padded with equal ones at the bottom."""
    rng = np.random.Generator(np.random.PCG64(3))
    v = _values(kind, 3000, rng)
    low = v.min()
    short = np.concatenate([np.full(2000, low, np.float32), v])
    bits, _, thr = api.pchase_classify([torch.from_numpy(short).cuda()])
    again, _, thr2 = api.pchase_classify([torch.from_numpy(short).cuda(), torch.from_numpy(
        np.full(400000, 1.0, np.float32)).cuda()])
    assert np.array_equal(thr.cpu().numpy()[:1], thr2.cpu().numpy()[:1], equal_nan=True)
    words = (short.size + 31) // 32
    assert torch.equal(bits[:words], again[:words])
