"""The least-squares judge (lsq.cu) against float64 where its estimates are at
their weakest and where its CTAs take several tiles.  Bounds as in
test_gpu_lsq.py: the error of FP32 sums of 512 terms, to first order, doubled."""
import numpy as np
import pytest

from oracle import inverse_ref as R
from test_gpu_lsq import _exact, _rows

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1509_02308_gb300 import inverse as INV


def _check(rates, y):
    best, res = INV.lsq_match(torch.from_numpy(rates).cuda(), torch.from_numpy(y).cuda())
    best, res = best.cpu().numpy(), res.cpu().numpy().astype(np.float64)
    assert best.min() >= 0 and best.max() < len(rates)
    for k in range(0, len(y), 1024):
        want, bound = _exact(rates, y[k:k + 1024])
        i = np.arange(len(want))
        assert (np.abs(res[k:k + 1024] - want[i, best[k:k + 1024]]) <= bound[i, best[k:k + 1024]]).all()
        assert (res[k:k + 1024] <= (want + bound).min(1)).all()
    # of equal rows the first answers
    first = {r.tobytes(): k for k, r in reversed(list(enumerate(rates)))}
    assert all(first[rates[b].tobytes()] == b for b in best)
    return best


@pytest.mark.parametrize("amp", [1e-1, 1e-2, 1e-3, 3e-4])
@pytest.mark.parametrize("base", [0.0, 0.25])
def test_judge_by_five_high_points_over_a_small_ramp(amp, base):
    """Rows of five high points over a ramp that is small against them: the
    traces' five dropped points are the high ones, so what is left of a row is
    a difference of nearly equal sums.  Traces that are such rows, and a
    competitor within 0.5 % of the variance for each."""
    rng = np.random.Generator(np.random.PCG64(int(1e6 * amp) + int(8 * base)))
    rows, y = [], []
    for _ in range(60):
        ramp = amp * rng.permutation(np.linspace(0.0, 1.0, R.POINTS))
        high = rng.choice(R.POINTS, 5, replace=False)
        few = base + ramp
        few[high] = rng.uniform(0.5, 1.0, 5) + base
        close = base + ramp + 0.07 * np.sqrt(np.var(ramp)) * rng.standard_normal(R.POINTS)
        close[high] = base + amp * rng.random(5)
        rows += [few, 0.5 / amp * (close - base)]
        y.append(few)
    rates, y = np.array(rows).astype(np.float32), np.array(y).astype(np.float32)
    best = _check(rates, y)
    if base == 0.0:  # (sums over rows far above their ramp decide nothing)
        assert (best == 2 * np.arange(60)).all()

# candidates per tile (on 152 SMs): 96, 128, 160, 224 and 256 in one wave, then
# two and three tiles to a CTA, with a second chunk of one candidate
@pytest.mark.parametrize("n,G", [(1000, 1308), (1500, 1308), (2047, 1307), (3000, 1308), (5000, 700),
                                 (2600, 1999), (4097, 1308), (4097, 2049), (8191, 1308)])
def test_judge_over_many_tiles(n, G):
    rng = np.random.Generator(np.random.PCG64(1000 * n + G))
    rates = _rows(G, rng)
    y = rates[rng.integers(0, G, n)] + 0.02 * rng.standard_normal((n, R.POINTS))
    y[rng.random(y.shape) < 0.005] *= 4.0
    _check(rates, y.astype(np.float32))
