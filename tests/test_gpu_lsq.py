"""The least-squares judge (lsq.cu) against float64 at the edges of its tiles
(128 traces x 128 candidates, chunks of 2048 candidates) and where its
estimates decide nothing: equal rows, constant and nearly constant rows, traces
far from zero.  Bound: the FP32 sums of 512 terms in point order err by at most
g = 512 2^-24 of the sums of their terms' magnitudes, and the residual
Var_y - Cov^2 / Var_r moves by dVar_y + 2 b dCov + b^2 dVar_r (b the slope) to
first order, doubled for what comes after."""
import numpy as np
import pytest

from oracle import inverse_ref as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1509_02308_gb300 import inverse as INV


def _rows(n, rng):
    """Step-like rows, each second one given twice, some constant or nearly so."""
    p = np.arange(R.POINTS)
    rows = []
    for k in range(n):
        knee, top = rng.integers(20, 500), rng.choice([0.125, 0.25, 0.5, 1.0])
        ramp = np.clip((p - knee) / rng.integers(1, 60), 0, 1) * top
        rows.append(np.round(ramp * 4096) / 4096)
    rows = np.array(rows)
    if n > 8:
        rows[n // 2] = rows[n // 3]
        rows[n - 1] = 0.75          # constant
        rows[n - 2] = 1.0
        rows[n - 2, 5] = 1.0 - 2.0 ** -10  # one point away from constant
        rows[n - 3] = 0.0
    return rows.astype(np.float32)


def _exact(rates, y):
    """Residuals and their bounds [n, G] in float64."""
    r, y = rates.astype(np.float64), y.astype(np.float64)
    thr = np.sort(y, 1)[:, R.KEEP - 1:R.KEEP]
    m = (y <= thr).astype(np.float64)
    cnt, sy, syy = m.sum(1, keepdims=True), (m * y).sum(1, keepdims=True), (m * y * y).sum(1, keepdims=True)
    dyr, dr, drr = (m * y) @ r.T, m @ r.T, m @ (r * r).T
    mag = (m * np.abs(y)) @ np.abs(r).T
    var_y, cov, var_r = syy - sy * sy / cnt, dyr - sy * dr / cnt, drr - dr * dr / cnt
    g = R.POINTS * 2.0 ** -24
    asy = (m * np.abs(y)).sum(1, keepdims=True)
    d_cov, d_var = g * (mag + 3 * asy * dr / cnt), g * (drr + 3 * dr * dr / cnt)
    d_vy = g * (syy + 3 * asy * asy / cnt)
    fits = (var_r > 2 * d_var + 1e-12) & (cov > d_cov)
    b = np.where(fits, cov / np.where(fits, var_r, 1.0), 0.0)
    res = np.maximum(var_y - b * b * var_r, 0.0)
    bound = 2 * (d_vy + 2 * b * d_cov + b * b * d_var)
    # where a sum's error decides between the fit and the plain variance, or
    # the variance is within its error, any value up to the variance may come
    near = (~fits) & (np.abs(cov) > 0) & (var_r + d_var > 1e-12) & (cov > -d_cov)
    return res, np.where(near, var_y + bound, bound)


@pytest.mark.parametrize("n,G", [(1, 1), (2, 2), (37, 127), (127, 128), (128, 129), (129, 300),
                                 (300, 2049), (257, 1308)])
@pytest.mark.parametrize("shift", [0.0, 30.0])
def test_judge_at_tile_edges(n, G, shift):
    rng = np.random.Generator(np.random.PCG64(1000 * n + G))
    rates = _rows(G, rng)
    truth = rng.integers(0, G, n)
    y = rates[truth] + 0.02 * rng.standard_normal((n, R.POINTS)) + shift
    y[rng.random(y.shape) < 0.005] *= 4.0
    y = y.astype(np.float32)
    best, res = INV.lsq_match(torch.from_numpy(rates).cuda(), torch.from_numpy(y).cuda())
    best, res = best.cpu().numpy(), res.cpu().numpy().astype(np.float64)
    assert best.min() >= 0 and best.max() < G
    want, bound = _exact(rates, y)
    i = np.arange(n)
    assert (np.abs(res - want[i, best]) <= bound[i, best]).all()
    assert (res <= (want + bound).min(1)).all()
    # of equal rows the first answers
    first = {r.tobytes(): k for k, r in reversed(list(enumerate(rates)))}
    assert all(first[rates[b].tobytes()] == b for b in best)
    # unaligned rates (rows on 4-byte boundaries) give the same answers
    buf = torch.zeros(rates.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(rates.reshape(-1)).cuda()
    b2, r2 = INV.lsq_match(buf[1:].view(G, R.POINTS), torch.from_numpy(y).cuda())
    assert np.array_equal(b2.cpu().numpy(), best) and np.array_equal(r2.cpu().numpy().astype(np.float64), res)


@pytest.mark.parametrize("n,G", [(3, 33), (16, 200), (130, 161), (40, 2100)])
def test_judge_by_few_points(n, G):
    """Rows that a trace's five dropped points can take most or all of (their
    residuals' lower bounds say nothing), and traces that fit so many rows
    equally well that their list overflows, between traces that do not."""
    rng = np.random.Generator(np.random.PCG64(77 * n + G))
    rates = _rows(G, rng)
    for k in range(0, G, 2):
        rates[k] = 0.0
        rates[k, rng.integers(0, R.POINTS, 1 + k // 2 % 12)] = rng.choice([0.25, 0.5, 1.0])
    y = rates[rng.integers(0, G, n)] + 0.02 * rng.standard_normal((n, R.POINTS))
    y[1::3] = rng.standard_normal((len(y[1::3]), R.POINTS)) + 500.0
    y = y.astype(np.float32)
    best, res = INV.lsq_match(torch.from_numpy(rates).cuda(), torch.from_numpy(y).cuda())
    best, res = best.cpu().numpy(), res.cpu().numpy().astype(np.float64)
    assert best.min() >= 0 and best.max() < G
    want, bound = _exact(rates, y)
    i = np.arange(n)
    assert (np.abs(res - want[i, best]) <= bound[i, best]).all()
    assert (res <= (want + bound).min(1)).all()
