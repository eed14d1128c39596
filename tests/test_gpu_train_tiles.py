"""A training step of so many traces that every CTA of the convolutions takes
several tiles (on 152 SMs: layer 2 twelve, layer 3 six, layer 4 three) and
conv0_back six traces, with ragged ends: buffers that a tile's outputs leave
from are filled again by the next one's."""
import numpy as np
import pytest

from oracle import inverse_ref as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1509_02308_gb300 import inverse as INV


def test_gradient_over_many_tiles_matches_oracle_element_by_element():
    """The bound is that of the small batches: operands agree up to one BF16
    rounding each, so an element lies within 2^-7 of the sum of its terms'
    magnitudes; the loss within 2^-12."""
    B = 1835
    net = INV.LearnedInverse(max_batch=B)
    net.init(seed=77)
    rng = np.random.Generator(np.random.PCG64(B))
    w0 = net.weights().cpu().numpy().astype(np.float64)
    x = rng.random((B, R.POINTS)).astype(np.float32)
    lab = np.stack([rng.integers(0, k, B) for k in (17, 4, 7, 3)], axis=1).astype(np.int32)
    dx, dl = torch.from_numpy(x).cuda(), torch.from_numpy(lab).cuda()
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    INV._check(net.L.pchase_inverse_train_step(net.h, net._p, net._w, dx.data_ptr(), dl.data_ptr(), B,
                                               1e-3, 0, loss.data_ptr(), None))
    torch.cuda.synchronize()
    assert net.status() == 0
    g = net.param_array(2).cpu().numpy().astype(np.float64)
    cache = R.forward_cache(w0, x)
    want, mag = R.backward(cache, lab.astype(np.int64))
    want_loss = R.xent(cache["logits"], lab.astype(np.int64))
    assert abs(float(loss.item()) - want_loss) <= 2.0 ** -12 * want_loss
    bad = np.abs(g - want) > 2.0 ** -7 * mag + 1e-12
    offs = np.cumsum([0] + [r * c + r for r, c in R.layer_shapes()])
    assert not bad.any(), [int(bad[offs[l]:offs[l + 1]].sum()) for l in range(6)]
