"""Training tiles of 128 rows, two at a time per CTA, one CTA per SM:
gradients of batches around those sizes against the FP64 reference."""
import numpy as np
import pytest

from oracle import lod_ref as R
from tests.test_gpu_mlp import _batch, _cuda, _mlp, _params

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 8, 17, 127, 128, 129, 191, 192, 193, 255, 257, 385, 152 * 192 + 1, 152 * 256 + 1,
                               2 * 152 * 192 + 200, 152 * 512 + 129])
def test_gradient_of_batches_around_the_tile(n):
    m = _mlp()
    p = _params(11)
    m.set_params(p)
    feat, band, tgt = _batch(20 + n, n, bad_bands=True)
    loss = m.train_step(_cuda(feat), _cuda(band), _cuda(tgt), 1e-3)
    g = m.grad().astype(np.float64)
    L, gr = R.loss_and_grad(p.astype(np.float64), feat, band, tgt, rounding=True)
    # a BF16 step is 2^-8: 2e-2 leaves room for a few flipped roundings of a row
    assert abs(loss - L) <= 1e-4 * L + 1e-5 * np.sqrt(L)
    for a, b in ((0, 3072), (3072, 3136), (3136, 7232), (7232, 7296), (7296, 7360), (7360, 7361)):
        assert np.linalg.norm(g[a:b] - gr[a:b]) <= 2e-2 * max(np.linalg.norm(gr[a:b]), 1e-30)


@pytest.mark.parametrize("n", [5, 128, 1000, 152 * 256 + 130])
def test_features_at_an_odd_multiple_of_8_bytes(n):
    """The bulk copy needs 16-byte alignment, the array 8: same gradient."""
    import torch
    p = _params(12)
    feat, band, tgt = _batch(40 + n, n)
    buf = torch.zeros(n * 32 + 2, device="cuda")
    shifted = buf[2:].view(n, 32)
    shifted.copy_(_cuda(feat))
    out = []
    for f in (_cuda(feat), shifted):
        m = _mlp()
        m.set_params(p)
        loss = m.train_step(f, _cuda(band), _cuda(tgt), 1e-3)
        out.append((loss, m.grad()))
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])
