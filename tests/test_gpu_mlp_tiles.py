"""Training tiles of 192 rows, 16 to a warp, one CTA per SM: gradients of
batches around those sizes against the FP64 reference."""
import numpy as np
import pytest

from oracle import lod_ref as R
from tests.test_gpu_mlp import _batch, _cuda, _mlp, _params

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 8, 17, 191, 192, 193, 385, 152 * 192 + 1, 2 * 152 * 192 + 200])
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
