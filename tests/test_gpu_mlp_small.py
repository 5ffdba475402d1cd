"""Training batches around one tile of 128 rows per SM and two: one group or
both at work in a CTA, partial sums of one CTA or many."""
import numpy as np
import pytest

from oracle import lod_ref as R
from tests.test_gpu_mlp import _batch, _cuda, _mlp, _params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles, rows", [(1, 0), (2, -1), (2, 1), ("sms", -1), ("sms", 0), ("sms", 1), ("sms", 129),
                                         ("2 sms", -127), ("2 sms", 0), ("2 sms", 1), ("4 sms", 1)])
def test_gradient_of_batches_around_the_grid(tiles, rows):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 128 * {"sms": sms, "2 sms": 2 * sms, "4 sms": 4 * sms}.get(tiles, tiles) + rows
    m = _mlp()
    p = _params(13)
    m.set_params(p)
    feat, band, tgt = _batch(60 + n, n, bad_bands=True)
    loss = m.train_step(_cuda(feat), _cuda(band), _cuda(tgt), 1e-3)
    g = m.grad().astype(np.float64)
    L, gr = R.loss_and_grad(p.astype(np.float64), feat, band, tgt, rounding=True)
    # a BF16 step is 2^-8: 2e-2 leaves room for a few flipped roundings of a row
    assert abs(loss - L) <= 1e-4 * L + 1e-5 * np.sqrt(L)
    for a, b in ((0, 3072), (3072, 3136), (3136, 7232), (7232, 7296), (7296, 7360), (7360, 7361)):
        assert np.linalg.norm(g[a:b] - gr[a:b]) <= 2e-2 * max(np.linalg.norm(gr[a:b]), 1e-30)
    m.close()
