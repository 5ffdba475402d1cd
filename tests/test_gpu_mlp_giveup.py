"""A training step whose tensor-core products are never reported complete
gives up after its bounded waits: every way to learn of it, and what stays."""
import numpy as np
import pytest

from tests.test_gpu_mlp import _batch, _cuda, _mlp, _params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, shift", [(100, 0), (128 * 700 + 5, 0), (300, 2)])
@pytest.mark.parametrize("first", ["step", "grad", "params", "loss"])
def test_a_step_that_gave_up_is_reported_and_changes_nothing(n, shift, first):
    from paper_2501_17792_gb300 import binding
    if first != "step" and n > 1000:
        pytest.skip("one size is enough")
    m = _mlp()
    p = _params(3)
    m.set_params(p)
    feat, band, tgt = _batch(50 + n, n)
    buf = torch.zeros(n * 32 + shift, device="cuda")  # (features off the 16-byte grid: no bulk copy)
    f = buf[shift:].view(n, 32)
    f.copy_(_cuda(feat))
    batch = (f, _cuda(band), _cuda(tgt))
    want_loss = m.train_step(*batch, 1e-3)
    want_grad, after = m.grad(), m.params()
    m.set_params(p)
    assert m.L.cs_debug_mlp_lose_product(m.h, 1) == binding.CS_OK
    if first == "loss":
        with pytest.raises(binding.CrowdSplatError, match="gave up") as e:
            m.train_step(*batch, 1e-3)
        assert e.value.code == binding.CS_ERR_CUDA
    else:
        m.train_step(*batch, 1e-3, want_loss=False)  # not waited for
        torch.cuda.synchronize()
        with pytest.raises(binding.CrowdSplatError, match="gave up"):
            dict(step=lambda: m.train_step(*batch, 1e-3, want_loss=False), grad=m.grad, params=m.params)[first]()
    # from here on by all, also with nothing lost any more
    m.L.cs_debug_mlp_lose_product(m.h, 0)
    for call in (m.grad, m.params, lambda: m.train_step(*batch, 1e-3), lambda: m.train_step(*batch, 1e-3, want_loss=False)):
        with pytest.raises(binding.CrowdSplatError, match="gave up"):
            call()
    got = np.empty(binding.MLP_PARAMS, np.float32)
    assert m.L.cs_mlp_get_params(m.h, got.ctypes.data) == binding.CS_ERR_CUDA
    assert np.array_equal(got, p)
    # setting the parameters starts again: the same step as before
    m.set_params(p)
    assert m.train_step(*batch, 1e-3) == want_loss
    assert np.array_equal(m.grad(), want_grad) and np.array_equal(m.params(), after)
    m.close()
