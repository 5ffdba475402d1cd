"""Statistics and training frames composite each 8x4 pixel block with one
walking warp, in batches of 32 pairs, training lists past 8,192 pairs in
parallel chunks.  Lists around those sizes, in images that cut tiles and
blocks, against the plain frame of the same scene and against each other."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C0 = 0.28209479177387814


def _scene(n, w, h, seed=3, f=30.0):
    """n faint Gaussians (opacity 0.006 to 0.016, grey) over a w x h view:
    with these a pixel takes about a thousand before it saturates."""
    from tests import scene_util as U
    rng = np.random.default_rng(seed)
    z = rng.uniform(2.0, 5.0, n)
    px, py = rng.uniform(0, w, n), rng.uniform(0, h, n)
    means = np.stack([(px - w / 2) * z / f, (py - h / 2) * z / f, z], 1)
    scales = (1.2 * z / f)[:, None] * np.exp(rng.normal(0, 0.3, (n, 3)))
    tpl = U.template_from(means, scales, rng.standard_normal((n, 4)), rng.uniform(0.006, 0.016, n),
                          np.zeros((n, 1, 3)))
    return U.scene_of([tpl], U.instances(1), U.identity_camera(w, h, f))


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1024, 1025, 8192, 8193, 20001])
@pytest.mark.parametrize("w, h", [(16, 16), (13, 19)])
def test_statistics_and_training_lists_against_plain_frames(n, w, h):
    from paper_2501_17792_gb300 import binding
    sc = _scene(n, w, h)
    r = binding.Renderer(device=0)
    r.upload_templates(sc.templates)
    r.set_instances(sc.instances.template_id, sc.instances.root, sc.instances.pose)
    plain = r.render(sc.camera)
    contrib = torch.zeros(n, device="cuda")
    stat = r.render_contrib(sc.camera, contrib)
    train = r.render_train(sc.camera)
    # Both T and the colour sums are products and sums of at most about a
    # thousand factors, each rounded to 6e-8: 6e-5 relative; a stop decided the
    # other way changes a pixel by at most 0.016 x 1e-4.
    for img in (stat, train):
        assert float((img - plain).abs().max()) <= 2e-4
    # every weight went to one Gaussian: the sums add up to the alpha channel
    total = float(stat[..., 3].double().sum())
    assert abs(float(contrib.double().sum()) - total) <= 1e-4 * max(total, 1e-3)
    # colour is linear in the degree-0 coefficient (grey 0.5, no clamp): the
    # gradient of the summed red channel is C0 times the Gaussian's weight;
    # the backward recovers T by divisions, 1e-4 relative over a thousand
    dl = torch.zeros((h, w, 4), device="cuda")
    dl[..., 0] = 1.0
    g = r.backward(dl, 1)
    assert torch.allclose(g["sh"][:, 0, 0], C0 * contrib, rtol=5e-4, atol=5e-4 * float(C0 * contrib.max()))
    assert float(g["sh"][:, 1:].abs().max()) == 0.0 and float(g["sh"][:, 0, 1:].abs().max()) == 0.0
    r.close()


@pytest.mark.parametrize("sh_degree", [0, 1, 2, 3])
def test_gradients_into_an_sh_array_off_the_16_byte_grid(sh_degree):
    """The SH gradients go out as 16-byte reductions where the caller's array
    allows; an array that starts on any float gets the same values."""
    import ctypes as C
    from paper_2501_17792_gb300 import binding
    from paper_2501_17792_gb300 import scene as S
    sc = S.single_avatar(n_gauss=700, size=48, sh_degree=sh_degree)
    r = binding.Renderer(device=0)
    r.upload_templates(sc.templates)
    r.set_instances(sc.instances.template_id, sc.instances.root, sc.instances.pose)
    r.render_train(sc.camera)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    dl = torch.randn((48, 48, 4), generator=g, device="cuda")
    want = r.backward(dl, 1)["sh"].reshape(-1)
    buf = torch.zeros(700 * 48 + 2, device="cuda")
    grads = binding.Grads(None, None, None, None, buf[1:].data_ptr(), None)
    assert r.L.cs_backward(r.h, dl.data_ptr(), C.byref(grads)) == binding.CS_OK
    torch.cuda.synchronize()
    # the pixels' sums reach a coefficient in any order
    assert torch.allclose(buf[1:-1], want, rtol=1e-4, atol=1e-5 * float(want.abs().max()))
    assert float(buf[0]) == 0.0 and float(buf[-1]) == 0.0 and float(want.abs().max()) > 0.0
    r.close()


def test_counts_of_a_new_context_after_contexts_of_one_frame():
    """The host polls a frame's counts in pinned memory that an earlier
    context may have used: contexts that render one frame of different sizes
    and go, then one of the first size again, all equal to a context that
    stays."""
    from paper_2501_17792_gb300 import binding
    from paper_2501_17792_gb300 import scene as S
    small, large = (S.crowd(n_templates=1, n_gauss=n, sh_degree=0, cols=c, rows=4, width=96, height=64)
                    for n, c in ((300, 3), (5000, 6)))
    for on_device in (False, True):
        want = {}
        for k in range(6):
            sc = (small, large)[k % 2]
            r = binding.Renderer(device=0)
            r.upload_templates(sc.templates)
            r.set_lod(sc.lod)
            inst = [sc.instances.template_id, sc.instances.root, sc.instances.pose]
            r.set_instances(*([torch.from_numpy(a).cuda() for a in inst] if on_device else inst))
            img = r.render(sc.camera).clone()
            r.close()
            assert torch.equal(img, want.setdefault(k % 2, img))
            assert float(img[..., 3].max()) > 0.5
