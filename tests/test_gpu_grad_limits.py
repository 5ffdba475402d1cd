"""Gradients at the limits of their index ranges and of their values: frames
of more than 2^32 / 12 splats, and values that are not finite, which spoil
what they belong to and nothing else."""
import math

import numpy as np
import pytest

from tests import scene_util as U

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _renderer(sc, **kw):
    from paper_2501_17792_gb300 import binding
    r = binding.Renderer(device=0, **kw)
    r.upload_templates(sc.templates)
    r.set_instances(sc.instances.template_id, sc.instances.root, sc.instances.pose)
    return r


def test_gradients_of_splats_past_two_to_the_32_sums():
    """Twelve floats of sums a splat: from splat 2^32 / 12 on their address
    needs more than 32 bits.  A frame of 357.9 million splats, all behind the
    camera but the last two instances', has the gradients of a frame of those
    two."""
    n, seen = 4096, 2
    hidden = 2 ** 32 // 12 // n + 2
    # 120 bytes a splat and a quarter more, and what the caller holds
    if torch.cuda.mem_get_info()[0] < 70 << 30:
        pytest.skip("needs 70 GB of device memory")
    rng = np.random.default_rng(5)
    tpl = U.template_from(rng.uniform(-0.3, 0.3, (n, 3)), rng.uniform(0.01, 0.03, (n, 3)), rng.standard_normal((n, 4)),
                          rng.uniform(0.1, 0.9, n), 0.3 * rng.standard_normal((n, 1, 3)))
    front = np.tile(np.eye(3, 4, dtype=np.float32), (seen, 1, 1))
    front[:, :, 3] = [[-0.3, 0.0, 2.5], [0.3, 0.1, 2.6]]
    back = np.tile(np.eye(3, 4, dtype=np.float32), (hidden, 1, 1))
    back[:, 2, 3] = -5.0
    cam = U.identity_camera(64, 48, 60.0)
    dl = torch.randn((48, 64, 4), generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    got = []
    for roots in (front, np.concatenate([back, front])):
        r = _renderer(U.scene_of([tpl], U.instances(len(roots), roots), cam), instance_cull=False)
        img, st = r.render_train(cam, stats=True)
        assert st["splats"] == len(roots) * n
        g = r.backward(dl, len(roots))
        torch.cuda.synchronize()
        g["pose"] = g["pose"][-seen:].clone()
        got.append(dict(g, img=img))
        r.close()
    assert torch.equal(got[0]["img"], got[1]["img"])
    for k, a in got[0].items():
        # the sums reach a value in any order
        assert float(a.abs().max()) > 0.0
        assert torch.allclose(got[1][k], a, rtol=1e-4, atol=1e-5 * float(a.abs().max())), k


def _two_gaussians(**kw):
    """Gaussians skinned to the left and to the right leg alone, in different
    8x4 pixel blocks of a 32 x 16 view."""
    z, f = 2.0, 30.0
    px = np.array([[6.5, 6.5], [25.5, 9.5]])
    means = np.stack([(px[:, 0] - 16) * z / f, (px[:, 1] - 8) * z / f, np.full(2, z)], 1)
    tpl = U.template_from(means, [[0.03, 0.05, 0.07], [0.06, 0.04, 0.05]], [[0.8, 0.2, 0.3, -0.1], [0.9, -0.3, 0.2, 0.2]],
                          np.full(2, 0.5),
                          **dict(dict(sh=np.full((2, 1, 3), 0.3), skin_idx=[[4, 5, 2, 3], [5, 4, 1, 3]]), **kw))
    return U.scene_of([tpl], U.instances(1), U.identity_camera(32, 16, f))


@pytest.mark.parametrize("bad", [math.nan, math.inf])
def test_a_bad_pixel_spoils_the_joints_of_its_gaussians_only(bad):
    sc = _two_gaussians()
    r = _renderer(sc)
    out = []
    for v in (0.0, bad):
        dl = torch.ones((16, 32, 4), device="cuda")
        dl[6, 6] = v  # a pixel of the first Gaussian
        r.render_train(sc.camera)
        out.append({k: v.cpu().numpy() for k, v in r.backward(dl, 1).items()})
    r.close()
    good, bad_ = out
    # joint 5 hangs from joint 2, joint 4 (the first Gaussian's) from joint 1
    assert not np.isfinite(bad_["pose"][0, 4]).all()
    assert np.abs(good["pose"][0, 5]).max() > 0.0
    # (the pixels' sums reach a value in any order)
    close = lambda a, b: np.allclose(a, b, rtol=1e-4, atol=1e-5 * np.abs(b).max())
    assert close(bad_["pose"][0, [2, 5]], good["pose"][0, [2, 5]])
    for k in ("means", "scales", "quats", "opacity", "sh"):
        assert close(bad_[k][1], good[k][1]), k


@pytest.mark.parametrize("coefficient", [-math.inf, math.nan])
def test_a_channel_clamped_at_zero_passes_no_gradient_whatever_its_coefficients(coefficient):
    """The red channel is clamped for any very negative coefficient: the same
    gradients as for -100."""
    out = []
    for v in (-100.0, coefficient):
        sh = 0.2 * np.random.default_rng(3).standard_normal((2, 4, 3))
        sh[0, 0, 0] = v
        sc = _two_gaussians(sh=sh)
        r = _renderer(sc)
        img = r.render_train(sc.camera).cpu().numpy()
        assert img[6, 6, 0] == 0.0 and img[6, 6, 1] > 0.0
        dl = torch.ones((16, 32, 4), device="cuda")
        out.append({k: g.cpu().numpy() for k, g in r.backward(dl, 1).items()})
        r.close()
    for k, a in out[0].items():
        assert np.abs(a).max() > 0.0
        assert np.allclose(out[1][k], a, rtol=1e-4, atol=1e-5 * np.abs(a).max()), k
