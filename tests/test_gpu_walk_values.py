"""The walking warps of the compositing with colours that are not finite."""
import math

import numpy as np
import pytest

from tests import scene_util as U

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

F = 30.0


def _pixel_scene(px, opacity, dc):
    """Small Gaussians (a pixel or two) at the centres px [n, 2] of a 16 x 16
    image, in this depth order, with the red channel's degree-0 coefficient."""
    px, opacity, dc = np.asarray(px, np.float64), np.asarray(opacity), np.asarray(dc)
    n = len(px)
    z = 1.0 + 1e-3 * np.arange(n)
    means = np.stack([(px[:, 0] - 8.5) * z / F, (px[:, 1] - 8.5) * z / F, z], 1)
    sh = np.zeros((n, 1, 3))
    sh[:, 0, 0] = dc
    tpl = U.template_from(means, np.full((n, 3), 1e-4), np.tile([1.0, 0, 0, 0], (n, 1)), opacity, sh)
    return U.scene_of([tpl], U.instances(1), U.identity_camera(16, 16, F, cx=8.5, cy=8.5))


def _renderer(sc):
    from paper_2501_17792_gb300 import binding
    r = binding.Renderer(device=0)
    r.upload_templates(sc.templates)
    r.set_instances(sc.instances.template_id, sc.instances.root, sc.instances.pose)
    return r


@pytest.mark.parametrize("kind, front", [("contrib", 0), ("contrib", 300), ("train", 0), ("train", 8200), ("plain", 32800)])
def test_an_infinite_colour_stays_in_its_pixels(kind, front):
    """Weight zero times an infinite colour must not reach the other pixels of
    the 8x4 block.  Behind `front` splats of another block: the lists' chunks
    in parallel (8,192 pairs and more in training frames, 32,768 in plain ones)."""
    px = [(2.5, 2.5)] * front + [(11.5, 13.5)]
    img = []
    for dc in (0.0, math.inf):
        sc = _pixel_scene(px, [0.5] * (front + 1), [0.0] * front + [dc])
        r = _renderer(sc)
        if kind == "contrib":
            img.append(r.render_contrib(sc.camera, torch.zeros(front + 1, device="cuda")).cpu().numpy())
        else:
            img.append((r.render_train if kind == "train" else r.render)(sc.camera).cpu().numpy())
        r.close()
    y, x = np.mgrid[0:16, 0:16] + 0.5
    away = (x - 11.5) ** 2 + (y - 13.5) ** 2 > 9.0  # past the splat's reach
    assert np.array_equal(img[1][away], img[0][away])
    assert np.isinf(img[1][13, 11, 0]) and np.array_equal(img[1][..., 1:], img[0][..., 1:])
