"""The walking warps of the compositing at the values where they decide:
colours that are not finite, and stops that hang on one rounding."""
import math

import numpy as np
import pytest

from tests import scene_util as U

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C0 = 0.28209479177387814
F = 30.0
f32 = np.float32


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


def _search(o_first, o, want):
    """Group 1: 1,024 splats of 1 - alpha = o_first; group 2: twelve of the
    values o, the last chosen so that the pair-by-pair T and T0 times the
    group's product fall on opposite sides of the stop threshold (`want`:
    which of the two is below).  Returns the group's indices into o, T before
    the last splat, T after it, T0 times the product."""
    T0 = f32(1.0)
    for _ in range(1024):
        T0 = T0 * o_first
    rng = np.random.default_rng(1)
    for _ in range(40):
        idx = rng.integers(0, len(o), (200000, 11))
        T, P = np.full(len(idx), T0, f32), np.ones(len(idx), f32)
        for k in range(idx.shape[1]):
            T, P = T * o[idx[:, k]], P * o[idx[:, k]]
        keep = (T > 1.2e-4) & (T < 1.9e-4)
        idx, T, P = idx[keep], T[keep], P[keep]
        T2, Tq = T[:, None] * o[None], T0 * (P[:, None] * o[None])
        hit = (T2 < f32(1e-4)) & (Tq >= f32(1e-4)) if want == "T" else (T2 >= f32(1e-4)) & (Tq < f32(1e-4))
        if hit.any():
            i, j = np.argwhere(hit)[0]
            return list(idx[i]) + [int(j)], T[i], T2[i, j], Tq[i, j]
    raise AssertionError("no such sequence")


@pytest.mark.parametrize("front", [0, 8192])
@pytest.mark.parametrize("case", ["reopened", "stays stopped", "closed by the product"])
def test_stops_that_hang_on_one_rounding(case, front):
    """Training frames settle T every 1,024 pairs as T0 times the product of
    the group.  A pixel that stopped by its pair-by-pair T, but not by that
    product, takes the stopping splat if nothing follows in the group, and
    stays stopped if something does; one that is below the threshold by the
    product alone takes no more.  The same in lists composited in turn and
    (behind 8,192 splats of another block) in chunks."""
    at, aside = (8.5, 8.5), (2.5, 2.5)
    levels = np.linspace(0.2, 0.45, 200)
    # 1 - alpha of each opacity as the frames compute it: alpha < 1/2, so the
    # image's 1 - (1 - alpha) is exact
    cal = _pixel_scene([at] * 201, [0.0045] + list(levels), [0.0] * 201)
    r = _renderer(cal)
    o = np.empty(201, f32)
    for k in range(201):
        r.set_lod_subset(0, 0, [k])
        o[k] = f32(1.0) - f32(r.render_train(cal.camera)[8, 8, 3].item())
    r.close()
    idx, T1, T2, Tq = _search(o[0], o[1:], "P" if case == "closed by the product" else "T")
    group2 = [levels[k] for k in idx] + ([0.3] if case == "stays stopped" else [])
    rest = 1024 - len(group2)
    opacity = [0.5] * front + [0.0045] * 1024 + group2 + [0.5] * rest + [0.3] * 2
    px = [aside] * front + [at] * (1024 + len(group2)) + [aside] * rest + [at] * 2
    dc = np.zeros(len(px))
    stop = front + 1024 + len(idx) - 1
    dc[stop] = 1e4 / C0
    dc[-2:] = 1e4 / C0
    sc = _pixel_scene(px, opacity, dc)
    r = _renderer(sc)
    img, st = r.render_train(sc.camera, stats=True)
    assert st["pairs"] == len(px)
    dl = torch.zeros((16, 16, 4), device="cuda")
    dl[8, 8, 0] = 1.0
    g = r.backward(dl, 1)["sh"][:, 0, 0].cpu().numpy()
    r.close()
    T = {"reopened": Tq, "stays stopped": T1, "closed by the product": T2}[case]
    red, alpha = float(img[8, 8, 0]), f32(img[8, 8, 3].item())
    assert alpha == f32(1.0) - T
    # the stopping splat's weight; the grey 0.5 of all taken ones
    w = 0.0 if case == "stays stopped" else float(1.0 - o[1 + idx[-1]]) * float(T1)
    # about a thousand roundings of the sum and of T
    assert abs(red - (0.5 * (1.0 - float(T)) + 1e4 * w)) <= 1e-4 + 1e-4 * 1e4 * w
    # the backward recovers T by divisions
    assert abs(g[stop] - C0 * w) <= 5e-4 * C0 * max(w, 1e-5)
    assert g[-1] == 0.0 and g[-2] == 0.0
