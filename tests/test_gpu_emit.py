"""Pair emission: every tile of every live splat's reach box, in depth order
and row-major, for splats of one tile, of a few and of the whole image, in
frames of one block and more, on both sides of the block size's limit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _pairs_of(rec, live_order, tiles_x):
    """(tile, splat) of the reach boxes, splats in depth order, then by tile (stable)."""
    rx, ry = rec[live_order, 12].view(np.uint32), rec[live_order, 13].view(np.uint32)
    x0, x1, y0, y1 = ((a >> 4).astype(np.int64) for a in (rx & 0xFFFF, rx >> 16, ry & 0xFFFF, ry >> 16))
    w, cnt = x1 - x0 + 1, (x1 - x0 + 1) * (y1 - y0 + 1)
    own = np.repeat(np.arange(len(cnt)), cnt)
    k = np.arange(int(cnt.sum())) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    tile = (y0[own] + k // w[own]) * tiles_x + x0[own] + k % w[own]
    by_tile = np.argsort(tile, kind="stable")
    return tile[by_tile], live_order[own][by_tile]


@pytest.mark.parametrize("n,instances,size", [(1, 1, 0.3), (33, 1, 0.05), (1024, 1, 0.3), (1025, 1, 0.01), (4099, 2, 0.02),
                                              (9000, 3, 0.002), (9000, 40, 0.002),
                                              (66000, 64, 0.001)])
def test_pairs_of_the_reach_boxes(n, instances, size):
    from paper_2501_17792_gb300 import binding
    from tests import scene_util as U
    rng = np.random.default_rng(n)
    z = rng.uniform(1.0, 6.0, n)
    means = np.stack([rng.uniform(-1.2, 1.2, n) * z, rng.uniform(-0.8, 0.8, n) * z, z], 1)
    means[::5, 2] *= -1.0  # behind the camera: culled
    if n == 1:
        means[0] = (0.0, 0.0, 2.0)
    scales = size * np.exp(rng.uniform(-2.0, 2.0, (n, 3)))
    tpl = U.template_from(means, scales, np.tile([1.0, 0, 0, 0], (n, 1)), rng.uniform(0.01, 1.0, n), np.zeros((n, 1, 3)))
    sc = U.scene_of([tpl], U.instances(instances), U.identity_camera(403, 259, 260.0))
    r = binding.Renderer(device=0, instance_cull=False)
    r.upload_templates(sc.templates)
    r.set_instances(sc.instances.template_id, sc.instances.root, sc.instances.pose)
    _, st = r.render(sc.camera, stats=True)
    order, keys = r.debug("depth_order").astype(np.int64), r.debug("depth_keys")
    tile, splat = _pairs_of(r.debug("records"), order[keys != 0xFFFFFFFF], st["tiles_x"])
    assert st["pairs"] == len(tile) > 0
    assert np.array_equal(r.debug("pair_tiles").astype(np.int64), tile)
    assert np.array_equal(r.debug("pair_splats").astype(np.int64), splat)
    r.close()
