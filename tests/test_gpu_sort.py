"""Sorts of up to 32,768 elements run in one launch (a cluster of up to eight
CTAs of 4,096), larger ones pass by pass.  Rankings around those sizes against
a stable sort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[1], [31], [4096], [4097], [12289, 3], [8192, 8192, 8191], [32768], [32769], [40000, 1]])
@pytest.mark.parametrize("levels", [3, 1 << 24])
def test_rankings_against_a_stable_sort(sizes, levels):
    from paper_2501_17792_gb300 import binding
    from tests import scene_util as U
    rng = np.random.default_rng(sum(sizes) + levels)
    tpls = [U.template_from(rng.uniform(-1, 1, (n, 3)), np.full((n, 3), 0.01), np.tile([1.0, 0, 0, 0], (n, 1)),
                            np.full(n, 0.5), np.zeros((n, 1, 3))) for n in sizes]
    r = binding.Renderer(device=0)
    r.upload_templates(tpls)
    # few levels: long runs of equal scores, whose order is by index
    score = (rng.integers(-levels, levels + 1, sum(sizes)) / np.float32(levels)).astype(np.float32)
    got = r.lod_rank(torch.from_numpy(score).cuda()).cpu().numpy()
    off = 0
    for n in sizes:
        want = np.argsort(-score[off:off + n], kind="stable")
        assert np.array_equal(got[off:off + n], want)
        off += n
    r.close()


@pytest.mark.parametrize("n", [1, 4096, 4097, 32768, 32769])
def test_depth_order_of_frames_around_the_one_launch_sort(n):
    """Key ties by splat id, culled splats last, in frames of n splats."""
    from paper_2501_17792_gb300 import binding
    from tests import scene_util as U
    rng = np.random.default_rng(n)
    z = rng.uniform(0.5, 6.0, n).astype(np.float32)
    z[::3] = np.round(z[::3] * 8) / 8  # equal depths
    means = np.stack([rng.uniform(-0.4, 0.4, n) * z, rng.uniform(-0.4, 0.4, n) * z, z], 1)
    means[::17, 2] *= -1.0  # behind the camera: culled
    tpl = U.template_from(means, np.full((n, 3), 0.01), np.tile([1.0, 0, 0, 0], (n, 1)), np.full(n, 0.5),
                          np.zeros((n, 1, 3)))
    sc = U.scene_of([tpl], U.instances(1), U.identity_camera(64, 48, 60.0))
    r = binding.Renderer(device=0, instance_cull=False)
    r.upload_templates(sc.templates)
    r.set_instances(sc.instances.template_id, sc.instances.root, sc.instances.pose)
    _, st = r.render(sc.camera, stats=True)
    order, keys = r.debug("depth_order").astype(np.int64), r.debug("depth_keys").astype(np.int64)
    assert np.array_equal(np.sort(order), np.arange(n))
    assert (np.diff(keys) >= 0).all()
    same = np.diff(keys) == 0
    assert (np.diff(order)[same] > 0).all()
    assert (keys != 0xFFFFFFFF).sum() == st["splats_live"]
    r.close()
