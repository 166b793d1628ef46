"""Trees over triangles that sort and cluster alike."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _scene(v):
    from paper_2407_19977_gb300 import scenes
    n = len(v)
    return scenes.Scene("ties", v.reshape(-1, 3).astype(np.float32), np.arange(3 * n, dtype=np.uint32).reshape(-1, 3),
                        np.zeros(n, np.uint32), scenes.diffuse((.5, .5, .5))[None], np.zeros((0, 13), np.float32),
                        scenes.uniform_env(1.0, 8, 4), scenes.Camera((0, 0, -4), (0, 0, 0), (0, 1, 0), 40.0, 16, 16), 1, 2)


def _rays():
    o = torch.from_numpy(np.random.default_rng(1).uniform(-2, 2, (4001, 3)).astype(np.float32)).cuda()
    return o, torch.nn.functional.normalize(-o + 0.01, dim=1)


def _equal(g, rays, want):
    a = g.trace(*rays)
    return torch.equal(a[0], want[0]) and torch.equal(a[1], want[1])


@pytest.mark.parametrize("n", [33, 2049, 9001])
def test_triangles_around_one_centroid(n):
    """Equal centroids up to rounding: most sort keys are equal or differ in their last bits."""
    from paper_2407_19977_gb300 import api, bvh_check, native as N
    e = np.random.default_rng(n).normal(0, 0.2, (n, 3, 3))
    g = api.Scene(_scene(e - e.mean(1, keepdims=True)))
    problems, _ = bvh_check.check(*g.export_bvh())
    assert not problems, problems[:3]
    rays = _rays()
    a = g.trace(*rays)
    g.build(builder=N.PT_BVH_LBVH)
    assert _equal(g, rays, a) and g.stats()["error_flags"] == 0


@pytest.mark.parametrize("n", [2, 33, 300, 2049, 9001])
def test_identical_triangles(n):
    """Every key and every cluster area is the same: one pair merges a round.  Trees of a few
    hundred are built; the chain of a few thousand is refused, and the radix tree still builds."""
    from paper_2407_19977_gb300 import api, bvh_check, native as N
    g = api.Scene(_scene(np.repeat(np.random.default_rng(1).normal(0, 0.5, (1, 3, 3)), n, 0)), build=False)
    rays = _rays()
    g.build(builder=N.PT_BVH_LBVH)
    want = g.trace(*rays)
    assert set(want[0].unique().tolist()) <= {-1, 0}      # the first of them at equal distance
    if n <= 300:
        g.build(builder=N.PT_BVH_PLOC)
        problems, _ = bvh_check.check(*g.export_bvh())
        assert not problems, problems[:3]
    else:
        with pytest.raises(Exception, match="did not terminate"):
            g.build(builder=N.PT_BVH_PLOC)
        g.build(builder=N.PT_BVH_LBVH)
    assert _equal(g, rays, want) and g.stats()["error_flags"] == 0
