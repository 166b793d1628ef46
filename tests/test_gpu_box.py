"""Box tests of the traversal in scenes whose extent takes their terms out of the float range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extent", [1e3, 1e15, 1e16, 1e17, 1e18])
@pytest.mark.parametrize("zero", [0.0, -0.0, 1e-21, -1e-21])
def test_rays_along_the_short_axes_of_a_wide_scene(extent, zero):
    """Strips as long as the scene and one unit wide: a ray across them, its direction zero along
    their length, meets exactly the strip below its origin, in every form of the traversal."""
    from paper_2407_19977_gb300 import api, scenes
    n = 96
    v, idx = [], []
    for k in range(n):
        z = float(k % 7)
        v += [(-extent, 2 * k, z), (extent, 2 * k, z), (extent, 2 * k + 1, z), (-extent, 2 * k + 1, z)]
        idx += [(4 * k, 4 * k + 1, 4 * k + 2), (4 * k, 4 * k + 2, 4 * k + 3)]
    sc = scenes.Scene("strips", np.asarray(v, np.float32), np.asarray(idx, np.uint32), np.zeros(2 * n, np.uint32),
                      scenes.diffuse((.5, .5, .5))[None], np.zeros((0, 13), np.float32), scenes.uniform_env(1.0, 8, 4),
                      scenes.Camera((0, 0, 40), (0, 0, 0), (0, 1, 0), 40.0, 16, 16), 1, 2)
    g = api.Scene(sc)
    rng = np.random.default_rng(1)
    k = np.repeat(np.arange(n), 8)
    x = (rng.uniform(-0.9, 0.9, k.size) * extent).astype(np.float32)
    y = (2 * k + rng.choice([0.25, 0.75, 1.5], k.size)).astype(np.float32)
    o = np.stack([x, y, np.full_like(x, 20.0)], 1)
    d = np.tile(np.array([[zero, 0.0, -1.0]], np.float32), (k.size, 1))
    inside = (y % 2) < 1
    for coop in (False, True):
        tri, t, _ = g.trace(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), coop=coop)
        assert np.array_equal(tri.cpu().numpy() >= 0, inside)
        # T and det are sums of three products of rounded terms
        assert np.allclose(t.cpu().numpy()[inside], (20.0 - k % 7)[inside], rtol=1e-6, atol=0)
        hit, _, _ = g.trace(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), any_hit=True, coop=coop)
        assert np.array_equal(hit.cpu().numpy() >= 0, inside)
    assert g.stats()["error_flags"] == 0
