"""Which route PT_MODE_AUTO takes, seen by the launches of a call."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _launches(g, *args, **kw):
    from paper_2407_19977_gb300 import native as N
    torch.cuda.synchronize()
    before = N.load().pt_launch_count()
    acc = g.render(*args, **kw)
    torch.cuda.synchronize()
    return N.load().pt_launch_count() - before, acc


# paths: below 2^17 the path kernel (one launch), from there the wavefront; a small frame in waves
# of fewer than 2^17 paths stays with the path kernel, a large one with its options does not
@pytest.mark.parametrize("width,height,spp,opts,one", [
    (64, 64, 31, {}, True), (64, 64, 32, {}, False), (255, 255, 2, {}, True), (255, 255, 3, {}, False),
    (255, 255, 3, dict(wave_paths=1000), True), (255, 255, 3, dict(wave_paths=(1 << 17) - 1), True),
    (255, 255, 3, dict(wave_paths=1 << 17), False), (255, 255, 3, dict(wave_paths=1 << 23), False),
    (320, 256, 1, {}, True), (320, 256, 1, dict(wave_paths=1 << 20), False), (320, 256, 1, dict(use_graph=True), False),
    (512, 256, 1, {}, False)])
def test_auto_route(width, height, spp, opts, one):
    from paper_2407_19977_gb300 import api, native as N, scenes
    g = api.Scene(scenes.cornell_box(seed=2, width=width, height=height, max_depth=4))
    n, acc = _launches(g, spp, seed=5, **opts)
    assert (n == 1) == one and n < 200
    want = g.render(spp, seed=5, mode=N.PT_MODE_MEGAKERNEL)
    assert torch.equal(acc.sum, want.sum) and torch.equal(acc.comp, want.comp)


def test_path_kernel_of_more_pixels_than_a_grid_has_blocks():
    """2^31 pixels and more with the smallest blocks, one pixel a block if its samples went side
    by side."""
    from paper_2407_19977_gb300 import api, native as N, scenes
    width, height = 65536, 32769
    if torch.cuda.mem_get_info()[0] < width * height * 28:
        pytest.skip("needs the accumulators' memory")
    sc = scenes.cornell_box(seed=2, width=width, height=height, max_depth=0)
    sc.lights = sc.lights[:0]
    sc.vertices = sc.vertices.copy()
    sc.vertices[:, 2] -= 1e4                    # far away: (nearly) every ray leaves the scene
    sc.env = scenes.uniform_env(0.5, 8, 4)
    g = api.Scene(sc)
    acc = api.Accum(width, height)
    g.render(17, seed=5, accum=acc, mode=N.PT_MODE_MEGAKERNEL, block_size=32)
    torch.cuda.synchronize()
    for rows in (slice(0, 64), slice(height - 64, height)):
        s = acc.sum[rows]
        assert float((s == 8.5).float().mean()) > 0.99
    assert float(acc.sum[height // 2, :, 0].max()) == 8.5
