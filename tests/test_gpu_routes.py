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
