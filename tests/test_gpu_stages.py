"""The staged traversal passes of the wavefront at ragged queue lengths."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scene,crop,spp", [("cornell", (5, 7, 1, 1), 1), ("cornell", (0, 0, 31, 1), 1),
                                            ("pushbutton", (40, 20, 33, 1), 1), ("pushbutton", (0, 0, 127, 9), 3),
                                            ("heavy", (3, 1, 129, 65), 2), ("many_lights", (0, 0, 128, 96), 2)])
def test_staged_passes_equal_path_kernel(scene, crop, spp):
    """Rays held in stages and lanes refilled from the queue (fewer rays than a warp, one more,
    odd counts) against one thread per path to its end: every sample and sum bit for bit."""
    from paper_2407_19977_gb300 import api, native as N, scenes
    make = {"cornell": lambda: scenes.cornell_box(seed=3, width=64, height=64, max_depth=5),
            "pushbutton": lambda: scenes.pushbutton(seed=3, n_profile=30, n_angular=40, width=192, height=108),
            "heavy": lambda: scenes.heavy_scene(seed=3, level=3, n_instances=4, width=160, height=90, max_depth=9),
            "many_lights": lambda: scenes.many_light_box(24, seed=3, width=128, height=96, max_depth=4)}[scene]
    g = api.Scene(make())
    out = []
    for mode, tail in ((N.PT_MODE_MEGAKERNEL, 0), (N.PT_MODE_WAVEFRONT, -1), (N.PT_MODE_WAVEFRONT, 0)):
        s = torch.full((crop[3], crop[2], spp, 3), -1.0, device="cuda")
        acc = g.render(spp, crop=crop, seed=9, mode=mode, tail_paths=tail, sample_out=s)
        out.append((s, acc.sum, acc.comp))
    for other in out[1:]:
        for x, y in zip(out[0], other):
            assert torch.equal(x, y)
    st = g.stats()
    assert st["error_flags"] == 0 and bool((out[0][0] >= 0).all())


@pytest.mark.parametrize("side,spp", [(64, 31), (64, 32), (181, 4), (255, 3)])
def test_auto_picks_either_route_with_the_same_sums(side, spp):
    """Frames on both sides of AUTO's line (131,072 paths), eager and under stream capture, where
    a small frame must not allocate: the sums of both explicit modes, bit for bit."""
    from paper_2407_19977_gb300 import api, native as N, scenes
    sc = scenes.cornell_box(seed=2, width=side, height=side, max_depth=4)
    g = api.Scene(sc)
    acc = api.Accum(side, side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.render(spp, seed=5, accum=acc)
    graph.replay()
    want = g.render(spp, seed=5, mode=N.PT_MODE_WAVEFRONT)
    for a in (acc, g.render(spp, seed=5), g.render(spp, seed=5, mode=N.PT_MODE_MEGAKERNEL)):
        assert torch.equal(a.sum, want.sum) and torch.equal(a.comp, want.comp)


def test_capture_after_a_smaller_call():
    """A captured call of more samples than the call that sized the wave's buffers runs in waves
    that fit them."""
    from paper_2407_19977_gb300 import api, scenes
    sc = scenes.cornell_box(seed=2, width=1536, height=1400, max_depth=3)     # above 2^21 pixels
    g = api.Scene(sc)
    g.render(1, seed=5)
    acc = api.Accum(1536, 1400)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.render(3, seed=5, accum=acc)
    graph.replay()
    want = g.render(3, seed=5)
    assert torch.equal(acc.sum, want.sum) and torch.equal(acc.comp, want.comp)
