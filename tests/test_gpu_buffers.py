"""Lifetime and size of the wavefront's work buffers."""
import gc

import pytest
import torch

pytestmark = pytest.mark.gpu


def _used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("captured,later,opts", [(3, 3, {}), (1, 5, {}), (1, 6, dict(wave_paths=1 << 24)),
                                                 (1, 4, dict(use_graph=True))])
def test_captured_call_replays_after_a_larger_call(captured, later, opts):
    """A larger call after a capture replaces the wave's buffers; the captured graph still holds
    the old ones, which live until the scene ends."""
    from paper_2407_19977_gb300 import api, native as N, scenes
    w, h = 1536, 700
    torch.cuda.synchronize()
    g = api.Scene(scenes.cornell_box(seed=2, width=w, height=h, max_depth=3))
    want = g.render(captured, seed=5, mode=N.PT_MODE_MEGAKERNEL)
    acc = api.Accum(w, h)
    big = api.Accum(w, h)
    g.render(1, seed=5, mode=N.PT_MODE_WAVEFRONT, wave_paths=1 << 20)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.render(captured, seed=5, accum=acc, mode=N.PT_MODE_WAVEFRONT, wave_paths=1 << 20)
    before = _used()
    g.render(later, seed=6, accum=big, mode=N.PT_MODE_WAVEFRONT, **opts)
    assert _used() > before             # new buffers beside those of the capture
    keep = big.sum.clone()
    for _ in range(2):
        acc.reset()
        graph.replay()
        assert torch.equal(acc.sum, want.sum) and torch.equal(acc.comp, want.comp)
    assert torch.equal(big.sum, keep)
    grown = _used()
    del graph, g
    gc.collect()
    assert _used() < grown - (160 << 20)    # both sets go with the scene (at least 2^20 paths)
