"""Lifetime and size of the wavefront's work buffers."""
import contextlib
import gc

import pytest
import torch

pytestmark = pytest.mark.gpu


def _used():
    """Device memory in use outside torch's own pool."""
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free - torch.cuda.memory_reserved()


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


@contextlib.contextmanager
def _only(leave):
    """Device memory taken so that about `leave` bytes are free."""
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    room = [torch.empty(free - leave, dtype=torch.uint8, device="cuda")]
    try:
        yield
    finally:
        room.clear()
        torch.cuda.empty_cache()


def _net(sc):
    from paper_2407_19977_gb300 import api
    lo, hi = sc.vertices.min(0) - 0.01, sc.vertices.max(0) + 0.01
    return api.Nrc(seed=3, box=(tuple(lo), tuple(hi)))


# bytes a path: 168 in the queues, 84 more with the cache's queries, 112 with reservoirs; the large
# wave holds 6.45M or 4.3M paths (1.08 / 0.72 GB of queues), the small one one sample of the frame
@pytest.mark.parametrize("kind,spp,leave", [("plain", 3, 700 << 20), ("plain after a small call", 3, 700 << 20),
                                            ("graph", 3, 700 << 20), ("cache", 3, 1300 << 20),
                                            ("cache after a plain call", 3, 400 << 20),
                                            ("reservoirs", 2, 900 << 20)])
def test_smaller_waves_where_the_large_one_does_not_fit(kind, spp, leave):
    """Without room for the automatic wave, or for the buffers that go with it, a call runs in
    smaller waves: the same sums, and later calls neither allocate nor free anything."""
    from paper_2407_19977_gb300 import api, native as N, scenes
    w, h = 1536, 1400
    sc = scenes.cornell_box(seed=2, width=w, height=h, max_depth=3)
    g = api.Scene(sc)
    net = _net(sc) if "cache" in kind else None
    opts = dict(seed=5, mode=N.PT_MODE_WAVEFRONT, nrc=net, use_graph=kind == "graph",
                restir=(4, 2, 5, 0) if kind == "reservoirs" else None)
    want = g.render(spp, wave_paths=w * h, **opts)
    del g
    g = api.Scene(sc)
    if kind == "plain after a small call":
        g.render(1, seed=1, wave_paths=1 << 21)
    if kind == "cache after a plain call":
        g.render(spp, seed=1, mode=N.PT_MODE_WAVEFRONT)
    acc = api.Accum(w, h)
    used = []
    with _only(leave):
        for _ in range(3):
            acc.reset()
            g.render(spp, accum=acc, **opts)
            used.append(_used())
            assert torch.equal(acc.sum, want.sum) and torch.equal(acc.comp, want.comp)
    assert used[0] == used[1] == used[2]
    if kind == "graph":
        assert g.stats()["graph_replays"] == 2


@pytest.mark.parametrize("leave,most", [(15, 360 << 20), (17, 1200 << 20)])
def test_large_wave_takes_a_sixteenth_of_the_free_memory_at_most(leave, most):
    """3 samples of 2.15M pixels: 1.08 GB of queues in one wave, 0.36 in waves of one sample."""
    from paper_2407_19977_gb300 import api, native as N, scenes
    w, h = 1536, 1400
    sc = scenes.cornell_box(seed=2, width=w, height=h, max_depth=3)
    want = api.Scene(sc).render(3, seed=5, mode=N.PT_MODE_MEGAKERNEL)
    g = api.Scene(sc)
    acc = api.Accum(w, h)
    with _only(leave * 3 * w * h * 168 + (16 << 20)):
        before = _used()
        g.render(3, seed=5, accum=acc)
        grown = _used() - before
    assert most * 0.85 < grown <= most
    assert torch.equal(acc.sum, want.sum) and torch.equal(acc.comp, want.comp)


def test_small_frame_without_room_for_a_wave():
    """A small frame that AUTO sends to the wavefront renders all the same where no wave fits."""
    from paper_2407_19977_gb300 import api, native as N, scenes
    g = api.Scene(scenes.cornell_box(seed=2, width=255, height=255, max_depth=3))
    want = g.render(64, seed=5, mode=N.PT_MODE_MEGAKERNEL)
    acc = api.Accum(255, 255)
    with _only(100 << 20):
        for _ in range(2):
            acc.reset()
            g.render(64, seed=5, accum=acc)
            assert torch.equal(acc.sum, want.sum) and torch.equal(acc.comp, want.comp)


def test_only_recorded_buffers_are_kept():
    """After a capture, calls that replace the cache's buffers again and again (two caches of
    different training sets) keep the recorded set and no other; the captured graph replays."""
    from paper_2407_19977_gb300 import api, native as N, scenes
    w, h = 1024, 640
    sc = scenes.cornell_box(seed=2, width=w, height=h, max_depth=3)
    lo, hi = tuple(sc.vertices.min(0) - 0.01), tuple(sc.vertices.max(0) + 0.01)
    g = api.Scene(sc)
    nets = [api.Nrc(seed=3, box=(lo, hi), frame_samples=1 << k) for k in (15, 16)]
    acc, other = api.Accum(w, h), api.Accum(w, h)
    opts = dict(seed=5, mode=N.PT_MODE_WAVEFRONT)
    want = g.render(1, nrc=nets[0], **opts)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.render(1, nrc=nets[0], accum=acc, **opts)
    used = []
    for k in range(6):
        g.render(1, nrc=nets[k % 2], accum=other, **opts)
        g.render(1, nrc=nets[(k + 1) % 2], accum=other, **opts)
        used.append(_used())
    assert used[-1] == used[1]
    acc.reset()
    graph.replay()
    assert torch.equal(acc.sum, want.sum) and torch.equal(acc.comp, want.comp)
