"""Tree build and scene checks at the sizes where the device build changes its route."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _soup(n, seed, same=False):
    from paper_2407_19977_gb300 import scenes
    rng = np.random.default_rng(seed)
    c = rng.uniform(-1, 1, (1 if same else n, 1, 3))
    v = (c + rng.normal(0, 0.05, (n, 3, 3))).reshape(-1, 3).astype(np.float32)
    return scenes.Scene("soup", v, np.arange(3 * n, dtype=np.uint32).reshape(-1, 3), np.zeros(n, np.uint32),
                        scenes.diffuse((.5, .5, .5))[None], np.zeros((0, 13), np.float32),
                        scenes.uniform_env(1.0, 8, 4), scenes.Camera((0, 0, -4), (0, 0, 0), (0, 1, 0), 40.0, 16, 16), 1, 2)


@pytest.mark.parametrize("n", [1, 2, 3, 33, 1024, 1025, 2047, 2048, 2049, 2050, 4097, 9001])
def test_clustered_tree_around_the_one_block_tail(n):
    """At most 2048 clusters are merged by one block: trees of fewer, exactly as many and more
    triangles are well formed and give the radix tree's hits."""
    from paper_2407_19977_gb300 import api, bvh_check, native as N
    g = api.Scene(_soup(n, n))
    problems, stats = bvh_check.check(*g.export_bvh())
    assert not problems, problems[:3]
    o = torch.from_numpy(np.random.default_rng(1).uniform(-2, 2, (4001, 3)).astype(np.float32)).cuda()
    d = torch.nn.functional.normalize(-o + 0.3, dim=1)
    a = g.trace(o, d)
    g.build(builder=N.PT_BVH_LBVH)
    b = g.trace(o, d)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert g.stats()["error_flags"] == 0


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("what,message", [("vertex", b"non-finite vertex"), ("index", b"vertex index"),
                                          ("material", b"material id"), ("env", b"env texel")])
def test_bad_arrays_are_refused(on_device, what, message):
    from paper_2407_19977_gb300 import api, native as N
    sc = _soup(700, 5)
    if what == "vertex":
        sc.vertices[1234, 1] = np.nan
    elif what == "index":
        sc.indices[699, 2] = 0xFFFFFFFF
    elif what == "material":
        sc.material_ids[699] = 1
    else:
        sc.env[1, 1, 1] = -1.0
    with pytest.raises(Exception):
        api.Scene(sc, on_device=on_device)
    assert message in N.load().pt_last_error()
