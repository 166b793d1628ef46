"""What this renderer is used for, as cases that can be timed and compared.

Each case is one call sequence of a program that uses the package: a preview tile, a still, a
progressive frame, opening a model, a many-light frame, a batch of thumbnails, a frame with the
radiance cache, the cache's training and queries, the denoiser.  Scenes come from the
package's seeded generators; the seed of a case picks the generator's seed and the samples.
"""
import math

import numpy as np
import torch

from paper_2407_19977_gb300 import api, native, scenes

BMFR_COLUMNS = 10
NRC_LEVELS, NRC_LOG2_TABLE, NRC_BASE, NRC_FINEST, NRC_WIDTH = 16, 19, 16, 2048, 64
NRC_PRIMES = (1, 2654435761, 805459861)

# extension + shadow rays a path takes on average in each kind of scene (measured with
# Scene.stats() at the depths below), and the box and triangle arithmetic of one such ray
RAYS_PER_PATH = {"cornell": 7.0, "pushbutton": 2.7, "velvet": 2.7, "heavy": 3.6, "many_lights": 7.0}
FLOPS_PER_RAY = {"cornell": 700, "pushbutton": 1700, "velvet": 1700, "heavy": 2200, "many_lights": 1500}


def listed():
    return [
        # a material or thumbnail preview: the smallest frame anybody renders, launch-bound
        dict(name="preview_tile", kind="frame", scene="cornell", tris=34, width=64, height=64, spp=16, depth=4,
             graph=False, wave=0, lens=0.0),
        # the published comparison's still: 512 x 512 at depth 5 on the ~100k-triangle mesh
        dict(name="still_512", kind="frame", scene="pushbutton", tris=106873, width=512, height=512, spp=25, depth=5,
             graph=False, wave=0, lens=0.0),
        # the headline workload: one progressive step of the CAD model at 1080p, four samples in one wave
        dict(name="cad_1080p", kind="frame", scene="pushbutton", tris=209600, width=1920, height=1080, spp=4, depth=8,
             graph=True, wave=1 << 23, lens=0.0),
        # glass, metal and coated spheres, deep paths, an odd window size, default options
        dict(name="glass_odd", kind="frame", scene="heavy", tris=1310720, width=1917, height=1079, spp=2, depth=12,
             graph=False, wave=0, lens=0.0),
        # fuzz layer through a thin lens, ragged size
        dict(name="velvet_lens", kind="frame", scene="velvet", tris=209600, width=961, height=541, spp=3, depth=8,
             graph=False, wave=0, lens=0.03),
        # interactive viewing: one sample, its features, the denoised image and the display resolve
        dict(name="view_denoised", kind="view", scene="pushbutton", tris=209600, width=1920, height=1080, depth=8),
        # opening a model: upload, tree build and the first picture
        dict(name="open_model", kind="open", scene="pushbutton", tris=1068735, width=640, height=360, depth=5),
        # many small lights with reservoir resampling
        dict(name="many_lights", kind="restir", lights=248, width=1920, height=1080, spp=1, depth=4,
             candidates=8, neighbors=5, radius=10, later=0),
        # a set of uneven scenes in one call
        dict(name="batch_12", kind="batch", scenes=12, max_tris=200000, side=512, spp=12, depth=8),
        # a frame that ends its paths in a trained radiance cache
        dict(name="cached_frame", kind="cached", width=1920, height=1080, spp=1, depth=4),
        # online training of the cache: one frame's samples, four optimiser steps
        dict(name="cache_train", kind="train", samples=32768, batch=8192),
        # the cache queried on its own
        dict(name="cache_query", kind="query", queries=1000003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "view", "open", "restir", "batch", "cached", "train", "query",
                       "denoise"])
    w = _log_int(rng, 64, 1920)
    h = max(16, min(1080, int(w * rng.uniform(0.5, 1.0))))
    if kind == "frame":
        scene = rng.choice(["cornell", "pushbutton", "heavy", "velvet"])
        spp = max(1, min(_log_int(rng, 1, 32), 8000000 // (w * h)))
        return dict(kind=kind, scene=scene, tris=_log_int(rng, 1000, 1000000) if scene != "cornell" else 34, width=w,
                    height=h, spp=spp, depth=rng.randint(2, 12), graph=rng.random() < 0.5,
                    wave=rng.choice([0, 0, 1 << 20, 1 << 23]), lens=rng.choice([0.0, 0.0, 0.03]))
    if kind == "view":
        return dict(kind=kind, scene=rng.choice(["pushbutton", "heavy"]), tris=_log_int(rng, 1000, 500000), width=w,
                    height=h, depth=rng.randint(2, 10))
    if kind == "open":
        return dict(kind=kind, scene=rng.choice(["pushbutton", "heavy"]), tris=_log_int(rng, 100, 1000000),
                    width=min(w, 640), height=min(h, 360), depth=5)
    if kind == "restir":
        return dict(kind=kind, lights=rng.randint(8, 248), width=w, height=h, spp=1, depth=rng.randint(1, 4),
                    candidates=rng.choice([4, 8, 32]), neighbors=rng.randint(0, 6), radius=rng.randint(3, 20),
                    later=rng.choice([0, 0, 8]))
    if kind == "batch":
        return dict(kind=kind, scenes=rng.randint(2, 12), max_tris=_log_int(rng, 2000, 200000),
                    side=rng.choice([128, 256, 512]), spp=rng.randint(1, 12), depth=rng.randint(3, 8))
    if kind == "cached":
        return dict(kind=kind, width=w, height=h, spp=1, depth=rng.randint(3, 6))
    if kind == "train":
        return dict(kind=kind, samples=_log_int(rng, 2000, 32768), batch=rng.choice([4096, 8192, 16384]))
    if kind == "query":
        return dict(kind=kind, queries=_log_int(rng, 33, 1000000))
    return dict(kind="denoise", width=w, height=h, block=rng.choice([8, 16, 32, 32]))


# ---------------------------------------------------------------------------------- inputs

def _scene(case, seed):
    name, depth = case["scene"], case["depth"]
    if name == "cornell":
        sc = scenes.cornell_box(seed=seed, max_depth=depth)
    elif name == "heavy":
        level = 0
        while level < 7 and 20 * 4 ** (level + 1) * 2 <= case["tris"]:
            level += 1
        n = int(min(max(round(case["tris"] / (20 * 4 ** level)), 1), 16))
        sc = scenes.heavy_scene(seed=seed, level=level, n_instances=n, max_depth=depth)
    else:
        n = max(int(round(math.sqrt(max(case["tris"], 64) / 3.2))), 4)
        make = scenes.pushbutton_fuzz if name == "velvet" else scenes.pushbutton
        sc = make(seed=seed, n_profile=n, n_angular=max(int(case["tris"] / (2 * n - 1)), 8), max_depth=depth)
    return sc


def _view(sc, case):
    kw = dict(width=case["width"], height=case["height"])
    if case.get("lens", 0.0) > 0.0:
        o, t = np.asarray(sc.camera.origin, float), np.asarray(sc.camera.target, float)
        kw.update(lens_radius=case["lens"], focus_distance=float(np.linalg.norm(t - o)))
    return sc.with_camera(**kw)


def _nrc_params(seed):
    """Weights and grid table of a cache as a program reads them back from a file."""
    rng = np.random.default_rng(seed + 11)
    w = []
    for i in range(5):
        rows = NRC_WIDTH if i < 4 else 16
        m = rng.normal(size=(rows, NRC_WIDTH)) * math.sqrt(2.0 / NRC_WIDTH)
        if i == 4:
            m[3:] = 0.0
        w.append(m.astype(np.float32))
    grid = rng.uniform(-0.5, 0.5, size=(NRC_LEVELS, 1 << NRC_LOG2_TABLE, 2)).astype(np.float32)
    return w, grid


def _nrc(seed, box=((0.0, 0.0, 0.0), (1.0, 1.0, 1.0)), batch=8192, load=True):
    net = api.Nrc(seed=seed, box=box, batch=batch)
    if load:
        w, grid = _nrc_params(seed)
        net.params(0).copy_(torch.from_numpy(np.concatenate([m.ravel() for m in w])))
        net.params(1).copy_(torch.from_numpy(grid.ravel()))
        net.commit()
    return net


def _records(seed, n):
    rng = np.random.default_rng(seed + 7)
    rec = np.zeros((n, 16), np.float32)
    rec[:, 0:3] = rng.random((n, 3))
    for c in (3, 6):
        d = rng.normal(size=(n, 3))
        rec[:, c:c + 3] = d / np.linalg.norm(d, axis=1, keepdims=True)
    rec[:, 9] = rng.random(n)
    rec[:, 10:13] = rng.random((n, 3))
    return rec


def _gbuffer(case, seed):
    """A noisy colour image and the features of a smooth surface with a band of sky."""
    h, w = case["height"], case["width"]
    rng = np.random.default_rng(seed + 3)
    y, x = np.meshgrid(np.arange(h) / h, np.arange(w) / w, indexing="ij")
    f1, f2, ph = rng.uniform(3, 9), rng.uniform(3, 9), rng.uniform(0, 6)
    z = 0.2 * np.sin(f1 * x + ph) * np.cos(f2 * y)
    zx = 0.2 * f1 * np.cos(f1 * x + ph) * np.cos(f2 * y)
    zy = -0.2 * f2 * np.sin(f1 * x + ph) * np.sin(f2 * y)
    nrm = np.stack([-zx, -zy, np.ones_like(z)], 2)
    nrm /= np.linalg.norm(nrm, axis=2, keepdims=True)
    feats = np.zeros((h, w, 12), np.float32)
    feats[..., 0:3] = nrm
    feats[..., 3] = np.where(y < 0.15 + 0.1 * np.sin(5 * x + ph), 0.0, 1.0)
    feats[..., 4:7] = np.stack([x, y, z], 2)
    feats[..., 8:11] = 0.2 + 0.6 * rng.random(3) * (0.6 + 0.4 * np.sign(np.sin(20 * x)))[..., None]
    color = (feats[..., 8:11] * (0.5 + nrm[..., 2:3]) * rng.exponential(1.0, size=(h, w, 1))).astype(np.float32)
    return color, feats


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("frame", "view"):
        sc = _view(_scene(case, seed), case)
        return dict(case=case, seed=seed, scene=api.Scene(sc), acc=api.Accum(case["width"], case["height"]))
    if kind == "open":
        return dict(case=case, seed=seed, desc=_view(_scene(case, seed), case))
    if kind == "restir":
        sc = scenes.many_light_box(case["lights"], seed=seed, width=case["width"], height=case["height"],
                                   max_depth=case["depth"])
        return dict(case=case, seed=seed, scene=api.Scene(sc), acc=api.Accum(case["width"], case["height"]))
    if kind == "batch":
        jobs = []
        for i, sp in enumerate(scenes.batch_specs(case["scenes"], seed=seed, max_tris=case["max_tris"])):
            side = case["side"] if i % 2 == 0 else case["side"] * 3 // 4 + 1
            sc = scenes.scene_from_spec(dict(sp, width=side, height=side))
            jobs.append((api.Scene(sc), sc.camera, 1 + (sp["spp"] * case["spp"]) // 33, case["depth"], sp["seed"],
                         api.Accum(side, side)))
        return dict(case=case, jobs=jobs)
    if kind == "cached":
        sc = scenes.cornell_box(seed=seed, width=case["width"], height=case["height"], max_depth=case["depth"])
        lo, hi = sc.vertices.min(0), sc.vertices.max(0)
        net = _nrc(seed, box=(tuple(map(float, lo)), tuple(map(float, hi))))
        return dict(case=case, seed=seed, scene=api.Scene(sc), net=net, acc=api.Accum(case["width"], case["height"]))
    if kind == "train":
        return dict(case=case, net=_nrc(seed, batch=case["batch"], load=False),
                    rec=torch.from_numpy(_records(seed, case["samples"])).cuda())
    if kind == "query":
        return dict(case=case, net=_nrc(seed), rec=torch.from_numpy(_records(seed, case["queries"])).cuda())
    color, feats = _gbuffer(case, seed)
    return dict(case=case, color=torch.from_numpy(color).cuda(), feats=torch.from_numpy(feats).cuda())


# ---------------------------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "frame":
        acc = state["acc"]
        acc.reset()   # the camera moved: a new progressive image
        state["scene"].render(case["spp"], max_depth=case["depth"], seed=state["seed"], accum=acc,
                              wave_paths=case["wave"], use_graph=case["graph"])
        return acc.sum, acc.comp
    if kind == "view":
        acc, sc = state["acc"], state["scene"]
        acc.reset()
        sc.render(1, max_depth=case["depth"], seed=state["seed"], accum=acc, use_graph=True)
        feats = sc.features(1, seed=state["seed"])
        return dict(sum=acc.sum, features=feats, denoised=api.bmfr(acc.image(), feats), display=acc.tonemap())
    if kind == "open":
        state["scene"] = api.Scene(state["desc"])   # replaces the model that was open before
        return state["scene"].render(1, max_depth=case["depth"], seed=state["seed"]).sum
    if kind == "restir":
        acc = state["acc"]
        acc.reset()
        state["scene"].render(case["spp"], max_depth=case["depth"], seed=state["seed"], accum=acc,
                              mode=native.PT_MODE_WAVEFRONT, use_graph=True,
                              restir=(case["candidates"], case["neighbors"], case["radius"], case["later"]))
        return acc.sum
    if kind == "batch":
        for job in state["jobs"]:
            job[5].reset()
        api.render_batch(state["jobs"], mode=native.PT_MODE_WAVEFRONT, merged=True, use_graph=True, wave_paths=1 << 23)
        return [job[5].sum for job in state["jobs"]]
    if kind == "cached":
        acc = state["acc"]
        acc.reset()
        state["scene"].render(case["spp"], max_depth=case["depth"], seed=state["seed"], accum=acc,
                              mode=native.PT_MODE_WAVEFRONT, nrc=state["net"], use_graph=True)
        return acc.sum
    if kind == "train":
        state["net"].train(state["rec"])
        # copies: params() views memory that ends with the cache
        return state["net"].params(0).clone(), state["net"].params(1).clone()
    if kind == "query":
        return state["net"].infer(state["rec"])
    return api.bmfr(state["color"], state["feats"], block=case["block"])


# ---------------------------------------------------------------------------------- floors

def _frame_work(scene, tris, width, height, spp, depth):
    paths = width * height * spp
    # positions (about half as many vertices as triangles), indices, material ids; sum and compensation out
    return dict(bytes=tris * (6 + 12 + 4) + width * height * 24,
                flops=paths * min(RAYS_PER_PATH[scene], 2 * depth + 1) * FLOPS_PER_RAY[scene])


def work(case):
    kind = case["kind"]
    if kind in ("frame", "view", "open"):
        w = _frame_work(case["scene"], case["tris"], case["width"], case["height"], case.get("spp", 1), case["depth"])
        if kind == "view":
            # a feature ray a pixel; features and the denoised and display images out
            px = case["width"] * case["height"]
            w = dict(bytes=w["bytes"] + px * (48 + 12 + 4), flops=w["flops"] + px * FLOPS_PER_RAY[case["scene"]])
        return w
    if kind == "restir":
        w = _frame_work("many_lights", 34 + 2 * case["lights"], case["width"], case["height"], case["spp"], case["depth"])
        return dict(bytes=w["bytes"], flops=w["flops"] + case["width"] * case["height"] * case["spp"] * 60.0 *
                    (case["candidates"] + 3 * case["neighbors"]))
    if kind == "batch":
        # sides alternate between the full and three quarters of it, triangles log-uniform from 1,000
        px = case["side"] ** 2 * 0.78
        tris = (case["max_tris"] - 1000) / max(math.log(case["max_tris"] / 1000.0), 1e-9)
        one = _frame_work("pushbutton", tris, 1, 1, 1, case["depth"])
        return dict(bytes=case["scenes"] * (tris * 22 + px * 24),
                    flops=case["scenes"] * px * (1 + case["spp"] / 2) * one["flops"])
    if kind == "cached":
        w = _frame_work("cornell", 34, case["width"], case["height"], case["spp"], 2)
        q = case["width"] * case["height"] * case["spp"]
        return dict(bytes=w["bytes"] + (NRC_LEVELS << NRC_LOG2_TABLE) * 4,
                    flops=w["flops"] + q * 2.0 * (4 * 64 * 64 + 3 * 64))
    if kind == "train":
        # each record once; the table's touched entries (at most all) read and written
        entries = min(NRC_LEVELS << NRC_LOG2_TABLE, case["samples"] * NRC_LEVELS * 8)
        return dict(bytes=case["samples"] * 52 + entries * 2 * 4 * 2,
                    flops=case["samples"] * 6.0 * (4 * 64 * 64 + 3 * 64))
    if kind == "query":
        entries = min(NRC_LEVELS << NRC_LOG2_TABLE, case["queries"] * NRC_LEVELS * 8)
        return dict(bytes=case["queries"] * (40 + 12) + entries * 4,
                    flops=case["queries"] * 2.0 * (4 * 64 * 64 + 3 * 64))
    px = case["width"] * case["height"]
    return dict(bytes=px * (44 + 12 + 12), flops=px * 2.0 * BMFR_COLUMNS * (BMFR_COLUMNS + 3) * 2)


# ---------------------------------------------------------------------------------- 64-bit values

def _exact_query(case, seed):
    w, grid = _nrc_params(seed)
    rec = torch.from_numpy(_records(seed, case["queries"])).cuda().double()
    w = [torch.from_numpy(m).cuda().double() for m in w]
    grid = torch.from_numpy(grid).cuda()
    table = 1 << NRC_LOG2_TABLE
    growth = math.exp((math.log(NRC_FINEST) - math.log(NRC_BASE)) / (NRC_LEVELS - 1))
    n = case["queries"]
    x = torch.zeros(n, NRC_WIDTH, dtype=torch.float64, device="cuda")
    for lv in range(NRC_LEVELS):
        res = int(math.floor(NRC_BASE * growth ** lv))
        p = rec[:, 0:3] * res
        cell = p.floor().clamp(0, res - 1)
        fr = p - cell
        cell = cell.long()
        for c in range(8):
            off = [(c >> a) & 1 for a in range(3)]
            wt = torch.ones(n, dtype=torch.float64, device="cuda")
            for a in range(3):
                wt = wt * (fr[:, a] if off[a] else 1.0 - fr[:, a])
            q = [cell[:, a] + off[a] for a in range(3)]
            if (res + 1) ** 3 <= table:
                idx = q[0] + (res + 1) * (q[1] + (res + 1) * q[2])
            else:
                idx = ((q[0] * NRC_PRIMES[0]) ^ (q[1] * NRC_PRIMES[1]) ^ (q[2] * NRC_PRIMES[2])) & (table - 1)
            x[:, 2 * lv:2 * lv + 2] += wt[:, None] * grid[lv][idx].double()
    x[:, 32:35], x[:, 35:38], x[:, 38], x[:, 39] = rec[:, 3:6], rec[:, 6:9], rec[:, 9], 1.0
    for m in w[:4]:
        x = (x @ m.T).clamp(min=0.0)
    return (x @ w[4].T)[:, :3]


def _exact_denoise(case, seed):
    """Least squares per block in 64 bits: columns 1, n, q, q^2 scaled to the block, near-constant
    features and dependent columns left out, colour over (albedo + 0.01)."""
    color, feats = (torch.from_numpy(a).cuda().double() for a in _gbuffer(case, seed))
    b, (h, w) = case["block"], color.shape[:2]
    nby, nbx = (h + b - 1) // b, (w + b - 1) // b

    def blocks(t):
        full = torch.zeros(nby * b, nbx * b, t.shape[2], dtype=torch.float64, device=t.device)
        full[:h, :w] = t
        return full.view(nby, b, nbx, b, -1).permute(0, 2, 1, 3, 4).reshape(nby * nbx, b * b, -1)

    f, c = blocks(feats), blocks(color)
    take = (f[:, :, 3] >= 1.0)
    cols = [take.double()]
    feature = torch.cat([f[:, :, 0:3], f[:, :, 4:7]], 2)
    big = torch.full_like(feature, math.inf)
    lo = torch.where(take[..., None], feature, big).amin(1, keepdim=True)
    hi = torch.where(take[..., None], feature, -big).amax(1, keepdim=True)
    some = take.any(1)[:, None, None]
    lo, hi = torch.where(some, lo, torch.zeros_like(lo)), torch.where(some, hi, torch.zeros_like(hi))
    use = (hi - lo) > 1e-4 * torch.maximum(torch.maximum(lo.abs(), hi.abs()), torch.full_like(lo, 1e-2))
    q = torch.where(use & take[..., None], 2.0 * (feature - lo) / torch.where(use, hi - lo, torch.ones_like(lo)) - 1.0,
                    torch.zeros_like(feature))
    cols += [q[:, :, i] for i in range(6)] + [q[:, :, i] ** 2 for i in range(3, 6)]
    albedo = f[:, :, 8:11] + 0.01
    rhs = torch.where(take[..., None], c / albedo, torch.zeros_like(c))
    fit, basis = torch.zeros_like(rhs), []
    for col in cols:
        r = col.clone()
        for _ in range(2):
            for e in basis:
                r = r - e * (e * r).sum(1, keepdim=True)
        n, n0 = r.norm(dim=1, keepdim=True), col.norm(dim=1, keepdim=True)
        e = torch.where((n > 1e-3 * n0) & (n > 0), r / n.clamp(min=1e-300), torch.zeros_like(r))
        basis.append(e)
        fit = fit + e[..., None] * (e[..., None] * rhs).sum(1, keepdim=True)
    out = torch.where(take[..., None], fit * albedo, c)
    return out.view(nby, nbx, b, b, 3).permute(0, 2, 1, 3, 4).reshape(nby * b, nbx * b, 3)[:h, :w].contiguous()


def exact(case, seed):
    if case["kind"] == "query":
        return _exact_query(case, seed)
    if case["kind"] == "denoise":
        return _exact_denoise(case, seed)
    # pictures are sums over random paths, training follows its own rounding: no closed value
    return None
