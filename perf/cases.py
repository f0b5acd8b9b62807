"""Measured cases of the perceptual-rasterization library: what a program that
links it does, through the Python binding's public entry points.

    listed()            the cases, dicts of plain values
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs and handles a program has in hand before the call
    run(state)          one pass through the public entry points, and its outputs
    work(case)          bytes and operations the pass cannot do without
    exact(case, seed)   the outputs in 64 bits by plain torch, where that is affordable

A case's sizes follow from its own fields alone (``layout`` seeds how many
objects of which kind a scene has, and the sizes and modes of a batch's
views); ``seed`` makes the values: placements, motions, colours, poses,
foveas, targets and images.  Scenes are those of ``scenes.py`` in kind and
range (icosphere and box instances, objects over a ground plane, loose
triangles), built on the device.
"""
from __future__ import annotations

import functools
import math
import random

import numpy as np
import torch

from paper_1806_05385_gb300 import binding as B
from paper_1806_05385_gb300 import foveation as F
from paper_1806_05385_gb300 import scenes as S
from paper_1806_05385_gb300.autograd import Renderer

D = math.sqrt(2.0)
CLASSIC, ROLLING, FOVEATED, JOINT, MIXED = 0, 1, 2, 3, -1


# ------------------------------------------------------------------ the cases

def _case(kind, **kw):
    c = dict(kind=kind, scene="instances", views=1, t_lo=1000, t_hi=1000, w=0, h=0, side_lo=512, side_hi=512,
             mode=JOINT, stereo=False, fp64=0, lens=False, specular=False, display="none", zoom=1.0, layout=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest frame: 256 x 256, 1,000 loose triangles, rolling scan; one call per stage, each waited for
        _case("plain", name="plain_256", scene="triangles", t_lo=1000, t_hi=1000, w=256, h=256, mode=ROLLING),
        # an optimisation step written in PyTorch: loss.backward() through the autograd function, 10k small triangles
        _case("autograd", name="autograd_512", scene="small_triangles", t_lo=10_000, t_hi=10_000, w=512, h=512),
        # a frame loop that may not allocate: one eye of a ragged size in the library's fixed scratch array
        _case("noalloc", name="noalloc_eye", scene="objects", t_lo=61_200, t_hi=61_200, w=1001, h=953),
        # a headset's frame: both eyes rendered and turned into their display images, poses new with every frame
        _case("render", name="headset_frame", scene="objects", t_lo=266_000, t_hi=266_000, w=1440, h=1600, stereo=True,
              views=2, display="mip"),
        # one eye behind a lens: sampled p, rolling highlight, odd size, the 5x5 display filter
        _case("render", name="lens_eye", scene="objects", t_lo=51_200, t_hi=51_200, w=1213, h=1353, lens=True,
              specular=True, display="projected"),
        # images of many unlike scenes and modes in one eager call
        _case("render", name="render_8_mixed", views=8, t_lo=1000, t_hi=500_000, side_lo=512, side_hi=2160, mode=MIXED,
              layout=8),
        # a training step of a headset's frame (captured graph, loss against 8-bit images)
        _case("train", name="train_headset", scene="objects", t_lo=266_000, t_hi=266_000, w=1440, h=1600, stereo=True,
              views=2),
        # a training step of a large frame in the precision form
        _case("train", name="train_large_fp64", t_lo=1_000_000, t_hi=1_000_000, w=2160, h=2160, stereo=True, views=2,
              fp64=1, layout=3),
        # the largest: a training step over 64 views of 64 scenes, every mode, 1k to 500k triangles
        _case("train", name="train_64_views", views=64, t_lo=1000, t_hi=500_000, side_lo=512, side_hi=2160, mode=MIXED,
              layout=4),
        # the adjoint on its own: upstream image gradients of several rendered views
        _case("backward", name="backward_4", views=4, t_lo=5000, t_hi=100_000, side_lo=640, side_hi=1440, mode=MIXED,
              layout=6),
        # the display step alone, many views in one call
        _case("display", name="display_mip_16", views=16, side_lo=512, side_hi=2160, mode=MIXED, display="mip", layout=7),
        # ... and its higher-quality filter on one eye, for a display of more pixels than the frame has
        _case("display", name="display_projected_eye", w=1440, h=1600, display="projected", zoom=1.25),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain", "autograd", "noalloc", "render", "render", "train", "train", "backward", "display"])
    scene = rng.choice(["instances", "objects", "small_triangles"])
    mode = rng.choice([CLASSIC, ROLLING, FOVEATED, JOINT, JOINT])
    c = _case(kind, scene=scene, mode=mode, layout=rng.randrange(1, 1 << 20))
    w = _log(rng, 96, 2160)
    h = max(64, min(2160, int(w * rng.uniform(0.7, 1.4))))
    t = _log(rng, 500, 400_000)
    many = kind in ("render", "train", "backward", "display") and rng.random() < 0.5
    if many:
        n = _log(rng, 2, 24)
        lo = _log(rng, 96, 700)
        t_lo = _log(rng, 500, 5000)
        c.update(views=n, side_lo=lo, side_hi=_log(rng, lo, 2160), t_lo=t_lo, t_hi=_log(rng, t_lo, 200_000),
                 mode=MIXED)
    else:
        c.update(w=w, h=h, t_lo=t, t_hi=t)
        if kind in ("render", "train") and rng.random() < 0.4:
            c.update(stereo=True, views=2)
    if kind == "noalloc":
        t = _log(rng, 500, 60_000)
        c.update(w=min(w, 1100), h=min(h, 1100), t_lo=t, t_hi=t, scene="objects")
    if kind in ("render", "train"):
        c.update(fp64=int(rng.random() < 0.25), specular=rng.random() < 0.25)
    if kind == "render":
        c.update(display=rng.choice(["none", "mip", "projected"]), lens=rng.random() < 0.25)
    if kind == "display":
        c.update(display=rng.choice(["mip", "projected"]), zoom=round(rng.uniform(0.6, 1.4), 3))
    return c


# ------------------------------------------------- sizes (the case's fields alone)

def _views(case):
    """(W, H, T, mode, scene index) of every view, and the scenes' T."""
    if case["w"]:
        n = case["views"]
        return [(case["w"], case["h"], case["t_lo"], case["mode"], 0)] * n, [case["t_lo"]]
    r = random.Random(case["layout"])
    out = []
    for k in range(case["views"]):
        side = _log(r, case["side_lo"], case["side_hi"])
        mode = r.randrange(4) if case["mode"] == MIXED else case["mode"]
        out.append((side, side, _log(r, case["t_lo"], case["t_hi"]), mode, k))
    return out, [v[2] for v in out]


_MESHES = {"ico3": lambda: S.icosphere(3), "ico2": lambda: S.icosphere(2), "box": S.unit_box,
           "ground": lambda: S.ground_plane(70, 71, 1.6, (-20.0, 20.0), (0.5, 40.5))}


@functools.lru_cache(maxsize=None)
def _mesh(name):
    v, f = _MESHES[name]()
    return v.astype(np.float32), f.astype(np.int32)


@functools.lru_cache(maxsize=256)
def _topology(scene, T, layout):
    """The scene's objects before placement: unit vertices [V, 3], the object
    of every vertex, the triangles (CPU tensors) and the objects' kinds."""
    if scene in ("triangles", "small_triangles"):
        return None, None, torch.arange(3 * T, dtype=torch.int32).view(T, 3), ()
    r = random.Random(layout * 7919 + T)
    kinds, total = [], 0
    ground = scene == "objects" and T > 20_000
    want = T - (_mesh("ground")[1].shape[0] if ground else 0)
    while total < want:
        kinds.append("ico3" if scene == "objects" else r.choice(("ico2", "box")))
        total += _mesh(kinds[-1])[1].shape[0]
    base, unit, owner, tri = 0, [], [], []
    left = want
    for k, name in enumerate(kinds):
        v, f = _mesh(name)
        unit.append(v)
        owner.append(np.full(v.shape[0], k, np.int64))
        tri.append(f[:left] + np.int32(base))
        left -= f.shape[0]
        base += v.shape[0]
    if ground:
        v, f = _mesh("ground")
        unit.append(v)
        owner.append(np.full(v.shape[0], len(kinds), np.int64))
        tri.append(f + np.int32(base))
    return (torch.from_numpy(np.concatenate(unit)), torch.from_numpy(np.concatenate(owner)),
            torch.from_numpy(np.concatenate(tri)), tuple(kinds) + (("ground",) if ground else ()))


def _vertices(scene, T, layout):
    unit = _topology(scene, T, layout)[0]
    return 3 * T if unit is None else unit.shape[0]


# ------------------------------------------------------------- inputs by seed

def _scene(case, T, k, seed, tan_x, tan_y):
    """Device arrays (pos, vel, col [V, 3] f32, tri [T, 3] i32) of scene k."""
    rng = np.random.default_rng([seed, k, 11])
    gen = torch.Generator(device="cuda").manual_seed(seed * 1009 + k)
    unit, owner, tri, kinds = _topology(case["scene"], T, case["layout"] + k)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")
    if unit is None:
        lo, hi = dev([-1.0, -1.0, 2.0]), dev([1.0, 1.0, 10.0])
        rand = lambda *s: torch.rand(*s, generator=gen, device="cuda")
        if case["scene"] == "triangles":
            pos = lo + (hi - lo) * rand(3 * T, 3)
        else:
            pos = (lo + (hi - lo) * rand(T, 3)).repeat_interleave(3, 0) + 0.3 * (rand(3 * T, 3) - 0.5)
        vel = 0.05 * torch.randn(3 * T, 3, generator=gen, device="cuda")
        return pos.contiguous(), vel, rand(3 * T, 3), tri.cuda()
    n = len(kinds)
    if case["scene"] == "objects":
        r, moving = rng.uniform(0.2, 1.5, n), np.ones(n)
    else:
        r, moving = np.exp(rng.uniform(math.log(0.005), 0.0, n)), (rng.uniform(size=n) < 0.5) * 1.0
    bound = r * np.array([math.sqrt(3.0) if m == "box" else 1.0 for m in kinds])
    z = rng.uniform(1.0 + bound, 30.0)
    centre = np.stack([rng.uniform(-1, 1, n) * z * tan_x, rng.uniform(-1, 1, n) * z * tan_y, z], 1)
    way = rng.normal(size=(n, 3))
    vel = way / np.linalg.norm(way, axis=1, keepdims=True) * (rng.uniform(0.0, 0.3, n) * moving)[:, None]
    if kinds and kinds[-1] == "ground":
        r[-1], centre[-1], vel[-1] = 1.0, 0.0, 0.0
    own = owner.cuda()
    pos = unit.cuda() * dev(r)[own, None] + dev(centre)[own]
    col = torch.rand(pos.shape[0], 3, generator=gen, device="cuda")
    return pos.contiguous(), dev(vel)[own].contiguous(), col, tri.cuda()


def _scene_views(case, seed):
    """The scenes' view objects (fields of scenes.View)."""
    rng = np.random.default_rng([seed, 5])
    sizes, _ = _views(case)
    out = []
    for k, (W, H, _, mode, _) in enumerate(sizes):
        loose = case["scene"] in ("triangles", "small_triangles")
        tx, ty = (0.5, 0.5 * H / W) if loose else S.hmd_fov(W, H, 100.0 if case["stereo"] else 90.0)
        if case["stereo"]:
            p0, p1 = S.head_poses(3.0, 1.0, (-0.032, 0.032)[k])
        else:
            p0, p1 = S.head_poses(rng.uniform(0.0, 3.0), rng.uniform(0.0, 1.0))
        v = S.View(W=W, H=H, tan_x=tx, tan_y=ty, pose0=p0, pose1=p1, mode=mode,
                   fovea=tuple(float(np.float32(x)) for x in rng.uniform(0.2, 0.8, size=2)), alpha=2.0)
        if case["specular"]:
            v.k_s, v.shininess = 0.25, 32.0
        if case["lens"]:
            v.p_lut = F.lens_samples(2.0)
        out.append(v)
    return out


def _scene_arrays(case, seed, views):
    sizes, ts = _views(case)
    first = {}
    for v, s in zip(views, sizes):
        first.setdefault(s[4], v)
    return [_scene(case, T, k, seed, first[k].tan_x, first[k].tan_y) for k, T in enumerate(ts)]


def _image(gen, H, W):
    """A rendered-looking planar image: smooth patches, hard edges, a background of zeros."""
    def up(c, n, mode):
        x = torch.rand(1, c, max(2, H // n), max(2, W // n), generator=gen, device="cuda")
        return torch.nn.functional.interpolate(x, size=(H, W), mode=mode)[0]
    return (up(3, 24, "bilinear") * (up(1, 40, "nearest") > 0.4)).contiguous()


_stream = None


def _use_stream():
    # graphs are captured on a stream of the program's own; every call and torch operation then follows on it
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    torch.cuda.set_stream(_stream)


class State:
    """Inputs, output buffers and handles of one case; frees its handles."""

    def __init__(self):
        self.graph = self.ws = self.disp_ws = self.renderer = None
        self.scenes = []

    def __del__(self):
        try:
            if self.graph:
                B.pr_graph_free(self.graph)
            for w in (self.ws, self.disp_ws):
                if w:
                    B.pr_workspace_free(w)
            for h in self.scenes:
                B.pr_scene_free(h)
            if self.renderer is not None:
                self.renderer.close()
        except Exception:  # interpreter shutdown
            pass


def _split(flat, counts):
    return list(torch.split(flat, counts))


def _cortical(v):
    """The view of the display step: behind a lens it samples back with the power map alone."""
    return S.View(**{**v.__dict__, "p_lut": None}) if v.p_lut is not None else v


def prepare(case, seed):
    _use_stream()
    s = State()
    s.case = case
    s.views = _scene_views(case, seed)
    s.pviews = [B.make_view(v) for v in s.views]
    px = [v.W * v.H for v in s.views]
    f32 = lambda n: torch.empty(n, dtype=torch.float32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(seed * 31 + 7)
    if case["display"] != "none":
        s.dsize = [(max(1, round(v.W * case["zoom"])), max(1, round(v.H * case["zoom"]))) for v in s.views]
        s.dviews = [B.make_view(_cortical(v)) for v in s.views]
        s.dflat = f32(3 * sum(a * b for a, b in s.dsize))
        s.dout = _split(s.dflat, [3 * a * b for a, b in s.dsize])
        s.disp_ws = B.pr_workspace_create()
    if case["kind"] == "display":
        s.rgb = [_image(gen, v.H, v.W) for v in s.views]
        s.disp = [(v, r, o, *d) for v, r, o, d in zip(s.dviews, s.rgb, s.dout, s.dsize)]
        return s
    s.arrays = _scene_arrays(case, seed, s.views)
    s.params = B.make_params(fp64_retest=case["fp64"])
    if case["kind"] == "autograd":
        pos, vel, col, tri = s.arrays[0]
        s.renderer = Renderer(tri, pos.shape[0], s.views[0], s.params)
        s.leaves = [x.clone().requires_grad_(True) for x in (col, pos, vel)]
        s.target = torch.rand(3, s.views[0].H, s.views[0].W, generator=gen, device="cuda")
        return s
    s.ids = torch.empty(sum(px), dtype=torch.int32, device="cuda")
    s.depth = f32(sum(px))
    if case["kind"] == "noalloc":
        return s
    s.scenes = [B.pr_scene_upload(*a) for a in s.arrays]
    s.rgb = f32(3 * sum(px))
    s.ws = B.pr_workspace_create()
    of = [v[4] for v in _views(case)[0]]
    ids, rgb = _split(s.ids, px), _split(s.rgb, [3 * n for n in px])
    s.entries = [(s.scenes[q], v, i, d, c) for q, v, i, d, c in zip(of, s.pviews, ids, _split(s.depth, px), rgb)]
    if case["display"] != "none":
        s.disp = [(v, r, o, *d) for v, r, o, d in zip(s.dviews, rgb, s.dout, s.dsize)]
    nv = [a[0].shape[0] for a in s.arrays]
    if case["kind"] in ("train", "backward"):
        s.grads = f32(9 * sum(nv))
        parts = [g.view(3, -1, 3) for g in _split(s.grads, [9 * n for n in nv])]
    if case["kind"] == "train":
        s.loss = f32(len(px))
        s.targets = torch.randint(0, 256, (3 * sum(px),), generator=gen, device="cuda", dtype=torch.uint8)
        s.frame_grads = [dict(target_u8=t, loss=s.loss[k:k + 1], dcol=parts[q][0], dpos=parts[q][1], dvel=parts[q][2])
                         for k, (q, t) in enumerate(zip(of, _split(s.targets, [3 * n for n in px])))]
        s.graph = B.pr_graph_capture_frame(s.ws, s.entries, s.frame_grads, s.params)
        s.update = [[a[j] for a in s.arrays] for j in range(3)]
    if case["kind"] == "backward":
        B.pr_rasterize_batch(s.ws, s.entries, s.params)  # the frame whose gradients are wanted
        s.upstream = torch.randn(3 * sum(px), generator=gen, device="cuda")
        s.back = [(s.scenes[q], v, i, g, *parts[q])
                  for q, v, i, g in zip(of, s.pviews, ids, _split(s.upstream, [3 * n for n in px]))]
    return s


# ------------------------------------------------------------------- one pass

def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "train":
        # the optimiser's parameters into the scenes, fresh gradients, the frame
        B.pr_scene_update_batch(s.scenes, *s.update)
        s.grads.zero_()
        s.loss.zero_()
        B.pr_graph_launch(s.graph)
        return {"loss": s.loss, "grads": s.grads, "ids": s.ids, "depth": s.depth, "rgb": s.rgb}
    if kind == "render":
        B.pr_rasterize_batch(s.ws, s.entries, s.params)
        out = {"ids": s.ids, "depth": s.depth, "rgb": s.rgb}
        if case["display"] != "none":
            B.pr_unfoveate_batch(s.disp_ws, s.disp, case["display"], 0.5)
            out["display"] = s.dflat
        return out
    if kind == "plain":
        B.pr_rasterize(s.scenes[0], s.pviews[0], s.params, s.ids, s.depth)
        B.pr_shade(s.scenes[0], s.pviews[0], s.ids, s.rgb)
        return {"ids": s.ids, "depth": s.depth, "rgb": s.rgb}
    if kind == "noalloc":
        B.pr_rasterize_noalloc(*s.arrays[0], s.pviews[0], s.params, s.ids, s.depth)
        return {"ids": s.ids, "depth": s.depth}
    if kind == "autograd":
        for x in s.leaves:
            x.grad = None
        rgb = s.renderer.render(*s.leaves)
        loss = ((rgb - s.target) ** 2).sum()
        loss.backward()
        return {"loss": loss.detach(), "rgb": rgb.detach(), "grads": [x.grad for x in s.leaves]}
    if kind == "backward":
        s.grads.zero_()
        B.pr_backward_batch(s.ws, s.back)
        return {"grads": s.grads}
    B.pr_unfoveate_batch(s.disp_ws, s.disp, case["display"], 0.5)
    return {"display": s.dflat}


# ----------------------------------------------------------------------- work

# operations per pixel that no form of the method goes without: one watertight
# test (39), the pixel's ray, barycentrics, normal, light and colour (about
# 100), and their adjoint (about 150); the display filters' taps (3 channels)
_TEST, _SHADE, _ADJOINT = 39, 100, 150
_TAPS = {"none": 0, "mip": 2 * 9 * 6, "projected": 25 * (6 + 8)}


def work(case):
    sizes, ts = _views(case)
    px = sum(W * H for W, H, *_ in sizes)
    verts = sum(_vertices(case["scene"], T, case["layout"] + k) for k, T in enumerate(ts))
    shown = sum(max(1, round(W * case["zoom"])) * max(1, round(H * case["zoom"])) for W, H, *_ in sizes)
    kind, mesh = case["kind"], 36 * verts + 12 * sum(ts)
    disp = case["display"]
    byts = {"train": mesh + 3 * px + 20 * px + 36 * verts, "render": mesh + 20 * px, "plain": mesh + 20 * px,
            "noalloc": mesh + 8 * px, "autograd": mesh + 24 * px + 36 * verts, "backward": mesh + 16 * px + 36 * verts,
            "display": 12 * px}[kind]
    flops = px * {"train": _TEST + _SHADE + _ADJOINT, "render": _TEST + _SHADE, "plain": _TEST + _SHADE,
                  "noalloc": _TEST, "autograd": _TEST + _SHADE + _ADJOINT, "backward": _SHADE + _ADJOINT,
                  "display": 0}[kind]
    if disp != "none":
        byts += 12 * shown
        flops += _TAPS[disp] * shown
    return {"bytes": byts, "flops": flops}


# -------------------------------------------------------------------- 64 bits

_MOST_PAIRS = 1.2e10  # pixel-triangle pairs that the brute-force search below takes on


def _f64(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float32), device="cuda").double()


class _View64:
    """A view's pixels in 64 bits: time, ray direction, light (conventions of pr.h)."""

    def __init__(self, v):
        self.v = v
        i = (torch.arange(v.W, device="cuda", dtype=torch.float64) + 0.5) / v.W
        j = (torch.arange(v.H, device="cuda", dtype=torch.float64) + 0.5) / v.H
        x = torch.stack([i.repeat(v.H), j.repeat_interleave(v.W)], 1)
        if v.mode in (FOVEATED, JOINT):
            f = _f64(v.fovea)
            e = x - f
            r = e.norm(dim=1, keepdim=True)
            if v.p_lut is not None:
                p = _f64(v.p_lut)
                n = p.numel() - 1
                at = r * n / D
                k = at.floor().long().clamp(0, n - 1)
                scale = (p[k] + (at - k) * (p[k + 1] - p[k])) / r.clamp_min(1e-300)
            else:
                scale = (r / D) ** (v.alpha - 1.0)
            x = f + e * torch.where(r > 0, scale, torch.zeros_like(scale))
        rolling = v.mode in (ROLLING, JOINT)
        self.t = x @ _f64(v.d) if rolling else torch.zeros_like(x[:, 0])
        tan = _f64([v.tan_x, v.tan_y])
        self.dir = torch.cat([(2 * x - 1) * tan, torch.ones_like(x[:, :1])], 1)
        self.R0, self.R1 = _f64(v.pose0)[:3, :3], _f64(v.pose1)[:3, :3]
        self.T0, self.T1 = _f64(v.pose0)[:3, 3], _f64(v.pose1)[:3, 3]

    def ends(self, pos, vel):
        """Camera-space vertices at t = 0 and their motion over the frame."""
        s = pos @ self.R0.T + self.T0
        return s, (pos + vel) @ self.R1.T + self.T1 - s

    def visible(self, pos, vel, tri):
        """Nearest triangle of every pixel (-1: none) and its depth, every pair tried.

        With w_0 = d . (B x C) (cyclically) the hit's barycentrics are w_k / sum w and its depth is
        A . (B x C) / sum w; the moved triangle makes them polynomials in t."""
        s, m = self.ends(pos, vel)
        s, m = s[tri], m[tri]
        cr = lambda a, b: torch.linalg.cross(a, b, dim=-1)
        coef = []
        for k in range(3):
            b, c = (k + 1) % 3, (k + 2) % 3
            sb, sc, mb, mc = s[:, b], s[:, c], m[:, b], m[:, c]
            coef.append(torch.cat([cr(sb, sc), cr(sb, mc) + cr(mb, sc), cr(mb, mc)], 1))
        dot = lambda a, b: (a * b).sum(1)
        a0, a1, (c0, c1, c2) = s[:, 0], m[:, 0], coef[0].split(3, 1)
        vol = torch.stack([dot(a0, c0), dot(a0, c1) + dot(a1, c0), dot(a0, c2) + dot(a1, c1), dot(a1, c2)], 1)
        n, T = self.t.numel(), tri.shape[0]
        ids = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        depth = torch.full((n,), math.inf, dtype=torch.float64, device="cuda")
        if T == 0:
            return ids, depth
        step = max(1, int(2.5e7 // T))
        for p in range(0, n, step):
            t, d = self.t[p:p + step, None], self.dir[p:p + step]
            f = torch.cat([d, t * d, t * t * d], 1)
            w0, w1, w2 = (f @ c.T for c in coef)
            z = torch.cat([torch.ones_like(t), t, t * t, t ** 3], 1) @ vol.T
            lo, hi = torch.minimum(torch.minimum(w0, w1), w2), torch.maximum(torch.maximum(w0, w1), w2)
            w0.add_(w1).add_(w2)
            z.div_(w0)
            z.masked_fill_(((lo < 0) & (hi > 0)) | (w0 == 0) | ~(z > self.v.z_near), math.inf)
            best, at = z.min(1)
            depth[p:p + step] = best
            ids[p:p + step] = torch.where(best < math.inf, at, -1)
        return ids, depth

    def shade(self, pos, vel, col, tri, ids):
        """Colours [3, H * W] of the pixels whose visible triangle is ids (differentiable)."""
        v = self.v
        on = (ids >= 0).nonzero()[:, 0]
        t, d, vi = self.t[on, None], self.dir[on], tri[ids[on]]
        s, m = self.ends(pos, vel)
        A, Bv, C = (s[vi[:, k]] + t * m[vi[:, k]] for k in range(3))
        cr = lambda a, b: torch.linalg.cross(a, b, dim=-1)
        dot = lambda a, b: (a * b).sum(1, keepdim=True)
        w = torch.cat([dot(d, cr(Bv, C)), dot(d, cr(C, A)), dot(d, cr(A, Bv))], 1)
        b = w / w.sum(1, keepdim=True)
        albedo = sum(b[:, k:k + 1] * col[vi[:, k]] for k in range(3))
        n = cr(Bv - A, C - A)
        n = torch.where(dot(n, d) > 0, -n, n)
        n = n / n.norm(dim=1, keepdim=True).clamp_min(1e-300)
        lw = _f64(v.light_w)
        lw = lw / lw.norm()
        li = (1 - t) * (self.R0 @ lw) + t * (self.R1 @ lw)
        li = li / li.norm(dim=1, keepdim=True)
        rgb = albedo * (float(np.float32(v.k_a)) + float(np.float32(v.k_d)) * dot(n, li).clamp_min(0))
        if v.k_s > 0:
            hv = li - d / d.norm(dim=1, keepdim=True)
            ndh = dot(n, hv / hv.norm(dim=1, keepdim=True))
            rgb = rgb + v.k_s * torch.where(ndh > 0, ndh.clamp_min(1e-12) ** v.shininess, torch.zeros_like(ndh))
        out = torch.zeros(ids.numel(), 3, dtype=torch.float64, device="cuda")
        return out.index_copy(0, on, rgb).T


def _display64(v, rgb, Wd, Hd, method):
    """The display image [3, Hd, Wd] of a framebuffer image [3, H, W] in 64 bits."""
    x = torch.stack([((torch.arange(Wd, device="cuda").double() + 0.5) / Wd).repeat(Hd),
                     ((torch.arange(Hd, device="cuda").double() + 0.5) / Hd).repeat_interleave(Wd)], 1)
    W, H = v.W, v.H
    u, stretch = x, torch.ones_like(x[:, 0])
    f = _f64(v.fovea)
    fov = v.mode in (FOVEATED, JOINT)
    if fov:
        e = x - f
        r = e.norm(dim=1)
        stretch = (r / D) ** (1.0 / v.alpha - 1.0)
        u = f + e * torch.where(r > 0, stretch, torch.zeros_like(r))[:, None]
    if method == "mip":
        levels = [rgb.double()]
        while levels[-1].shape[1] > 1 or levels[-1].shape[2] > 1:
            a = levels[-1]
            pad = (0, a.shape[2] % 2, 0, a.shape[1] % 2)
            ones = torch.nn.functional.pad(torch.ones_like(a[:1]), pad)
            a = torch.nn.functional.pad(a, pad)
            quad = lambda y: y[:, 0::2, 0::2] + y[:, 0::2, 1::2] + y[:, 1::2, 0::2] + y[:, 1::2, 1::2]
            levels.append(quad(a) / quad(ones))
        lod = torch.log2(stretch * max(W / Wd, H / Hd)).clamp(0, len(levels) - 1)

        def bspline(y):
            y = y.abs()
            return torch.where(y < 1, 2 / 3 - y * y + y ** 3 / 2, torch.where(y < 2, (2 - y) ** 3 / 6, 0 * y))

        out = torch.zeros(3, Wd * Hd, dtype=torch.float64, device="cuda")
        for k, lev in enumerate(levels):
            weight = (1 - (lod - k).abs()).clamp_min(0)
            on = (weight > 0).nonzero()[:, 0]
            if not on.numel():
                continue
            h, w = lev.shape[1:]
            sx, sy = u[on, 0] * w - 0.5, u[on, 1] * h - 0.5
            cx, cy = (sx + 0.5).floor(), (sy + 0.5).floor()
            acc, norm = 0, 0
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    g = bspline(sx - cx - dx) * bspline(sy - cy - dy)
                    at = (cy + dy).long().clamp(0, h - 1) * w + (cx + dx).long().clamp(0, w - 1)
                    acc, norm = acc + g * lev.reshape(3, -1)[:, at], norm + g
            out[:, on] += weight[on] * acc / norm
        return out
    i = (u[:, 0] * W).floor().long().clamp(0, W - 1)
    j = (u[:, 1] * H).floor().long().clamp(0, H - 1)
    size = torch.tensor([Wd, Hd], device="cuda").double()

    def taps():
        for dy in range(-2, 3):
            for dx in range(-2, 3):
                pi, pj = i + dx, j + dy
                ok = (pi >= 0) & (pi < W) & (pj >= 0) & (pj < H)
                c = torch.stack([(pi + 0.5) / W, (pj + 0.5) / H], 1)
                if fov:
                    e = c - f
                    r = e.norm(dim=1, keepdim=True)
                    c = f + e * torch.where(r > 0, (r / D) ** (v.alpha - 1.0), torch.zeros_like(r))
                d2 = (((x - c) * size) ** 2).sum(1)
                yield (pj.clamp(0, H - 1) * W + pi.clamp(0, W - 1)), torch.where(ok, d2, math.inf)

    near = None
    for _, d2 in taps():
        near = d2 if near is None else torch.minimum(near, d2)
    acc, norm, flat = 0, 0, rgb.double().reshape(3, -1)
    for at, d2 in taps():
        g = torch.exp(-(d2 - near) / (2 * 0.5 * 0.5))
        acc, norm = acc + g * flat[:, at], norm + g
    return acc / norm


def exact(case, seed):
    kind = case["kind"]
    sizes, ts = _views(case)
    of = [z[4] for z in sizes]
    if kind == "display":
        if case["display"] == "mip" and sum(W * H for W, H, *_ in sizes) > 6e7:
            return None
        s = prepare(case, seed)
        return {"display": torch.cat([_display64(v, r, *d, case["display"]).reshape(-1)
                                      for v, r, d in zip(s.views, s.rgb, s.dsize)])}
    pairs = sum(W * H * T for W, H, T, _, _ in sizes)
    if kind != "backward" and pairs > _MOST_PAIRS:
        return None
    s = prepare(case, seed)
    arrays = [tuple(x.double() for x in a[:3]) + (a[3].long(),) for a in s.arrays]
    views = [_View64(v) for v in s.views]
    train = kind in ("train", "autograd", "backward")
    if train:
        for a in arrays:
            for x in a[:3]:
                x.requires_grad_(True)
    split = lambda flat: [x.view(3, -1) for x in _split(flat, [3 * v.W * v.H for v in s.views])]
    losses, depths, images = [], [], []
    if kind == "backward":  # the visible triangles are an input of the adjoint
        ids_in = [x.long() for x in _split(s.ids, [v.W * v.H for v in s.views])]
        up = split(s.upstream)
    for k, (q, w) in enumerate(zip(of, views)):
        pos, vel, col, tri = arrays[q]
        if kind == "backward":
            ids = ids_in[k]
        else:
            with torch.no_grad():
                ids, depth = w.visible(pos, vel, tri)
            depths.append(depth)
            if kind == "noalloc":
                continue
        rgb = w.shade(pos, vel, col, tri, ids)
        if train:
            if kind == "backward":
                loss = (rgb * up[k]).sum()
            else:
                target = split(s.targets)[k].double() / 255 if kind == "train" else s.target.double().view(3, -1)
                loss = ((rgb - target) ** 2).sum()
            loss.backward()
            losses.append(loss.detach())
        images.append(rgb.detach().reshape(-1))
    out = {"depth": torch.cat(depths)} if depths else {}
    if kind == "noalloc":
        return {**out, "ids": None}
    if train:
        zero = lambda x: x.grad if x.grad is not None else torch.zeros_like(x)
        grads = [torch.stack([zero(a[2]), zero(a[0]), zero(a[1])]) for a in arrays]
        if kind == "backward":
            return {"grads": torch.cat([g.reshape(-1) for g in grads])}
        if kind == "autograd":
            return {"loss": losses[0], "rgb": images[0].view(s.target.shape), "grads": list(grads[0])}
        return {**out, "ids": None, "rgb": torch.cat(images), "loss": torch.stack(losses),
                "grads": torch.cat([g.reshape(-1) for g in grads])}
    out.update(ids=None, rgb=torch.cat(images))
    if case["display"] != "none":  # of the frame's own image in 64 bits
        px = [3 * v.W * v.H for v in s.views]
        out["display"] = torch.cat([_display64(_cortical(v), r.view(3, v.H, v.W), *d, case["display"]).reshape(-1)
                                    for v, r, d in zip(s.views, _split(out["rgb"], px), s.dsize)])
    return out
