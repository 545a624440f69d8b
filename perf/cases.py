"""Performance cases of the hybrid depth-of-field framework.

Each case is work that a program built on the framework has it do, through
the public entry points of the binding (``Renderer``, ``Batch``,
``HdofPost`` and the single calls):

* ``frame``       consecutive frames of a shot after a cut (history reset);
* ``batch``       many views of several scenes, one launch per stage;
* ``fit``         a lens/colour fitting step: post-path forward and backward;
* ``postfilter``  the CoC post-filter alone (round or shaped bokeh);
* ``reconstruct`` temporal and spatial reconstruction, then the composite;
* ``bvh``         rebuild of a scene's acceleration structure, its G-buffer and ray queries;
* ``reference``   full ray-traced frame and the error map against an image.

``listed()`` holds the named cases, ``draw(rng)`` gives others of the same
ranges, ``prepare``/``run`` make a case's state and run one pass on it,
``work`` states the bytes and operations a pass cannot do without, and
``exact`` gives a pass's outputs in 64-bit arithmetic where that is in reach.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import hdof_inputs as hi
import paper_2210_04981_gb300.hdof as H

DEV = "cuda"


# ------------------------------------------------------------------ cases --

def listed():
    return [
        # the smallest frame (the two-quad scene at 128x128, 16 rays per edge
        # pixel): previews and thumbnails, bound by launches and latency
        dict(name="frame_tiny", kind="frame", scene="tiny", width=128, height=128, frames=4, spp=16, r_max=16.0,
             focus=2.0, aperture=0.05, variance=0, mixed=0, alpha_k=0.0, spec=0.0, mask_coc=0),
        # the headline: a moving camera through the 165k-triangle room at
        # 1080p, f/1.4 lens, FP32 planes
        dict(name="frame_1080p", kind="frame", scene="room", boxes=64, spheres=32, subdiv=4, width=1920, height=1080,
             frames=4, spp=8, r_max=32.0, focus=3.0, aperture=hi.ROOM_APERTURE, variance=1, mixed=0, alpha_k=0.0,
             spec=0.0, mask_coc=0),
        # an odd window size with a wide lens (rays of a pixel far apart),
        # glossy materials, per-pixel blend factors and the CoC-scaled mask
        dict(name="frame_wide_odd", kind="frame", scene="room", boxes=64, spheres=28, subdiv=4, width=1279, height=717,
             frames=2, spp=16, r_max=32.0, focus=1.5, aperture=0.06, variance=1, mixed=0, alpha_k=0.5, spec=2.0,
             mask_coc=1),
        # 4K with FP16/BF16 planes over the 5.25M-triangle scene: the largest frame
        dict(name="frame_4k_mixed", kind="frame", scene="room", boxes=512, spheres=256, subdiv=5, width=3840,
             height=2160, frames=2, spp=8, r_max=64.0, focus=3.0, aperture=hi.ROOM_APERTURE, variance=1, mixed=1,
             alpha_k=0.0, spec=0.0, mask_coc=0),
        # twelve views of four rooms (50k to 500k triangles), 256x256 to
        # 1080p, narrow and wide lenses, rendered together
        dict(name="batch_12", kind="batch", views=12, frames=2),
        # one step of fitting the lens and the colour image at 1024x1024
        dict(name="fit_1024", kind="fit", width=1024, height=1024, focus=2.0, aperture=0.03, tris=100_000),
        # the post-filter as a filter of its own at 1080p: near and far
        # surfaces at many depths
        dict(name="postfilter_1080p", kind="postfilter", width=1920, height=1080, focus=3.0, aperture=0.02, r_max=32.0,
             mixed=0, blades=0, aberration=0.0),
        # hexagonal bokeh with a bright rim at an odd size
        dict(name="postfilter_hexagon", kind="postfilter", width=1279, height=719, focus=2.0, aperture=0.02,
             r_max=24.0, mixed=0, blades=6, aberration=0.4),
        # reconstruction and composite of a heavily traced 1080p frame
        dict(name="reconstruct_1080p", kind="reconstruct", width=1920, height=1080, frac=0.5, alpha_k=0.0),
        # a dynamic scene: its structure rebuilt, its G-buffer, then picking rays
        dict(name="bvh_rebuild", kind="bvh", boxes=64, spheres=32, subdiv=4, rays=20_000, width=1280, height=720),
        # ground truth for quality work: every pixel ray traced, compared with an image
        dict(name="reference_720p", kind="reference", width=1280, height=720, spp=8, passes=4, focus=3.0,
             aperture=hi.ROOM_APERTURE),
    ]


def _log(rng, lo, hi_):
    return math.exp(rng.uniform(math.log(lo), math.log(hi_)))


def _size(rng, lo, hi_):
    """Width and height: area log-uniform between lo^2 and hi_^2, odd sizes as likely as even ones."""
    side, aspect = _log(rng, lo, hi_), rng.uniform(0.8, 1.9)
    w, h = int(side * math.sqrt(aspect)), int(side / math.sqrt(aspect))
    return max(w, 17), max(h, 17)


def draw(rng):
    kind = rng.choice(("frame", "frame", "frame", "batch", "fit", "postfilter", "postfilter", "reconstruct", "bvh",
                       "reference"))
    if kind == "frame":
        if rng.random() < 0.2:
            w, h = _size(rng, 40, 400)
            return dict(kind=kind, scene="tiny", width=w, height=h, frames=rng.choice((2, 4)),
                        spp=rng.choice((4, 7, 16)), r_max=rng.uniform(6, 24), focus=rng.uniform(1.0, 2.5),
                        aperture=rng.uniform(0.01, 0.08), variance=rng.choice((0, 1)), mixed=rng.choice((0, 1)),
                        alpha_k=rng.choice((0.0, 0.5)), spec=0.0, mask_coc=rng.choice((0, 1)))
        w, h = _size(rng, 200, 1500)
        return dict(kind=kind, scene="room", boxes=rng.randint(16, 96), spheres=rng.randint(8, 64),
                    subdiv=rng.choice((3, 4)), width=w, height=h, frames=2, spp=rng.choice((4, 8, 11, 16)),
                    r_max=rng.uniform(12, 48), focus=rng.uniform(0.8, 6.0), aperture=_log(rng, 0.004, 0.06),
                    variance=1, mixed=rng.choice((0, 0, 1)), alpha_k=rng.choice((0.0, 0.5)),
                    spec=rng.choice((0.0, 0.0, 2.0)), mask_coc=rng.choice((0, 1)))
    if kind == "batch":
        return dict(kind=kind, views=rng.randint(2, 10), frames=2)
    if kind == "fit":
        w, h = _size(rng, 100, 1000)
        return dict(kind=kind, width=w, height=h, focus=rng.uniform(1.2, 5.5), aperture=rng.uniform(0.01, 0.04),
                    tris=rng.randint(20_000, 150_000))
    if kind == "postfilter":
        w, h = _size(rng, 100, 1400)
        shaped = rng.random() < 0.4
        return dict(kind=kind, width=w, height=h, focus=rng.uniform(0.8, 5.0), aperture=_log(rng, 0.004, 0.04),
                    r_max=rng.uniform(6, 24 if shaped else 40), mixed=rng.choice((0, 1)),
                    blades=rng.choice((0, 5, 6, 8)) if shaped else 0,
                    aberration=rng.uniform(-0.5, 0.5) if shaped else 0.0)
    if kind == "reconstruct":
        w, h = _size(rng, 100, 1600)
        return dict(kind=kind, width=w, height=h, frac=rng.uniform(0.1, 0.9), alpha_k=rng.choice((0.0, 0.5)))
    if kind == "bvh":
        w, h = _size(rng, 100, 1000)
        return dict(kind=kind, boxes=rng.randint(1, 200), spheres=rng.randint(1, 60), subdiv=rng.choice((2, 3, 4)),
                    rays=int(_log(rng, 100, 20_000)), width=w, height=h)
    w, h = _size(rng, 100, 1000)
    return dict(kind=kind, width=w, height=h, spp=rng.choice((4, 8, 16)), passes=rng.randint(1, 4),
                focus=rng.uniform(1.0, 5.0), aperture=_log(rng, 0.004, 0.05))


# ------------------------------------------------------------ preparation --

def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _scene_of(case, seed):
    if case.get("scene") == "tiny":
        # the two quads, with an occluder whose depth follows the seed
        sc = hi.tiny_scene()
        v = sc.verts.copy()
        v[4:, 2] += np.float32(0.05 * np.random.default_rng(seed).uniform(-1, 1))
        return hi.Scene(v, sc.idx, sc.mat, sc.uv)
    return hi.room_scene(seed=seed, n_boxes=case["boxes"], n_spheres=case["spheres"], subdiv=case["subdiv"],
                         aspect=case.get("width", 16) / case.get("height", 9), specular=case.get("spec", 0.0))


def _bvh(scene):
    return H.hdof_build_bvh(_t(scene.verts), _t(scene.idx), _t(scene.mat), _t(scene.uv))


def _lens(case):
    return hi.Lens(case["focus"], case["aperture"], hi.ROOM_FOCAL).f32()


def _frame_params(case, seed):
    base = hi.Params() if case["scene"] == "tiny" else hi.room_params()
    return base.replace(spp_max=case["spp"], r_max=case["r_max"], variance_on=case["variance"], seed=seed & 0x7fffffff,
                        camera_moved=1 if case["scene"] == "room" else 0, alpha_k=case["alpha_k"],
                        mask_coc=case["mask_coc"], spec_pref=0.5 if case["spec"] > 0 else 0.0)


def _prepare_frame(case, seed):
    p = _frame_params(case, seed)
    W, Hh = case["width"], case["height"]
    dt = dict(nd_dtype=torch.float16, col_dtype=torch.bfloat16) if case["mixed"] else {}
    r = H.Renderer(_bvh(_scene_of(case, seed)), W, Hh, p, **dt)
    r.g.tri.fill_(-1)  # no previous frame yet
    step = 0.01 if case["scene"] == "room" else 0.0
    cams = [hi.room_camera(k, W, Hh, seed=seed, step=step) for k in range(case["frames"])]
    return dict(r=r, cams=cams, lens=_lens(case), ps=[p.replace(frame=k) for k in range(case["frames"])])


def _run_frame(st):
    r = st["r"]
    r.reset_history()
    for k, p in enumerate(st["ps"]):
        out = r.frame(st["cams"][k], st["cams"][max(k - 1, 0)], st["lens"], p)
    h = r.history
    return dict(out=out, near=h.near, far=h.far, mom=h.mom, hlen=h.hlen, spp=r.spp, tri=r.g.tri)


def _prepare_batch(case, seed):
    scenes = hi.batch_scenes(seeds=tuple(seed * 4 + k for k in range(4)))
    bvhs = [_bvh(s) for s in scenes]
    vs = hi.batch_views(case["views"], seed=seed)
    for v, w in zip(vs, hi.batch_views(case["views"])):  # the workload's sizes, poses and lenses by the seed
        v.width, v.height = w.width, w.height
    b = H.Batch([bvhs[v.room] for v in vs], [(v.width, v.height) for v in vs], [v.params for v in vs])
    for r in b.views:
        r.g.tri.fill_(-1)
    cams = [[v.camera(k, seed=seed) for v in vs] for k in range(case["frames"])]
    ps = [[v.params.replace(frame=k, camera_moved=1) for v in vs] for k in range(case["frames"])]
    return dict(b=b, cams=cams, ps=ps, lenses=[v.lens for v in vs])


def _run_batch(st):
    b = st["b"]
    for r in b.views:
        r.reset_history()
    for k, ps in enumerate(st["ps"]):
        outs = b.frame(st["cams"][k], st["cams"][max(k - 1, 0)], st["lenses"], ps)
    return [dict(out=o, near=r.history.near, far=r.history.far, hlen=r.history.hlen, tri=r.g.tri)
            for o, r in zip(outs, b.views)]


def _fit_inputs(case, seed):
    """Colour, depth, mask, frozen hit records, history samples and target of a fitting step."""
    W, Hh = case["width"], case["height"]
    col, z = hi.diff_inputs(W, Hh, seed)
    p = hi.room_params(r_max=32.0, variance_on=1, seed=seed & 0x7fffffff)
    cam = hi.Camera(width=W, height=Hh).f32()
    bvh = _bvh(hi.room_scene_target(seed, case["tris"], aspect=W / Hh))
    r = H.Renderer(bvh, W, Hh, p)
    H.hdof_gbuffer(bvh, cam, cam, p, r.g)
    H.hdof_mask(r.g, None, p, r.edge, r.spp, r.ws)
    spp = r.spp.clone()
    rec = torch.zeros((max(int(spp.to(torch.int64).sum()), 1), 4), device=DEV)
    ray_off = torch.zeros((Hh, W), dtype=torch.int32, device=DEV)
    H.hdof_trace(bvh, cam, hi.Lens(2.5, 0.04, 0.05).f32(), p, spp, r.rt, r.stats, r.ws, rec=rec, ray_off=ray_off)
    torch.cuda.synchronize()
    hs = _t(hi.random_hist_samples(W, Hh, seed))
    target = _t(np.random.default_rng(seed + 3).uniform(0, 1, (Hh, W, 3)).astype(np.float32))
    return _t(col), _t(z), spp, rec, ray_off, hs, target, cam, p


def _prepare_fit(case, seed):
    col, z, spp, rec, ray_off, hs, target, cam, p = _fit_inputs(case, seed)
    return dict(path=H.PostPath(z, spp, rec, ray_off, hs, cam, p), target=target, col=col.requires_grad_(),
                lens=torch.tensor([case["focus"], case["aperture"]], device=DEV, requires_grad=True))


def _run_fit(st):
    st["col"].grad = st["lens"].grad = None
    out = H.HdofPost.apply(st["col"], st["lens"], st["path"])
    ((out - st["target"]) ** 2).mean().backward()
    return dict(out=out.detach(), grad_col=st["col"].grad, grad_lens=st["lens"].grad)


def _gbuffer_planes(W, Hh, seed):
    g = hi.random_gbuffer(W, Hh, seed)
    g["nd"][..., 3] = np.clip(g["nd"][..., 3], 0.3, 12.0)  # slanted surfaces stay in front of the camera
    return g


def _pf_inputs(case, seed):
    g = _gbuffer_planes(case["width"], case["height"], seed)
    nd, col = _t(g["nd"]), _t(g["col"])
    if case["mixed"]:
        nd, col = nd.to(torch.float16), col.to(torch.bfloat16)
    p = hi.room_params(r_max=case["r_max"], blades=case["blades"], blade_rot=0.3, aberration=case["aberration"])
    return nd, col, p


def _prepare_postfilter(case, seed):
    nd, col, p = _pf_inputs(case, seed)
    W, Hh = case["width"], case["height"]
    return dict(g=H.GBuffer.from_tensors(nd, col), cam=hi.Camera(width=W, height=Hh).f32(), lens=_lens(case), p=p,
                pp=torch.empty((Hh, W, 4), device=DEV),
                ws=torch.empty(H.hdof_workspace_bytes(W, Hh, p), dtype=torch.uint8, device=DEV))


def _run_postfilter(st):
    H.hdof_postfilter(st["g"], st["cam"], st["lens"], st["p"], st["pp"], st["ws"])
    return st["pp"]


def _rec_inputs(case, seed):
    W, Hh = case["width"], case["height"]
    rng = np.random.default_rng(seed + 17)
    # traced 16x16 tiles, as the mask gives them
    tiles = rng.uniform(size=((Hh + 15) // 16, (W + 15) // 16)) < case["frac"]
    spp = np.kron(tiles, np.ones((16, 16), np.uint8))[:Hh, :W] * 8
    g, hist = _gbuffer_planes(W, Hh, seed), hi.random_history(W, Hh, seed)
    rt = hi.random_rt(W, Hh, spp, seed)
    pp = rng.uniform(0, 1, (Hh, W, 4)).astype(np.float32)
    p = hi.room_params(camera_moved=1, alpha_k=case["alpha_k"])
    cams = hi.room_camera(1, W, Hh, seed=seed), hi.room_camera(0, W, Hh, seed=seed)
    return (_t(spp.astype(np.uint8)), {k: _t(v) for k, v in g.items()}, {k: _t(v) for k, v in hist.items()}, _t(rt),
            _t(pp), p, cams, hi.room_lens())


def _prepare_reconstruct(case, seed):
    spp, g, hist, rt, pp, p, (cam, prev), lens = _rec_inputs(case, seed)
    W, Hh = case["width"], case["height"]
    z = lambda c: torch.zeros((Hh, W, c), device=DEV)  # noqa: E731
    return dict(spp=spp, g=H.GBuffer.from_tensors(g["nd"], g["col"], g["mv"]), rt=rt, pp=pp, p=p, cam=cam, prev=prev,
                lens=lens, hin=H.History.from_tensors(hist["near"], hist["far"], hist["mom"], hist["hlen"]),
                hout=H.History(W, Hh), crt=z(4), crec=z(4), out=z(4), hacc=torch.zeros((Hh, W), device=DEV))


def _run_reconstruct(st):
    s = st
    H.hdof_reconstruct(s["rt"], s["g"], s["spp"], s["cam"], s["prev"], s["lens"], s["p"], s["hin"], s["hout"],
                       s["crt"], s["hacc"], s["crec"])
    H.hdof_composite(s["g"], s["spp"], s["pp"], s["crt"], s["crec"], s["hacc"], s["cam"], s["lens"], s["p"], s["out"])
    h = s["hout"]
    return dict(crt=s["crt"], hacc=s["hacc"], crec=s["crec"], near=h.near, far=h.far, mom=h.mom, hlen=h.hlen,
                out=s["out"])


def _bvh_inputs(case, seed):
    sc = _scene_of(case, seed)
    rng = np.random.default_rng(seed + 5)
    n = case["rays"]
    org = rng.uniform((-1.5, -1.0, -0.4), (1.5, 1.0, 0.0), (n, 3)).astype(np.float32)
    d = rng.normal(size=(n, 3))
    d[:, 2] = np.abs(d[:, 2]) + 0.5
    return sc, org, d.astype(np.float32)


def _prepare_bvh(case, seed):
    sc, org, d = _bvh_inputs(case, seed)
    n, W, Hh = case["rays"], case["width"], case["height"]
    return dict(geo=[_t(a) for a in (sc.verts, sc.idx, sc.mat, sc.uv)], org=_t(org), dir=_t(d), p=hi.room_params(),
                cam=hi.room_camera(0, W, Hh, seed=seed), g=H.GBuffer(W, Hh),
                ids=torch.empty(n, dtype=torch.int32, device=DEV), ts=torch.empty(n, device=DEV))


def _run_bvh(st):
    bvh = H.hdof_build_bvh(*st["geo"])
    H.hdof_gbuffer(bvh, st["cam"], st["cam"], st["p"], st["g"])
    H.hdof_closest_hits(bvh, st["org"], st["dir"], st["ids"], st["ts"])
    return dict(ids=st["ids"], ts=st["ts"], nd=st["g"].nd, col=st["g"].col, tri=st["g"].tri)


def _prepare_reference(case, seed):
    W, Hh = case["width"], case["height"]
    p = hi.room_params(spp_max=case["spp"], seed=seed & 0x7fffffff)
    bvh = _bvh(hi.room_scene(seed=seed, aspect=W / Hh))
    image = _t(np.random.default_rng(seed).uniform(0, 1, (Hh, W, 4)).astype(np.float32))
    return dict(bvh=bvh, p=p, cam=hi.room_camera(0, W, Hh, seed=seed), lens=_lens(case), passes=case["passes"],
                g=H.GBuffer(W, Hh), rt=torch.empty((Hh, W, 4), device=DEV), image=image,
                err=torch.empty((Hh, W), device=DEV),
                stats=torch.zeros(H.ERR_SCRATCH, dtype=torch.float64, device=DEV),
                ws=torch.empty(H.hdof_workspace_bytes(W, Hh, p), dtype=torch.uint8, device=DEV))


def _run_reference(st):
    s = st
    H.hdof_gbuffer(s["bvh"], s["cam"], s["cam"], s["p"], s["g"])
    H.hdof_reference_rt(s["bvh"], s["cam"], s["lens"], s["p"], s["passes"], s["rt"], s["ws"], hint=s["g"].tri)
    H.hdof_error_map(s["image"], s["rt"], s["stats"], err=s["err"])
    return dict(rt=s["rt"], err=s["err"], stats=s["stats"][:H.ERR_STATS])


_PREPARE = dict(frame=_prepare_frame, batch=_prepare_batch, fit=_prepare_fit, postfilter=_prepare_postfilter,
                reconstruct=_prepare_reconstruct, bvh=_prepare_bvh, reference=_prepare_reference)
_RUN = dict(frame=_run_frame, batch=_run_batch, fit=_run_fit, postfilter=_run_postfilter, reconstruct=_run_reconstruct,
            bvh=_run_bvh, reference=_run_reference)


def prepare(case, seed):
    st = _PREPARE[case["kind"]](case, seed)
    st["kind"] = case["kind"]
    return st


def run(state):
    return _RUN[state["kind"]](state)


# ------------------------------------------------------------------- work --

def _tris(case):
    if case.get("scene") == "tiny":
        return 4
    return 12 + 12 * case.get("boxes", 64) + case.get("spheres", 32) * 20 * 4 ** case.get("subdiv", 4)


def work(case):
    k = case["kind"]
    px = case.get("width", 0) * case.get("height", 0)
    if k == "frame":
        # per frame: triangles (vertices, material), history in and out (41 B),
        # the image, hit ids and ray counts; per pixel one hit and its shading,
        # the mask's 5x5 Gaussian and Sobel, the blend (a quarter of the
        # pixels traced with spp rays)
        return dict(bytes=case["frames"] * (_tris(case) * 68 + px * (41 * 2 + 16 + 4 + 1)),
                    flops=case["frames"] * px * (100 + 4 * 30 + 60 + 0.25 * case["spp"] * 150))
    if k == "batch":
        # mean of the workload's four resolutions and four scene sizes
        mean_px = sum(w * h for w, h in hi.BATCH_RESOLUTIONS) / 4
        px = case["views"] * mean_px
        return dict(bytes=case["frames"] * (sum(hi.BATCH_TRIS) * 68 + px * (41 * 2 + 16 + 4 + 1)),
                    flops=case["frames"] * px * (280 + 0.25 * 16 * 150))
    if k == "fit":
        # colour, depth, mask, history samples and target in; image and
        # gradient out; per pixel a disk of mean radius 5 px forward and back
        return dict(bytes=px * (12 + 4 + 1 + 48 + 12 + 12 + 12), flops=px * (78 * 8 + 78 * 20))
    if k == "postfilter":
        # G-buffer in, image out; per pixel its disk's border once (the
        # interior of a disk can be had from sums along the rows)
        b = 16 if case["mixed"] else 32
        return dict(bytes=px * (b + 16), flops=px * 8 * 2 * math.pi * case["r_max"] / 2)
    if k == "reconstruct":
        traced = px * case["frac"]
        return dict(bytes=px * (16 + 16 + 16 + 1 + 16 + 16) + traced * (48 + 8 + 41 * 2 + 4 + 16),
                    flops=px * 60 + traced * (200 + 8 * math.pi * 5 ** 2))
    if k == "bvh":
        n = _tris(case)
        return dict(bytes=n * (12 + 36 + 32 + 24) + n * 100 + case["rays"] * 32 + px * 36,
                    flops=n * math.log2(n + 1) * 20 + (case["rays"] + px) * 100)
    rays = px * case["spp"] * case["passes"]
    return dict(bytes=_tris(case) * 68 + px * (16 + 16 + 4), flops=rays * 300)


# ------------------------------------------------------------ exact values --
# The defining sums in 64 bits, full windows, plain torch.

def _f32(x):
    return float(np.float32(x))


def _clamp01(x):
    return x.clamp(0.0, 1.0)


def _w_near(c):
    return _clamp01((c + math.sqrt(2.0)) / (2.0 * math.sqrt(2.0)))


def _coc(z, zf, A, Hh, t):
    return A * Hh / t * (1.0 / z - 1.0 / zf)


_AREA = {}


def _disk_area(r):
    """Lattice area sum_o clamp(r + 1/2 - |o|, 0, 1) of the soft disk (piecewise linear in r)."""
    if "x" not in _AREA:
        n = 66
        y, x = np.mgrid[-n:n + 1, -n:n + 1]
        d2, mult = np.unique((x * x + y * y)[x * x + y * y <= n * n], return_counts=True)
        d = np.sqrt(d2.astype(np.float64))
        xs = np.unique(np.concatenate([d - 0.5, d + 0.5]))
        xs = xs[(xs >= 0) & (xs <= n - 1)]
        a = np.array([(np.clip(v + 0.5 - d, 0, 1) * mult).sum() for v in xs])
        _AREA["x"], _AREA["a"] = _t(xs), _t(a)
    xs, a = _AREA["x"], _AREA["a"]
    k = (torch.searchsorted(xs, r.detach(), right=True) - 1).clamp(0, xs.numel() - 2)
    return a[k] + (a[k + 1] - a[k]) / (xs[k + 1] - xs[k]) * (r - xs[k])


def _pad(a, R, v=0.0):
    return torch.nn.functional.pad(a, (R, R, R, R), value=v)


def _rows(fn, G, tensors, grad):
    """Sum of fn(dy, *tensors) over dy = -G..G; with grad each row is recomputed in the backward."""
    tot = None
    for dy in range(-G, G + 1):
        s = checkpoint(fn, dy, *tensors, use_reentrant=False) if grad else fn(dy, *tensors)
        tot = s if tot is None else tuple(a + b for a, b in zip(tot, s))
    return tot


def _postfilter64(col, z, c, r_max, kz_rel, grad=False):
    """col [3,H,W], z and CoC c [H,W] -> post-filtered colour [3,H,W] and coverage [H,W]."""
    Hh, W = z.shape
    r = (c.abs() * 0.5).clamp(max=r_max)
    ia, wn = 1.0 / _disk_area(r), _w_near(c)
    one = torch.ones_like(z)[None]
    rgb1 = torch.cat([col, one])
    G = int(math.ceil(float(r.detach().max()) + 0.5))
    top = float(r.detach().max()) + 0.5

    def row(dy, rh, zq, near, far, zp):
        S = [torch.zeros((4, Hh, W), dtype=torch.float64, device=DEV) for _ in range(2)]
        w = int(math.sqrt(max(top * top - dy * dy, 0.0))) + 1
        for dx in range(-min(w, G), min(w, G) + 1):
            d = math.sqrt(dx * dx + dy * dy)
            if d >= top:
                continue
            v = (..., slice(G + dy, G + dy + Hh), slice(G + dx, G + dx + W))
            s = _clamp01(rh[v] - d)
            S[0] = S[0] + s * near[v]
            S[1] = S[1] + s * _clamp01(1.0 - (zq[v] - zp) / (kz_rel * zp)) * far[v]
        return S[0], S[1]

    args = (_pad(r + 0.5, G, -1.0), _pad(z, G, 1.0), _pad(rgb1 * (wn * ia), G), _pad(rgb1 * ((1.0 - wn) * ia), G), z)
    Sn, Sf = _rows(row, G, args, grad)
    alpha = _clamp01(Sn[3])
    N = torch.where(Sn[3] > 1e-8, Sn[:3] / Sn[3].clamp(min=1e-30), torch.zeros_like(col))
    F = torch.where(Sf[3] > 1e-8, Sf[:3] / Sf[3].clamp(min=1e-30), col)
    return alpha * N + (1.0 - alpha) * F, alpha


def _shaped64(col, z, c, r_max, kz_rel, blades, rot, ab):
    """The shaped post-filter: aperture norm D, radial weight, lattice area of the weighted shape."""
    Hh, W = z.shape
    r = (c.abs() * 0.5).clamp(max=r_max)
    top = float(r.max()) + 0.5
    G = int(math.ceil(top))

    def norm(dx, dy):
        d = math.hypot(dx, dy)
        if blades < 3 or d == 0.0:
            return d
        sect = 2.0 * math.pi / blades
        m = (math.atan2(dy, dx) - rot) % sect
        return d * math.cos(m - 0.5 * sect) / math.cos(0.5 * sect)

    def radial(rr, d):
        t = (d / rr.clamp(min=1e-6)).clamp(max=1.0)
        return torch.where(rr < 1.0, torch.ones_like(rr), 1.0 + ab * (2.0 * t * t - 1.0))

    area = torch.zeros_like(r)
    offs = [(dx, dy) for dy in range(-G, G + 1) for dx in range(-G, G + 1) if math.hypot(dx, dy) < top]
    for dx, dy in offs:
        area += _clamp01(r - norm(dx, dy) + 0.5) * radial(r, math.hypot(dx, dy))
    wn = _w_near(c)
    rgb1 = torch.cat([col, torch.ones_like(z)[None]])
    near, far = _pad(rgb1 * (wn / area), G), _pad(rgb1 * ((1.0 - wn) / area), G)
    rp, zq = _pad(r, G, -2.0), _pad(z, G, 1.0)
    Sn, Sf = torch.zeros_like(rgb1), torch.zeros_like(rgb1)
    for dx, dy in offs:
        v = (..., slice(G + dy, G + dy + Hh), slice(G + dx, G + dx + W))
        w = radial(rp[v], math.hypot(dx, dy))
        Sn += _clamp01(rp[v] - norm(dx, -dy) + 0.5) * w * near[v]
        Sf += _clamp01(rp[v] - norm(-dx, dy) + 0.5) * w * _clamp01(1.0 - (zq[v] - z) / (kz_rel * z)) * far[v]
    alpha = _clamp01(Sn[3])
    N = torch.where(Sn[3] > 1e-8, Sn[:3] / Sn[3].clamp(min=1e-30), torch.zeros_like(col))
    F = torch.where(Sf[3] > 1e-8, Sf[:3] / Sf[3].clamp(min=1e-30), col)
    return alpha * N + (1.0 - alpha) * F, alpha


def _spatial64(C, c, traced, mom, hlen, r_s, var_ref, grad=False):
    """Gather of the traced neighbours' colours C [3,H,W] by CoC c, blended by the luminance spread."""
    Hh, W = c.shape
    r = torch.where(traced, (c * 0.5).clamp(max=r_s), torch.full_like(c, -1.0))
    G = int(math.ceil(max(float(r.detach().max()), 0.0) + 0.5))
    top = max(float(r.detach().max()), 0.0) + 0.5

    def row(dy, rq, Cq, rp):
        S = torch.zeros((4, Hh, W), dtype=torch.float64, device=DEV)
        for dx in range(-G, G + 1):
            d = math.sqrt(dx * dx + dy * dy)
            if d >= top:
                continue
            v = (..., slice(G + dy, G + dy + Hh), slice(G + dx, G + dx + W))
            S = S + _clamp01(rp + 0.5 - d) * _clamp01(rq[v] + 0.5 - d) * Cq[v]
        return (S,)

    rgb1 = torch.cat([C, torch.ones_like(c)[None]])
    (S,) = _rows(row, G, (_pad(r, G, -1.0), _pad(rgb1, G), r), grad)
    var = (mom[..., 1] - mom[..., 0] ** 2).clamp(min=0.0)
    sig = torch.where(var > 0, var.clamp(min=1e-300).sqrt(), torch.zeros_like(var))
    beta = torch.where(hlen < 2, torch.ones_like(sig), _clamp01(sig / var_ref))
    return torch.where(traced, C + beta * (S[:3] / S[3].clamp(min=1e-30) - C), torch.zeros_like(C))


def _composite64(col, c, traced, pp, crt_c, crec, hacc, h_tau):
    ce = torch.where(traced, crt_c, c.abs())
    b = _clamp01(hacc / h_tau)
    near = torch.where(traced, crec, pp)
    far = torch.where(traced, crec + b * (pp - crec), pp)
    wn, f = _w_near(c), _clamp01(math.sqrt(2.0) + 0.5 - ce)
    blur = wn * near + (1.0 - wn) * far
    return blur + f * (col - blur)


def _ema64(h, Cn, Cf, nok, fok, cn, cf, hn, hf, hm, vn, vf, al, moved):
    """One temporal step over sampled history; planes [..], colours [3,..], history [4,..], moments [2,..]."""
    Ccur = torch.where(nok, torch.where(fok, h * Cn + (1.0 - h) * Cf, Cn), Cf)
    Y = 0.2126 * Ccur[0] + 0.7152 * Ccur[1] + 0.0722 * Ccur[2]
    cur_n, cur_f = torch.cat([h * Cn, h[None]]), torch.cat([(1.0 - h) * Cf, (1.0 - h)[None]])
    on = torch.where(vn, hn + al * (cur_n - hn), cur_n)
    of = torch.where(vf, hf + al * (cur_f - hf), cur_f)
    m = torch.stack([Y, Y * Y])
    om = torch.where(vn, hm + al * (m - hm), m)
    Bn, Bf = on[3], of[3]
    Hacc = torch.where(Bn + Bf >= 1e-6, Bn / (Bn + Bf).clamp(min=1e-30), h)
    an, af = Bn >= 1e-6, Bf >= 1e-6
    A, B = on[:3] / Bn.clamp(min=1e-30), of[:3] / Bf.clamp(min=1e-30)
    hw = h if moved else Hacc
    C = torch.where(~an, torch.where(af, B, torch.zeros_like(B)), torch.where(~af, A, hw * A + (1.0 - hw) * B))
    c = torch.where(~nok, cf, torch.where(~fok, cn, Hacc * cn + (1.0 - Hacc) * cf))
    return on, of, om, Hacc, C, c


def _chan(a):
    return a.movedim(-1, 0).double()


def _exact_postfilter(case, seed):
    nd, col, p = _pf_inputs(case, seed)
    Hh, cam, lens = case["height"], hi.Camera().f32(), _lens(case)
    z = nd[..., 3].double()
    c = _coc(z, lens.focus_dist, lens.aperture_radius, Hh, cam.tan_half_fovy)
    args = (_chan(col)[:3], z, c, _f32(p.r_max), _f32(p.kz_rel))
    if case["blades"] >= 3 or case["aberration"] != 0.0:
        o, a = _shaped64(*args, case["blades"], _f32(p.blade_rot), _f32(p.aberration))
    else:
        o, a = _postfilter64(*args)
    return torch.cat([o, a[None]]).movedim(0, -1)


def _sample64(planes, hlen, ux, uy):
    """Bilinear history sample [C,H,W] over taps with history, its validity and the taps' largest hlen."""
    Hh, W = hlen.shape
    x0, y0 = ux.floor(), uy.floor()
    fx, fy = ux - x0, uy - y0
    ws, out = torch.zeros_like(ux), torch.zeros((planes.shape[0],) + tuple(ux.shape), dtype=torch.float64, device=DEV)
    hmax = torch.zeros_like(hlen, dtype=torch.int64)
    for b in (0, 1):
        for a in (0, 1):
            x, y = x0 + a, y0 + b
            ok = (x >= 0) & (y >= 0) & (x < W) & (y < Hh)
            xi, yi = x.clamp(0, W - 1).long(), y.clamp(0, Hh - 1).long()
            hl = hlen[yi, xi].long()
            w = torch.where(ok & (hl > 0), (fx if a else 1.0 - fx) * (fy if b else 1.0 - fy), torch.zeros_like(fx))
            ws = ws + w
            out = out + w * planes[:, yi, xi]
            hmax = torch.where(w > 0, torch.maximum(hmax, hl), hmax)
    return out / ws.clamp(min=1e-30), ws >= 1e-3, hmax


def _exact_reconstruct(case, seed):
    spp, g, hist, rt, pp, p, (cam, prev), lens = _rec_inputs(case, seed)
    W, Hh = case["width"], case["height"]
    r = _chan(rt)
    traced = spp > 0
    h, cn, cf = r[3], r[7], r[11]
    nok, fok = cn >= 0, cf >= 0
    j, i = torch.meshgrid(torch.arange(Hh, device=DEV, dtype=torch.float64),
                          torch.arange(W, device=DEV, dtype=torch.float64), indexing="ij")
    mv = g["mv"].double()
    hn, vn, _ = _sample64(_chan(hist["near"]), hist["hlen"], i - mv[..., 0], j - mv[..., 1])
    hm, _, _ = _sample64(_chan(hist["mom"]), hist["hlen"], i - mv[..., 0], j - mv[..., 1])
    # far position: own far hits, else the traced neighbours', else the surface
    ok = (traced & fok).double()
    P, pok = _pad(r[8:11] * ok, 1), _pad(ok, 1)
    S, n = torch.zeros_like(r[8:11]), torch.zeros_like(ok)
    for b in (0, 1, 2):
        for a in (0, 1, 2):
            if (a, b) != (1, 1):
                S, n = S + P[:, b:b + Hh, a:a + W], n + pok[b:b + Hh, a:a + W]
    asp, t = W / Hh, cam.tan_half_fovy
    X = (2.0 * (i + 0.5 + cam.jitter[0]) / W - 1.0) * asp * t
    Yd = (1.0 - 2.0 * (j + 0.5 + cam.jitter[1]) / Hh) * t
    vec = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV)[:, None, None]  # noqa: E731
    surf = vec(cam.pos) + g["nd"][..., 3].double() * (X * vec(cam.right) + Yd * vec(cam.up) + vec(cam.fwd))
    Pw = torch.where(fok, r[8:11], torch.where(n > 0, S / n.clamp(min=1.0), surf)) - vec(prev.pos)
    zc = (Pw * vec(prev.fwd)).sum(0)
    Xp, Yp = (Pw * vec(prev.right)).sum(0) / zc, (Pw * vec(prev.up)).sum(0) / zc
    uf = (Xp / (asp * prev.tan_half_fovy) + 1.0) * 0.5 * W - 0.5 - prev.jitter[0]
    vf_ = (1.0 - Yp / prev.tan_half_fovy) * 0.5 * Hh - 0.5 - prev.jitter[1]
    big = torch.full_like(uf, 1e9)
    hf, vf, _ = _sample64(_chan(hist["far"]), hist["hlen"], torch.where(zc > 0, uf, big), torch.where(zc > 0, vf_, big))
    al = torch.full_like(h, _f32(p.ema_alpha))
    Cn, Cf = r[0:3], r[4:7]
    if case["alpha_k"] > 0:
        Ccur = torch.where(nok, torch.where(fok, h * Cn + (1.0 - h) * Cf, Cn), Cf)
        Y = 0.2126 * Ccur[0] + 0.7152 * Ccur[1] + 0.0722 * Ccur[2]
        sg = (hm[1] - hm[0] ** 2).clamp(min=0.0).sqrt()
        ak = _f32(case["alpha_k"])
        lam = _clamp01(((Y - hm[0]).abs() - ak * sg) / torch.maximum(Y, hm[0]).clamp(min=1e-3))
        se = ((hn[3] * (1.0 - hn[3])).clamp(min=0.0) / spp.double().clamp(min=1.0)).sqrt()
        lam = torch.maximum(lam, _clamp01((h - hn[3]).abs() - ak * se))
        al = torch.where(vn, al + (1.0 - al) * lam, al)
    on, of, om, Hacc, C, c = _ema64(h, Cn, Cf, nok, fok, cn, cf, hn, hf, hm, vn, vf, al, p.camera_moved)
    _, _, hmax = _sample64(_chan(hist["mom"]), hist["hlen"], i - mv[..., 0], j - mv[..., 1])
    hlen = torch.where(vn, hmax + 1, torch.ones_like(hmax)).clamp(max=255)
    crec = _spatial64(C * traced, c, traced, om.movedim(0, -1), hlen, _f32(p.r_s), _f32(p.var_ref))
    cz = _coc(g["nd"][..., 3].double(), lens.focus_dist, lens.aperture_radius, Hh, t)
    out = _composite64(_chan(g["col"])[:3], cz, traced, _chan(pp)[:3], c, crec, Hacc, _f32(p.h_tau))
    zero = torch.zeros((1, Hh, W), dtype=torch.float64, device=DEV)
    last = lambda a: a.movedim(0, -1)  # noqa: E731
    crt = torch.where(traced, torch.cat([C, c[None]]), torch.cat([zero, zero, zero, zero - 1.0]))
    return dict(crt=last(crt), hacc=Hacc * traced, crec=last(torch.cat([crec, zero])), near=last(on * traced),
                far=last(of * traced), mom=last(om * traced), hlen=None, out=last(torch.cat([out, zero])))


def _exact_fit(case, seed):
    col, z, spp, rec, ray_off, hs, target, cam, p = _fit_inputs(case, seed)
    W, Hh = case["width"], case["height"]
    C = _chan(col).requires_grad_()
    lens = torch.tensor([_f32(case["focus"]), _f32(case["aperture"])], dtype=torch.float64, device=DEV,
                        requires_grad=True)
    zf, A = lens[0], lens[1]
    t, z = cam.tan_half_fovy, z.double()
    # the trace accumulation re-evaluated from the hit records
    n = spp.long().flatten()
    pix = torch.repeat_interleave(torch.arange(W * Hh, device=DEV), n)
    first = torch.cumsum(n, 0) - n
    k = ray_off.flatten().long()[pix] + torch.arange(pix.numel(), device=DEV) - first[pix]
    rr = rec[k].double()
    c = A * Hh / t * (1.0 / rr[:, 3] - 1.0 / zf)  # 1/inf = 0: a miss
    w, ac, L = _w_near(c), c.abs(), rr[:, :3]
    vals = torch.cat([w[:, None] * L, (1.0 - w)[:, None] * L, torch.stack([w, 1.0 - w, w * ac, (1.0 - w) * ac], 1)], 1)
    S = torch.zeros((W * Hh, 10), dtype=torch.float64, device=DEV).index_add(0, pix, vals).T.reshape(10, Hh, W)
    Sw, Sf = S[6], S[7]
    nok, fok = Sw >= 1e-6, Sf >= 1e-6
    dw, df = Sw.clamp(min=1e-6), Sf.clamp(min=1e-6)
    zero3 = torch.zeros_like(S[0:3])
    Cn, Cf = torch.where(nok, S[0:3] / dw, zero3), torch.where(fok, S[3:6] / df, zero3)
    cn = torch.where(nok, S[8] / dw, torch.full_like(Sw, -1.0))
    cf = torch.where(fok, S[9] / df, torch.full_like(Sw, -1.0))
    h = Sw / spp.double().clamp(min=1.0)
    hp = _chan(hs)
    vn, vf = (hp[10].long() & 1) > 0, (hp[10].long() & 2) > 0
    traced = spp > 0
    _, _, om, Hacc, Ct, ct = _ema64(h, Cn, Cf, nok, fok, cn, cf, hp[0:4], hp[4:8], hp[8:10], vn, vf,
                                    _f32(p.ema_alpha), p.camera_moved)
    hlen = torch.where(vn, hp[11] + 1, torch.ones_like(hp[11]))
    crec = _spatial64(torch.where(traced, Ct, zero3), torch.where(traced, ct, torch.zeros_like(ct)), traced,
                      om.movedim(0, -1), hlen, _f32(p.r_s), _f32(p.var_ref), grad=True)
    cz = _coc(z, zf, A, Hh, t)
    pp, _ = _postfilter64(C, z, cz, _f32(p.r_max), _f32(p.kz_rel), grad=True)
    out = _composite64(C, cz, traced, pp, ct, crec, Hacc, _f32(p.h_tau)).movedim(0, -1)
    ((out - target.double()) ** 2).mean().backward()
    return dict(out=out.detach(), grad_col=C.grad.movedim(0, -1), grad_lens=lens.grad)


def _exact_bvh(case, seed):
    sc, org, d = _bvh_inputs(case, seed)
    tv = _t(sc.tri_verts()).double().reshape(-1, 3, 3)
    v0, e1, e2 = tv[:, 0], tv[:, 1] - tv[:, 0], tv[:, 2] - tv[:, 0]
    org, d = _t(org).double(), _t(d).double()
    ts = torch.empty(org.shape[0], dtype=torch.float64, device=DEV)
    step = max(1, (1 << 24) // tv.shape[0])
    for a in range(0, org.shape[0], step):
        o, r = org[a:a + step, None], d[a:a + step, None]
        pv = torch.linalg.cross(r.expand(-1, tv.shape[0], -1), e2.expand(o.shape[0], -1, -1))
        det = (pv * e1).sum(-1)
        s = o - v0
        u = (s * pv).sum(-1) / det
        qv = torch.linalg.cross(s, e1.expand(o.shape[0], -1, -1))
        v = (qv * r).sum(-1) / det
        t = (qv * e2).sum(-1) / det
        ok = (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0)
        ts[a:a + step] = torch.where(ok, t, torch.full_like(t, math.inf)).amin(1)
    # the planes' million primary rays against every triangle would take a minute
    return dict(ids=None, ts=ts, nd=None, col=None, tri=None)


_EXACT = dict(postfilter=_exact_postfilter, reconstruct=_exact_reconstruct, fit=_exact_fit, bvh=_exact_bvh)


def exact(case, seed):
    """None for whole traced frames: millions of rays against every triangle in
    64 bits take minutes (their parts are the other kinds' exact values)."""
    fn = _EXACT.get(case["kind"])
    return fn(case, seed) if fn else None
