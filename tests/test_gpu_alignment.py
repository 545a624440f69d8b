"""Workspaces that start at a multiple of 16 bytes only: every call that takes
one gives the results it gives on a 256-byte aligned one, bit for bit."""
import numpy as np
import pytest

import hdof_inputs as hi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2210_04981_gb300.hdof as H  # noqa: E402
from gpu_util import bvh_of, dev, gbuf_from  # noqa: E402


def _ws(n, off):
    """n bytes that start off bytes after a multiple of 256."""
    buf = torch.zeros(n + 512, dtype=torch.uint8, device="cuda")
    first = -buf.data_ptr() % 256 + off
    return buf[first:first + n]


def _same(call, n, off):
    """call(workspace) -> tensors: equal on an aligned workspace and off bytes behind one."""
    outs = []
    for o in (0, off):
        outs.append([t.clone() for t in call(_ws(n, o))])
        H.hdof_sync()
    for a, b in zip(*outs):
        assert torch.equal(a, b)


@pytest.mark.parametrize("off", [16, 240])
@pytest.mark.parametrize("W,Hh", [(61, 47), (64, 48)])
@pytest.mark.parametrize("shape", [{}, dict(blades=6, blade_rot=0.3, aberration=0.4)])
def test_postfilter_workspace_alignment(shape, W, Hh, off):
    gb = hi.random_gbuffer(W, Hh, seed=2)
    gb["col"][..., 3] = gb["col"][..., 0]
    cam, lens = hi.Camera(width=W, height=Hh).f32(), hi.Lens(2.0, 0.06, 0.05).f32()
    p = hi.Params(r_max=12.0, **shape)
    n = H.hdof_workspace_bytes(W, Hh, p)
    for dt in ({}, dict(nd_dtype=torch.float16, col_dtype=torch.bfloat16)):
        g = gbuf_from(gb["nd"], gb["col"], **dt)
        for fn in (H.hdof_postfilter, H.hdof_postfilter_spec):
            def call(ws):
                pp = torch.zeros((Hh, W, 4), device="cuda")
                fn(g, cam, lens, p, pp, ws)
                return [pp]
            _same(call, n, off)


def test_trace_mask_reference_workspace_alignment():
    scene, cam, lens, p = hi.tiny_config()
    bvh = bvh_of(scene)
    W, Hh = cam.width, cam.height
    g = H.GBuffer(W, Hh)
    H.hdof_gbuffer(bvh, cam, cam, p, g)

    def call(ws):
        edge, spp = (torch.zeros((Hh, W), dtype=torch.uint8, device="cuda") for _ in range(2))
        rt, out = torch.zeros((Hh, W, 12), device="cuda"), torch.zeros((Hh, W, 4), device="cuda")
        H.hdof_mask(g, None, p, edge, spp, ws)
        H.hdof_trace(bvh, cam, lens, p, spp, rt, torch.zeros(2, dtype=torch.int32, device="cuda"), ws)
        H.hdof_reference_rt(bvh, cam, lens, p, 2, out, ws)
        return edge, spp, rt, out
    _same(call, H.hdof_workspace_bytes(W, Hh, p), 16)


@pytest.mark.parametrize("W,Hh", [(33, 21), (48, 32)])
def test_post_path_workspace_alignment(W, Hh):
    rng = np.random.default_rng(W)
    spp = rng.integers(0, 5, (Hh, W)).astype(np.uint8)
    n = int(spp.sum())
    rec = np.concatenate([rng.uniform(0, 1, (n, 3)), rng.uniform(0.5, 6.0, (n, 1))], -1).astype(np.float32)
    off = (np.cumsum(spp.astype(np.int64).ravel()) - spp.ravel()).reshape(Hh, W).astype(np.int32)
    p = hi.room_params(r_max=10.0)
    path = H.PostPath(dev(rng.uniform(0.5, 6.0, (Hh, W)).astype(np.float32)), dev(spp), dev(rec), dev(off),
                      dev(hi.random_hist_samples(W, Hh, 1)), hi.Camera(width=W, height=Hh).f32(), p)
    col, g = (dev(rng.uniform(-1, 1, (Hh, W, 3)).astype(np.float32)) for _ in range(2))

    def call(ws):
        path.ws = ws
        out = path.forward(col, 2.0, 0.05)
        return [out, *path.backward(g, 2.0, 0.05)]
    _same(call, H.hdof_post_workspace_bytes(W, Hh, p), 16)


def test_batch_workspace_alignment():
    scene, cam, lens, p = hi.tiny_config()
    b = H.Batch([bvh_of(scene)], [(cam.width, cam.height)], [p])
    r = b.views[0]
    r.g.tri.fill_(-1)

    def call(ws):
        r.ws = ws
        r.reset_history()
        return [b.frame([cam], [cam], [lens], [p])[0]]
    _same(call, r.ws.numel(), 16)
