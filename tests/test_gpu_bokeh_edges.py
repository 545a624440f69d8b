"""The shaped post-filter at the ends of its inputs: a narrow depth test, and
sources that are not finite."""
import numpy as np
import pytest

import hdof_inputs as hi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2210_04981_gb300.hdof as H  # noqa: E402
from gpu_util import frac_close, gbuf_from, host, report, workspace  # noqa: E402

SHAPES = [dict(blades=6, blade_rot=0.3, aberration=0.4), dict(blades=5, blade_rot=0.0, aberration=0.0)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kz_rel", [1e-5, 1e-4, 0.05])
def test_shaped_depth_test_at_a_narrow_range(orc, shape, kz_rel):
    """A far plane whose depths differ by up to the depth test's own width
    kz_rel z, dark where it lies behind its middle: the test's weights spread
    over [0, 1].  z_q - z_p is exact in floats, so a weight is off by a few
    2^-24; the filtered colours (means of values up to 0.9) agree to 1e-4 as
    elsewhere.  With the test as (1 + 1/kz_rel) - z_q / (kz_rel z_p) a weight
    would be off by 2^-24 / kz_rel = 6e-3 at 1e-5."""
    W, Hh = 67, 45
    rng = np.random.default_rng(1)
    cam, lens = hi.Camera(width=W, height=Hh).f32(), hi.Lens(1.0, 0.2, 0.05).f32()
    u = rng.uniform(-1.0, 1.0, (Hh, W))
    nd, col = np.zeros((Hh, W, 4), np.float32), np.zeros((Hh, W, 4), np.float32)
    nd[..., 2] = -1.0
    nd[..., 3] = 4.0 * (1.0 + kz_rel * u)
    col[..., :3] = np.where(u > 0, 0.1, 0.9)[..., None]
    p = hi.Params(r_max=12.0, kz_rel=float(np.float32(kz_rel)), **shape)
    pp = torch.empty((Hh, W, 4), device="cuda")
    H.hdof_postfilter(gbuf_from(nd, col), cam, lens, p, pp, workspace(W, Hh, p))
    H.hdof_sync()
    ref = orc.postfilter(nd.astype(np.float64), col.astype(np.float64), lens, cam.tan_half_fovy, p)
    assert ref[..., :3].max() - ref[..., :3].min() > 0.05
    assert frac_close(host(pp), ref, 1e-4) >= 0.999, report("pp", host(pp), ref)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("zf", [0.5, 2.0, 8.0])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_shaped_source_that_is_not_finite(shape, zf, bad):
    """A source of infinite or NaN colour changes no pixel outside its own disk
    (those are equal to the image with a finite one there, bit for bit: it
    adds nothing to them), and is not finite where it weighs."""
    W, Hh, y, x = 211, 97, 40, 150
    g = hi.random_gbuffer(W, Hh, seed=3)
    g["nd"][..., 3] = np.clip(g["nd"][..., 3], 0.4, 12.0)
    cam, lens = hi.Camera(width=W, height=Hh).f32(), hi.Lens(zf, 0.05, 0.05).f32()
    p = hi.Params(r_max=20.0, **shape)
    outs = []
    for c in (0.5, bad):
        g["col"][y, x, :3] = c
        pp = torch.empty((Hh, W, 4), device="cuda")
        H.hdof_postfilter(gbuf_from(g["nd"], g["col"]), cam, lens, p, pp, workspace(W, Hh, p))
        H.hdof_sync()
        outs.append(host(pp))
    K = lens.aperture_radius * Hh / cam.tan_half_fovy
    r = min(abs(K * (1.0 / g["nd"][y, x, 3] - 1.0 / zf)) / 2, 20.0)
    yy, xx = np.mgrid[0:Hh, 0:W]
    outside = np.hypot(yy - y, xx - x) > r + 0.5 + 1e-3
    assert outside.any() and np.array_equal(outs[0][outside], outs[1][outside])
    assert not np.isfinite(outs[1][y, x, :3]).all()
