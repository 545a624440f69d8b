"""The round post-filter where its far layer is wide (the focus in front of
every surface), and where a bright source shares rows with dark pixels."""
import numpy as np
import pytest

import hdof_inputs as hi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2210_04981_gb300.hdof as H  # noqa: E402
from gpu_util import frac_close, gbuf_from, host, report, workspace  # noqa: E402


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("W,Hh,r", [(97, 61, 10.0), (64, 80, 20.0), (131, 45, 30.0)])
def test_wide_far_layer(orc, W, Hh, r, mixed):
    """Every surface behind the focus, radii up to r.  FP32: sums of at most
    (2 x 30 + 1)^2 positive terms, 1e-4 as elsewhere.  BF16 records: each
    term's colour and weight are off by 2^-9 of themselves, so a quotient of
    their sums by 2^-8 of values below 1."""
    gb = hi.random_gbuffer(W, Hh, seed=W, zrange=(0.6, 8.0))
    gb["nd"][..., 3] = np.clip(gb["nd"][..., 3], 0.6, 12.0)
    cam = hi.Camera(width=W, height=Hh).f32()
    lens = hi.Lens(0.5, 2.0 * r * 0.5 * cam.tan_half_fovy / Hh, 0.05).f32()
    p = hi.Params(r_max=r)
    g = gbuf_from(gb["nd"], gb["col"], **(dict(nd_dtype=torch.float16, col_dtype=torch.bfloat16) if mixed else {}))
    pp = torch.empty((Hh, W, 4), device="cuda")
    H.hdof_postfilter(g, cam, lens, p, pp, workspace(W, Hh, p))
    H.hdof_sync()
    nd, col = host(g.nd).astype(np.float64), host(g.col).astype(np.float64)
    ref = orc.postfilter(nd, col, lens, cam.tan_half_fovy, p)
    assert (ref[..., 3] < 0.5).mean() > 0.9  # far layer
    tol = 2.0 ** -8 if mixed else 1e-4
    assert frac_close(host(pp), ref, tol) >= 0.999, report("pp", host(pp), ref)


@pytest.mark.parametrize("bright", [1.0, 1e3, 1e6])
def test_bright_source_in_a_dark_blurred_row(orc, bright):
    """A strongly blurred near plane, dark but for a few bright pixels.  A
    pixel's sums take at most two prefix entries in each of 2 r + 1 rows, each
    rounded in at most 5 + 7 + ceil(W/256) additions by 2^-24 of its row's
    colour sum (the bright record's b / area and the dark ones' together); N
    divides by a weight of about 1.  At a bright pixel itself, alpha's own
    error (1e-6) times its colour comes on top."""
    W, Hh, r = 333, 90, 14.0
    rng = np.random.default_rng(3)
    cam = hi.Camera(width=W, height=Hh).f32()
    zf, z0 = 4.0, 1.0
    lens = hi.Lens(zf, 2.0 * r * cam.tan_half_fovy / Hh / (1.0 / z0 - 1.0 / zf), 0.05).f32()
    nd, col = np.zeros((Hh, W, 4), np.float32), np.zeros((Hh, W, 4), np.float32)
    nd[..., 2] = -1.0
    nd[..., 3] = z0 + 0.05 * np.sin(np.arange(W) / 40.0)
    col[..., :3] = rng.uniform(0.02, 0.06, (Hh, W, 3))
    spots = np.zeros((Hh, W), bool)
    spots[[20, 45, 70], [60, 160, 300]] = True
    col[spots, :3] = bright
    p = hi.Params(r_max=32.0)
    pp = torch.empty((Hh, W, 4), device="cuda")
    H.hdof_postfilter(gbuf_from(nd, col), cam, lens, p, pp, workspace(W, Hh, p))
    H.hdof_sync()
    ref = orc.postfilter(nd.astype(np.float64), col.astype(np.float64), lens, cam.tan_half_fovy, p)
    area = np.pi * 12.0 ** 2  # below every disk's area here
    row_sum = (bright + 0.06 * W) / area
    tol = 2 * (2 * 17 + 1) * (5 + 7 + 2) * 2.0 ** -24 * row_sum + 1e-6
    d = np.abs(host(pp)[..., :3] - ref[..., :3])
    # the taps of the rim: a weight is off by a few 2^-22 x r of the source's record
    tol += 4 * 2.0 ** -22 * 17 * (bright / area)
    assert (d[~spots] <= tol).all(), (d[~spots].max(), tol)
    assert (d[spots] <= tol + 4e-6 * bright).all()
