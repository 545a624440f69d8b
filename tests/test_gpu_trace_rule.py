"""The trace on both sides of the line from which a view's rays are listed by
lens bin."""
import numpy as np
import pytest

import hdof_inputs as hi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2210_04981_gb300.hdof as H  # noqa: E402
from gpu_util import bvh_of, dev, host, report, rt_close, workspace  # noqa: E402


@pytest.mark.parametrize("W,Hh,spp_max,K", [(19, 130, 16, 3.5), (19, 130, 16, 3.6), (33, 128, 17, 3.4),
                                            (33, 128, 17, 3.5), (40, 40, 255, 0.88), (40, 40, 255, 0.9),
                                            (9, 230, 5, 6.3), (9, 230, 5, 6.4), (2, 700, 1, 14.1), (2, 700, 1, 14.2)])
def test_trace_at_the_line_of_the_sorted_list(orc, W, Hh, spp_max, K):
    """Just below and above K^2 spp = 200 (lists staged and not, ragged tiles,
    tiles with no ray): both forms give the same bits, each record at its
    pixel's place, and the oracle's radiance."""
    scene = hi.room_scene(seed=3, n_boxes=24, n_spheres=6, subdiv=2, aspect=W / Hh)
    cam = hi.Camera(width=W, height=Hh).f32()
    lens = hi.Lens(3.0, K * 3.0 * cam.tan_half_fovy / Hh, 0.05).f32()
    p = hi.room_params(spp_max=spp_max)
    bvh = bvh_of(scene)
    rng = np.random.default_rng(W)
    spp = rng.integers(0, spp_max + 1, (Hh, W)) * (rng.uniform(size=(Hh, W)) < 0.6)
    spp = spp.astype(np.uint8)
    spp[Hh // 2:Hh // 2 + 32] = 0
    n = int(spp.astype(np.int64).sum())
    outs = []
    for refill in (-1, 0, 4):
        rt = torch.zeros((Hh, W, 12), dtype=torch.float32, device="cuda")
        rec = torch.zeros((n, 4), dtype=torch.float32, device="cuda")
        off = torch.zeros((Hh, W), dtype=torch.int32, device="cuda")
        stats = torch.zeros(2, dtype=torch.int32, device="cuda")
        ids = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        ws = workspace(W, Hh, p)
        H.hdof_trace(bvh, cam, lens, p, dev(spp), rt, stats, ws, rec=rec, ray_off=off, tune=H.tuning(128, refill))
        H.hdof_trace_hits(bvh, cam, p, dev(spp), ws, ids)
        H.hdof_sync()
        assert host(stats).tolist() == [int((spp > 0).sum()), n]
        outs.append((rt, rec, ids))
    for o in outs[1:]:
        for a, b in zip(outs[0], o):
            assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    assert (outs[0][2] >= -1).all()
    ref = orc.trace(orc.OScene(scene), cam, lens, p, spp)
    ok = rt_close(host(outs[0][0]), ref, spp > 0)
    assert ok.mean() >= 0.998, report("rt", host(outs[0][0])[spp > 0], ref[spp > 0])
