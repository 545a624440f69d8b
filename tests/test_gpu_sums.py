"""Reductions that are returned, or that cancel, in double: the bits that a
double sum keeps are kept."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2210_04981_gb300.hdof as H  # noqa: E402
from gpu_util import dev, host  # noqa: E402


@pytest.mark.parametrize("W,Hh", [(1, 1), (5, 1), (640, 411)])
@pytest.mark.parametrize("d,n", [((1.0, 2.0 ** -25, 2.0 ** -49), 7), ((1.0, 2.0 ** -13, 2.0 ** -25), 7)])
def test_error_map_sums_keep_a_doubles_bits(W, Hh, d, n):
    """Differences of which every partial sum is exact in a double (multiples
    of 2^-49 and 2^-50 below 8, 53 bits): the sums of |d| (first set) and of
    d^2 (second set) are exact, in any order, from one pixel to a whole grid."""
    a = np.zeros((Hh, W, 4), np.float32)
    px = np.random.default_rng(W).choice(W * Hh, min(n, W * Hh), replace=False)
    a.reshape(-1, 4)[px, :3] = d
    region = np.zeros((Hh, W), np.uint8)
    region.reshape(-1)[px[: len(px) // 2 + 1]] = 1
    stats = torch.empty(H.ERR_SCRATCH, dtype=torch.float64, device="cuda")
    H.hdof_error_map(dev(a), torch.zeros((Hh, W, 4), device="cuda"), stats, region=dev(region))
    H.hdof_sync()
    got = host(stats)
    x = a[..., :3].astype(np.float64)
    for k, v in ((0, x), (4, x[region > 0])):
        if d[2] == 2.0 ** -49:
            assert got[k + 1] == v.sum()
        else:
            assert got[k + 2] == (v * v).sum()


@pytest.mark.parametrize("zf", [2.9, 3.0, 3.1, 3.3])
def test_lens_gradient_keeps_a_doubles_bits(zf):
    """A lens gradient whose terms cancel within a warp.  32x8 traced pixels,
    all alike: near surfaces (near weight 1, its slope 0), one near hit each
    inside the composite's focus ramp, no history, no spatial reach.  A
    pixel's term is then linear in its image gradient, so that gradients 1,
    2^-25, 2^-28, -1, -2^-25 at five pixels of a row add up to 2^-28 times the
    term x of one pixel.  Every partial sum of the row fits a double's 53 bits
    (24 of x, 28 of the scales), so the result is exact; what is 2^-48 below x
    is lost in a pair of floats, and 4 units in the last place of the result
    with it."""
    import hdof_inputs as hi
    W, Hh, A = 32, 8, 0.5
    cam = hi.Camera(width=W, height=Hh).f32()
    K = A * Hh / cam.tan_half_fovy
    z = np.full((Hh, W), 1.0, np.float32)
    rec = np.empty((W * Hh, 4), np.float32)
    rec[:] = [0.7, 0.3, 0.2, 1.0 / (1.6 / K + 1.0 / zf)]  # |c| = 1.6: between sqrt 2 and sqrt 2 + 1/2
    p = hi.room_params(r_s=0.0, r_max=8.0, variance_on=0)
    path = H.PostPath(dev(z), torch.ones((Hh, W), dtype=torch.uint8, device="cuda"), dev(rec),
                      torch.arange(W * Hh, dtype=torch.int32, device="cuda").reshape(Hh, W), None, cam, p)
    col = torch.full((Hh, W, 3), 0.123, device="cuda")

    def grad(terms):
        g = torch.zeros((Hh, W, 3), device="cuda")
        for lane, v in terms.items():
            g[2, lane, 0] = v
        path.forward(col, zf, A)
        return host(path.backward(g, zf, A)[1])

    one = grad({0: 1.0})
    assert (one != 0).all() and np.isfinite(one).all()
    assert np.array_equal(grad({0: 2.0 ** -28}), one * np.float32(2.0 ** -28))
    got = grad({0: 1.0, 16: 2.0 ** -25, 8: 2.0 ** -28, 4: -1.0, 20: -2.0 ** -25})
    assert np.array_equal(got, one * np.float32(2.0 ** -28)), (got, one)
