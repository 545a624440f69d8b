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
