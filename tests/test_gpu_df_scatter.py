"""The pairwise scatter of the 512-thread double-float kernels (M = 9216 and 12288 points, and the general
lengths) at the edges of its lanes and warps: 1e-11, that operator's tolerance."""
import numpy as np
import pytest

import oracle as O
from helpers import assert_close
from test_gpu_half3 import LAM, scan_with

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker


@pytest.mark.parametrize("L", [16384, 18432, 24576])
@pytest.mark.parametrize("pixels,nx", [("raster", 16), ("random", 8), ("steps", 16), ("still", 8)])
def test_pairwise_scatter_of_every_fill(L, pixels, nx):
    """Blocks that end inside a lane's pair, lane or warp, start at odd samples (single weights), hold one
    sample; lanes with one, two and eight pixels."""
    full = L - LAM
    scan = scan_with([full, 1, 2, 3, full - 1, 255, 256, 257, 1151, 7, 9], pixels, nx, L + nx)
    c = MM.Context(0, None, MM.MM_FP32_MIXED)
    c.set_option("filter", 2)
    c.set_option("fft_len", L)
    c.set_option("apply_precision", 2)
    c.setup_scan(scan)
    x = np.random.default_rng(L).standard_normal((2, scan.n_pix, 3))
    y = c.apply_A(x)
    assert c.get_option("plan_whole") == 2
    prob = O.Problem.from_scan(scan)
    for r in range(2):
        assert_close(y[r], O.apply_A(prob, x[r]), 1e-11)
    d = np.random.default_rng(1).standard_normal((1, scan.n_samples)).astype(c.tod_dtype)
    assert_close(c.rhs(d)[0], O.rhs(prob, d[0].astype(np.float64)), 1e-11)
    c.close()
