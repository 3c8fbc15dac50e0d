"""M_BD of a block longer than one grid of its sums' slices (1024 of 8192 samples): walked, not refused."""
import numpy as np
import pytest

import synth
from helpers import assert_close

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker


@pytest.mark.parametrize("prec", [MM.MM_FP64, MM.MM_FP32_MIXED])
@pytest.mark.parametrize("n_t", [1024 * 8192, 1024 * 8192 + 1, 2 * 1024 * 8192 + 4099])
def test_blocks_at_and_beyond_one_grid_of_slices(n_t, prec):
    nx, f = 8, 1.7
    g = torch.Generator(device="cuda").manual_seed(n_t)
    pix = (torch.arange(n_t, device="cuda") // 5 % (nx * nx)).int()
    pix[torch.rand(n_t, generator=g, device="cuda") < 0.01] = -1
    psi = torch.rand(n_t, generator=g, device="cuda") * 3.1
    c = MM.Context(0, None, prec)
    c.setup_pointing(pix, psi, np.array([0, n_t], dtype=np.int64), np.zeros(1, dtype=np.int32), np.array([[f]]), nx * nx)
    assert c.build_bd(1e-3) == 0
    ok = pix >= 0
    p, a = pix[ok].long(), 2.0 * psi[ok].double()
    w = torch.stack([torch.ones_like(a), torch.cos(a), torch.sin(a)], 1)
    S = torch.zeros((nx * nx, 9), device="cuda", dtype=torch.float64)
    S.index_add_(0, p, f * (w[:, :, None] * w[:, None, :]).reshape(-1, 9))
    x = torch.randn((nx * nx, 3), generator=g, device="cuda", dtype=torch.float64)
    want = torch.linalg.solve(S.view(-1, 3, 3), x)
    got = c.apply_precond(MM.MM_PRECOND_BD, x[None].contiguous())[0]
    # sums of 1e5 to 4e5 terms a pixel in float64: 4e5 x 1.1e-16 = 5e-11, conditioning below 4
    assert_close(got.cpu().numpy(), want.cpu().numpy(), 2e-10)
    c.close()
