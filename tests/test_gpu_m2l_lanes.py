"""M_2l on the CUDA cores around the sizes where its lanes per pixel and its chunks change: 1e-9 against
Eq. m2l in float64 (E of random columns has a condition number below 1e4)."""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import assert_close

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker


# four lanes and one (16384 pixels over all right-hand sides), chunks of one CTA per SM, two, and the most
@pytest.mark.parametrize("nx,ny,nrhs", [(128, 127, 1), (128, 128, 1), (129, 128, 1), (91, 90, 2), (181, 180, 1),
                                        (240, 200, 1), (280, 280, 1)])
def test_m2l_around_its_rules(nx, ny, nrhs):
    k = 9
    scan = synth.make_scan(nx=nx, ny=ny, n_det=4, n_t=20 * nx * ny // 4 * 4, n_int=2, half_bw=0, f_knee=0.0, seed=nx)
    scan.pix[:] = np.arange(scan.n_samples) // 3 % scan.n_pix   # every pixel, twenty hits
    c = MM.Context(0, None, MM.MM_FP64)
    c.setup_scan(scan)
    assert c.build_bd(1e-6) == 0
    rng = np.random.default_rng(nx)
    Z, x = rng.standard_normal((k, scan.n_pix, 3)), rng.standard_normal((nrhs, scan.n_pix, 3))
    c.set_coarse(Z)
    y = c.apply_precond(MM.MM_PRECOND_2L, x)
    prob = O.Problem.from_scan(scan)
    blocks, _ = O.bd_blocks(prob)
    M = np.linalg.inv(blocks)
    AZ = np.stack([O.apply_A(prob, z) for z in Z])
    E = np.einsum("apc,bpc->ab", Z, AZ)
    for r in range(nrhs):
        u = np.linalg.solve(0.5 * (E + E.T), np.einsum("apc,pc->a", Z, x[r]))
        ref = np.einsum("pij,pj->pi", M, x[r] - np.einsum("apc,a->pc", AZ, u)) + np.einsum("apc,a->pc", Z, u)
        assert_close(y[r], ref, 1e-9)
    c.close()
