"""Gram matrices, column combinations and the one-right-hand-side M_2l kernels at the edges of their tiles.

M_2l x is invariant to the basis chosen for span Z, so a coarse space set from random columns (Gram
matrices, orthonormalisation, A Z, E) and M_2l are checked together against Eq. m2l in float64: 1e-9
(E of random columns has a condition number below 1e4).
"""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import assert_close

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker


@pytest.mark.parametrize("nx,k", [(3, 1), (5, 7), (8, 31), (8, 32), (9, 33), (16, 65), (40, 40)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_coarse_space_of_every_size(nx, k, nrhs):
    """Maps of less than a stage of pixels, of many slices; k below, at and above a tile of 32 columns and
    the groups of eight and four."""
    scan = synth.make_scan(nx=nx, ny=nx, n_det=2, n_t=max(2048, 40 * nx * nx), n_int=2, half_bw=16, f_knee=1.0, seed=nx)
    k = min(k, nx * nx)
    c = MM.Context(0, None, MM.MM_FP64)
    c.setup_scan(scan)
    assert c.build_bd(1e-6) == 0
    rng = np.random.default_rng(k)
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
