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


@pytest.mark.parametrize("nx", [7, 9, 32])
@pytest.mark.parametrize("nrhs,k", [(8, 3), (33, 17), (64, 64), (128, 40)])
def test_tensor_core_path_reads_and_writes_three_wide_maps(nx, nrhs, k):
    """mm_apply_precond's own arrays as operands: odd pixel counts (rows off 16-byte boundaries), an array
    that starts at an odd element, in place, and an output that overlaps the input shifted by a map
    (staged, the same values).  2e-5, the tensor-core path's tolerance, against float64."""
    import torch
    scan = synth.make_scan(nx=nx, ny=nx, n_det=2, n_t=max(4096, 40 * nx * nx), n_int=2, half_bw=16, f_knee=1.0, seed=nx)
    c = MM.Context(0, None, MM.MM_FP64)
    c.setup_scan(scan)
    assert c.build_bd(1e-6) == 0
    rng = np.random.default_rng(nrhs)
    c.set_coarse(rng.standard_normal((min(k, nx * nx), scan.n_pix, 3)))
    x = torch.from_numpy(rng.standard_normal((nrhs, scan.n_pix, 3))).cuda()
    c.set_option("tc_coarse", 0)
    ref = c.apply_precond(MM.MM_PRECOND_2L, x).cpu().numpy()
    c.set_option("tc_coarse", 2)
    n = x.numel()
    buf = torch.zeros(2 * n + 3 * scan.n_pix + 1, dtype=torch.float64, device="cuda")
    for shift, out_at in ((0, n), (1, n + 1), (0, 0), (1, 1), (0, 3 * scan.n_pix)):
        xs = buf[shift:shift + n].view(nrhs, scan.n_pix, 3)
        xs.copy_(x)
        ys = buf[out_at:out_at + n].view(nrhs, scan.n_pix, 3)
        c.apply_precond(MM.MM_PRECOND_2L, xs, out=ys)
        assert_close(ys.cpu().numpy().reshape(-1, 3), ref.reshape(-1, 3), 2e-5)
    c.close()


@pytest.mark.parametrize("k", [1, 13])
def test_batch_past_four_lanes_a_pixel(k):
    """40 right-hand sides of 2304 pixels (one lane a pixel, chunks of 256) against each alone (four lanes,
    chunks of 64): the same sums in another order, E's condition below 1e4."""
    scan = synth.make_scan(nx=48, ny=48, n_det=2, n_t=40 * 2304, n_int=2, half_bw=16, f_knee=1.0, seed=8)
    c = MM.Context(0, None, MM.MM_FP64)
    c.setup_scan(scan)
    assert c.build_bd(1e-6) == 0
    rng = np.random.default_rng(k)
    c.set_coarse(rng.standard_normal((k, scan.n_pix, 3)))
    x = rng.standard_normal((40, scan.n_pix, 3))
    y = c.apply_precond(MM.MM_PRECOND_2L, x)
    for r in (0, 17, 39):
        assert_close(y[r], c.apply_precond(MM.MM_PRECOND_2L, x[r:r + 1])[0], 1e-9)
    c.close()
