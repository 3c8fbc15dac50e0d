"""Set-up kernels: M_BD's sums and weights, the spectra of a plan.

M_BD tolerance 1e-11: sums of at most a few thousand float64 terms (relative error below 1e-14), blocks
inverted at a condition number of at most 1/rcond_min = 1e3.  A x with the double-float weights: 1e-11,
as elsewhere for that operator.
"""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import assert_close

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker

TOL = 1e-11


def odd_scan(pixels, lengths, angles, seed):
    rng = np.random.default_rng(seed)
    n = int(np.sum(lengths))
    s = synth.make_scan(nx=6, ny=6, n_det=1, n_t=n, n_int=1, half_bw=5, f_knee=1.0, seed=seed)
    if pixels == "random":
        s.pix[:] = rng.integers(0, 36, n)
    elif pixels == "still":
        s.pix[:] = np.arange(n) * 36 // n
    s.pix[rng.random(n) < 0.01] = -1
    if angles == "wide":      # negative, large, beyond the table's range, the nodes' midpoints
        s.psi[:] = rng.uniform(-130, 130, n).astype(np.float32)
        s.psi[::17] = rng.uniform(-3e4, 3e4, s.psi[::17].size).astype(np.float32)
        s.psi[5::19] = (np.arange(s.psi[5::19].size) + 0.5) * np.float32(np.pi / 4096)
    s.block_off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    s.block_band = np.zeros(len(lengths), dtype=np.int32)
    return s


@pytest.mark.parametrize("prec", [MM.MM_FP64, MM.MM_FP32_MIXED])
@pytest.mark.parametrize("pixels", ["raster", "random", "still"])
@pytest.mark.parametrize("angles", ["hwp", "wide"])
def test_mbd_and_weights(prec, pixels, angles):
    """Blocks of one sample, of a lane's eight samples, across warps' and slices' edges; runs shorter and
    longer than a lane; angles in and beyond the table's range; stored and computed weights."""
    scan = odd_scan(pixels, [1, 7, 8, 9, 255, 256, 257, 2049, 8192, 8193, 300], angles, 5)
    c = MM.Context(0, None, prec)
    c.setup_scan(scan)
    dropped = c.build_bd(1e-3)
    prob = O.Problem.from_scan(scan)
    w0 = np.repeat(scan.band[scan.block_band, 0], np.diff(scan.block_off))
    ok = scan.pix >= 0
    a = 2.0 * scan.psi.astype(np.float64)
    row = np.stack([np.ones_like(a), np.cos(a), np.sin(a)], 1)[ok]
    S = np.zeros((scan.n_pix, 3, 3))
    np.add.at(S, scan.pix[ok], w0[ok][:, None, None] * row[:, :, None] * row[:, None, :])
    hits = np.bincount(scan.pix[ok], minlength=scan.n_pix)
    ev = np.linalg.eigvalsh(S)
    good = (hits >= 3) & (ev[:, 0] >= 1e-3 * ev[:, 2])
    assert dropped == int((~good).sum())
    inv = np.zeros_like(S)
    inv[good] = np.linalg.inv(S[good])
    x = np.random.default_rng(6).standard_normal((scan.n_pix, 3))
    assert_close(c.apply_precond(MM.MM_PRECOND_BD, x)[0], np.einsum("pij,pj->pi", inv, x), TOL)
    # the same weights in double-float and native float64 products
    for which in (1, 2):
        c.set_option("apply_precision", which)
        prob.pix = np.where((scan.pix >= 0) & good[np.maximum(scan.pix, 0)], scan.pix, -1)
        assert_close(c.apply_A(x)[0], O.apply_A(prob, x), TOL)
    c.close()


@pytest.mark.parametrize("n_bands", [1, 40])
def test_spectra_of_few_and_many_bands(n_bands):
    """Plans whose spectra come from the cosine sums (one band) and from the transform (more than 1e8
    terms), after a scan of another shape left its plan's buffers behind; float32, 1e-5."""
    lam, nb = 600, 18432 - 600
    first = odd_scan("raster", [500, 700], "hwp", 1)
    scan = synth.make_scan(nx=8, ny=8, n_det=n_bands, n_t=nb, n_int=1, half_bw=lam, f_knee=(0.1, 2.0), seed=9)
    c = MM.Context(0, None, MM.MM_FP32_MIXED)
    c.set_option("filter", 2)
    c.setup_scan(first)
    c.apply_A(np.zeros((1, first.n_pix, 3)))
    c.set_option("fft_len", 18432)
    c.setup_scan(scan)
    x = np.random.default_rng(7).standard_normal((scan.n_pix, 3))
    assert_close(c.apply_A(x)[0], O.apply_A(O.Problem.from_scan(scan), x), 1e-5)
    assert (1e8 > n_bands * lam * 9216) == (n_bands == 1)
    c.close()


@pytest.mark.parametrize("n_bands,length,lam,n_fft", [(5600, 1024, 256, 1536), (70000, 16, 2, 256)])
@pytest.mark.parametrize("half", [0, 2])
def test_tables_of_very_many_bands(n_bands, length, lam, n_fft, half):
    """A band per block: more bands than one group of transforms (2^28 / (33 * 1536) = 5295) and than the
    65535 rows of a grid; float64, 1e-11."""
    scan = odd_scan("random", [length] * n_bands, "hwp", 3)
    rng = np.random.default_rng(4)
    scan.band = rng.standard_normal((n_bands, lam + 1)) * np.exp(-np.arange(lam + 1) / (lam / 4 + 1))
    scan.block_band = np.arange(n_bands, dtype=np.int32)
    c = MM.Context(0, None, MM.MM_FP64)
    c.set_option("filter", 2)
    c.set_option("half_transform", half)
    c.set_option("fft_len", n_fft)
    c.setup_scan(scan)
    x = rng.standard_normal((scan.n_pix, 3))
    assert_close(c.apply_A(x)[0], O.apply_A(O.Problem.from_scan(scan), x), TOL)
    c.close()
