"""The three-pass whole-block float32 filter at the edges of its tiles.

Tolerance 1e-5 (relative 2-norm, per Stokes column too): the float32 operator's.
"""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import assert_close

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker

TOL32 = 1e-5
LAM = 37


def scan_with(lengths, pixels, nx, seed):
    """A one-detector scan of blocks of the given lengths; pixels: "raster", "random" (a new pixel
    every sample, anywhere on the map), "steps" (runs of 1 to 12 samples) or "still" (one pixel)."""
    rng = np.random.default_rng(seed)
    n = int(np.sum(lengths))
    s = synth.make_scan(nx=nx, ny=nx, n_det=1, n_t=n, n_int=1, half_bw=LAM, f_knee=1.0, seed=seed, flag_frac=0.002)
    if pixels == "random":
        s.pix[:] = rng.integers(0, nx * nx, n)
    elif pixels == "steps":
        s.pix[:] = np.repeat(rng.integers(0, nx * nx, n), rng.integers(1, 13, n))[:n]
    elif pixels == "still":
        s.pix[:] = 5
    s.pix[rng.random(n) < 0.002] = -1
    s.block_off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    s.block_band = np.zeros(len(lengths), dtype=np.int32)
    return s


@pytest.mark.parametrize("L", [4608, 9216, 18432])
@pytest.mark.parametrize("pixels,nx", [("raster", 16), ("random", 8), ("random", 80), ("steps", 16), ("still", 8)])
def test_blocks_of_every_fill(L, pixels, nx):
    """Blocks that fill the transform exactly, end inside a chunk, a row or a pair of samples, hold a
    single sample, start at every offset from a 16-byte boundary; pixel windows that are staged and
    that are not; lanes with one, two and more pixels."""
    full = L - LAM
    scan = scan_with([full, 1, 2, 3, full - 1, 255, 257, full // 2, L // 8, L // 8 + 1, 7], pixels, nx, L + nx)
    c = MM.Context(0, None, MM.MM_FP32_MIXED)
    c.set_option("filter", 2)
    c.set_option("fft_len", L)
    c.setup_scan(scan)
    x = np.random.default_rng(L).standard_normal((2, scan.n_pix, 3))
    y = c.apply_A(x)
    assert c.get_option("plan_whole") == 2 and c.get_option("plan_fft_len") == L
    prob = O.Problem.from_scan(scan)
    for r in range(2):
        assert_close(y[r], O.apply_A(prob, x[r]), TOL32)
    c.close()


def test_device_pixels_out_of_range_are_refused_and_leave_the_scan():
    """A device array with a pixel outside [-1, n_pix) is refused before the context changes."""
    import torch
    scan = scan_with([1000, 3000], "raster", 8, 3)
    c = MM.Context(0, None, MM.MM_FP64)
    c.setup_scan(scan)
    x = np.random.default_rng(3).standard_normal((1, scan.n_pix, 3))
    y = c.apply_A(x)
    for bad in (-2, scan.n_pix):
        pix = torch.from_numpy(scan.pix).cuda()
        pix[2345] = bad
        with pytest.raises(MM.MapMakerError) as e:
            c.setup_pointing(pix, torch.from_numpy(scan.psi).cuda(), scan.block_off, scan.block_band, scan.band, scan.n_pix)
        assert e.value.status == MM.MM_ERR_ARG
        assert_close(c.apply_A(x)[0], y[0], 1e-13)
    c.close()


@pytest.mark.parametrize("prec", ["f64", "df"])
@pytest.mark.parametrize("L", [512, 4608, 9216])
@pytest.mark.parametrize("pixels,nx", [("raster", 16), ("random", 8), ("steps", 16), ("still", 8)])
def test_float64_scatter_of_every_fill(prec, L, pixels, nx):
    """The eight-samples-a-lane scatter of the float64 and double-float filters, as overlap-save segments
    (512) and whole blocks: 1e-11, those operators' tolerance."""
    full = 4608 - LAM
    scan = scan_with([full, 1, 2, 3, full - 1, 255, 257, 1151, 7, 9], pixels, nx, L + nx)
    c = MM.Context(0, None, MM.MM_FP64 if prec == "f64" else MM.MM_FP32_MIXED)
    c.set_option("filter", 2)
    c.set_option("fft_len", L)
    if prec == "df":
        c.set_option("apply_precision", 2)
    c.setup_scan(scan)
    x = np.random.default_rng(L).standard_normal((2, scan.n_pix, 3))
    y = c.apply_A(x)
    prob = O.Problem.from_scan(scan)
    for r in range(2):
        assert_close(y[r], O.apply_A(prob, x[r]), 1e-11)
    d = np.random.default_rng(1).standard_normal((1, scan.n_samples)).astype(c.tod_dtype)
    assert_close(c.rhs(d)[0], O.rhs(prob, d[0].astype(np.float64)), 1e-11)
    c.close()


@pytest.mark.parametrize("L", [4608, 9216, 18432])
@pytest.mark.parametrize("pixels,nx", [("raster", 16), ("random", 8), ("steps", 16)])
def test_float64_block_split_over_two_ctas(L, pixels, nx):
    """A x and b of blocks split by frequency, every fill of the transform: 1e-11; a whole solve with it
    reaches the map of the unsplit plan (1e-7 at a tolerance of 1e-11: pixels with three hits and an rcond
    of 1e-3 amplify the residual)."""
    full = L - LAM
    scan = scan_with([full, 1, 2, 3, full - 1, 255, 257, full // 2, L // 4, L // 4 + 1, 7], pixels, nx, L + nx)
    maps = []
    for half in (2, 1):
        c = MM.Context(0, None, MM.MM_FP64)
        c.set_option("filter", 2)
        c.set_option("half_transform", half)
        c.set_option("fft_len", L)
        c.setup_scan(scan)
        x = np.random.default_rng(L).standard_normal((2, scan.n_pix, 3))
        y = c.apply_A(x)
        assert c.get_option("plan_whole") == (3 if half == 2 else 2)
        prob = O.Problem.from_scan(scan)
        for r in range(2):
            assert_close(y[r], O.apply_A(prob, x[r]), 1e-11)
        d = np.random.default_rng(1).standard_normal((1, scan.n_samples))
        assert_close(c.rhs(d)[0], O.rhs(prob, d[0]), 1e-11)
        c.build_bd(1e-3)
        m, info = c.solve(d, tol=1e-11, max_iter=1000)
        assert info[0]["status"] == "MM_OK"
        maps.append(m[0])
        c.close()
    assert_close(maps[0], maps[1], 1e-7)


@pytest.mark.parametrize("lam", [0, 3, 4, 8, 9, 16])
@pytest.mark.parametrize("tile", [1024, 2048])
@pytest.mark.parametrize("pixels,nx", [("raster", 16), ("random", 8), ("steps", 16)])
def test_narrow_bands_of_every_fill(lam, tile, pixels, nx):
    """The direct filter's eight outputs per thread: every padded band width, tiles that end inside a
    thread's outputs or inside the halo, blocks shorter than the halo; 1e-5."""
    scan = scan_with([2048, 1, 2, 7, 8, 9, 15, 17, 1023, 1025, 2047, 2049, 4099, 64], pixels, nx, lam + nx)
    scan.band = np.stack([synth.scan.toeplitz_band(lam, 1.0)])
    c = MM.Context(0, None, MM.MM_FP32_MIXED)
    c.set_option("filter", 1)
    c.set_option("direct_tile", tile)
    c.setup_scan(scan)
    x = np.random.default_rng(tile).standard_normal((2, scan.n_pix, 3))
    y = c.apply_A(x)
    prob = O.Problem.from_scan(scan)
    for r in range(2):
        assert_close(y[r], O.apply_A(prob, x[r]), TOL32)
    c.close()
