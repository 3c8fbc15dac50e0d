"""Narrow bands: listed segments of one, two, four and eight tiles, cut into tiles by the kernel; 1e-5."""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import assert_close
from test_gpu_half3 import scan_with

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker


@pytest.mark.parametrize("lam", [0, 5, 16])
@pytest.mark.parametrize("tile", [1024, 2048])
@pytest.mark.parametrize("longest", [1024, 2047, 2048, 4096, 8191, 16384, 16385, 40001])
def test_segments_of_several_tiles(lam, tile, longest):
    """Blocks that end at a tile's edge, one sample before or behind it, inside the first and the last tile
    of a segment; bands that change between the two blocks of a CTA."""
    lengths = [n for n in (longest, 1, 1023, 1024, 1025, 3072, 8193, 16383, longest - 1, 2 * tile + 3) if n <= longest]
    scan = scan_with(lengths, "steps", 16, longest)
    scan.band = np.stack([synth.scan.toeplitz_band(lam, f) for f in (1.0, 0.3)])
    scan.block_band = (np.arange(len(lengths)) % 2).astype(np.int32)
    c = MM.Context(0, None, MM.MM_FP32_MIXED)
    c.set_option("filter", 1)
    c.set_option("direct_tile", tile)
    c.setup_scan(scan)
    x = np.random.default_rng(tile).standard_normal((2, scan.n_pix, 3))
    y = c.apply_A(x)
    prob = O.Problem.from_scan(scan)
    for r in range(2):
        assert_close(y[r], O.apply_A(prob, x[r]), 1e-5)
    c.close()
