"""The template-filtered product at the edges of its tiles: subscans from one sample to a whole block
(every number of parts, more units than one round of the projection's shared sums), bins that last one
sample or many lanes, blocks that end inside a lane's eight samples.  Tolerances as for the operator:
float64 and double-float 1e-11, float32 1e-5.
"""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import assert_close

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker


@pytest.mark.parametrize("prec", ["f64", "f32", "df"])
@pytest.mark.parametrize("order,stokes", [(0, 1), (1, 1), (1, 0), (3, 2)])
@pytest.mark.parametrize("bins", ["short", "long"])
def test_every_subscan_and_bin_length(prec, order, stokes, bins):
    rng = np.random.default_rng(11)
    lengths = [1, 7, 8, 9, 255, 256, 257, 1021, 4096, 3000]
    n = int(np.sum(lengths))
    s = synth.make_scan(nx=6, ny=6, n_det=1, n_t=n, n_int=1, half_bw=0, f_knee=0.0, seed=4, hwp=False)
    s.psi[:] = rng.uniform(0, np.pi, n).astype(np.float32)
    s.pix[:] = np.repeat(rng.integers(-1, 36, n), rng.integers(1, 20, n))[:n]
    s.block_off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    s.block_band = np.zeros(len(lengths), dtype=np.int32)
    cuts = [s.block_off]
    # one subscan, a few, 20, and more than two rounds of units in the last two blocks
    for b, k in ((4, 2), (5, 4), (6, 20), (8, 150), (9, 40)):
        cuts.append(s.block_off[b] + 1 + rng.choice(lengths[b] - 1, size=k, replace=False))
    sub = np.unique(np.concatenate(cuts)).astype(np.int64)
    nb = 37
    az = np.repeat(rng.integers(-1, nb, n), rng.integers(1, 4 if bins == "short" else 90, n))[:n].astype(np.int32)
    tp = O.TemplateProblem(s.pix, s.psi, s.block_off, s.band[s.block_band, 0], s.n_pix, sub, order, az, nb, stokes)
    c = MM.Context(0, None, MM.MM_FP32_MIXED if prec == "f32" else MM.MM_FP64)
    c.setup_scan(s)
    c.set_templates(order, sub, az, nb, stokes)
    if prec == "df":
        c.set_option("fp64_products", 2)
    x = rng.standard_normal((2, s.n_pix, 3))
    y = c.apply_A(x)
    for r in range(2):
        assert_close(y[r], O.apply_A_T(tp, x[r]), 1e-5 if prec == "f32" else 1e-11)
    c.close()


@pytest.mark.parametrize("prec", ["f64", "df"])
@pytest.mark.parametrize("block,n_blocks", [(16384, 2), (12000, 3), (1024, 8), (1000, 160)])
def test_every_thread_count(prec, block, n_blocks):
    """Blocks of which an SM holds one, two or many, fewer and more of them than SMs."""
    rng = np.random.default_rng(12)
    n = block * n_blocks
    s = synth.make_scan(nx=9, ny=9, n_det=1, n_t=n, n_int=n_blocks, half_bw=0, f_knee=0.0, seed=6, hwp=False)
    s.psi[:] = rng.uniform(0, np.pi, n).astype(np.float32)
    sub = np.unique(np.concatenate([s.block_off, np.arange(0, n, 397)])).astype(np.int64)
    az = (np.arange(n) // 50 % 23).astype(np.int32)
    tp = O.TemplateProblem(s.pix, s.psi, s.block_off, s.band[s.block_band, 0], s.n_pix, sub, 1, az, 23, 1)
    c = MM.Context(0, None, MM.MM_FP64)
    c.setup_scan(s)
    c.set_templates(1, sub, az, 23, 1)
    if prec == "df":
        c.set_option("fp64_products", 2)
    x = rng.standard_normal((s.n_pix, 3))
    assert_close(c.apply_A(x)[0], O.apply_A_T(tp, x), 1e-11)
    c.close()
