"""The three-pass float32 filter's wait for its pointing when it gives up (a limit of zero): the call
returns MM_ERR_TIMEOUT, and the next one, with the usual limit, is right again."""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import assert_close

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker

TOL32 = 1e-5


def context(L, n_t, n_int, **kw):
    """A scan whose float32 products run as three passes of L / 2 points."""
    scan = synth.make_scan(nx=8, ny=8, n_det=2, n_t=n_t, n_int=n_int, half_bw=37, f_knee=1.0, seed=4, **kw)
    c = MM.Context(0, None, MM.MM_FP32_MIXED)
    c.set_option("filter", 2)
    c.set_option("fft_len", L)
    c.setup_scan(scan)
    return scan, c


# blocks of one chunk, of as many chunks as are in flight, of all of them; ends inside a chunk and none
@pytest.mark.parametrize("L,n_t", [(4608, 7), (4608, 4571), (9216, 7 * 1152), (9216, 9179), (18432, 3 * 2304),
                                   (18432, 18395)])
def test_a_wait_that_gives_up_is_reported_and_leaves_the_context_usable(L, n_t):
    scan, c = context(L, 2 * n_t, 2)
    x = np.random.default_rng(L).standard_normal((2, scan.n_pix, 3))
    want = [O.apply_A(O.Problem.from_scan(scan), v) for v in x]
    for _ in range(2):
        c.set_option("wait_limit_ns", 0)
        with pytest.raises(MM.MapMakerError) as e:
            c.apply_A(x)
        assert e.value.status == MM.MM_ERR_TIMEOUT
        c.set_option("wait_limit_ns", 1e9)
        y = c.apply_A(x)
        assert c.get_option("plan_whole") == 2
        for a, b in zip(y, want):
            assert_close(a, b, TOL32)
    for bad in (-1, 2e9, float("nan")):
        with pytest.raises(MM.MapMakerError):
            c.set_option("wait_limit_ns", bad)
    c.close()
