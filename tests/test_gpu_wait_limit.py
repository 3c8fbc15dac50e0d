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


def timed_out(f):
    with pytest.raises(MM.MapMakerError) as e:
        f()
    assert e.value.status == MM.MM_ERR_TIMEOUT


@pytest.mark.parametrize("call", ["set_coarse", "build_coarse", "build_coarse_from_solve", "tuner", "solve", "uneven"])
def test_the_call_whose_products_gave_up_reports_it(call):
    """Each call that forms float32 products reports its own wait and leaves nothing of them behind;
    the next call is right and reports nothing."""
    import torch
    scan, c = context(4608, 4 * 4571, 4)
    c.build_bd(1e-3)
    rng = np.random.default_rng(9)
    Z = rng.standard_normal((3, scan.n_pix, 3))
    x = rng.standard_normal((1, scan.n_pix, 3))
    d = rng.standard_normal((2, scan.n_samples)).astype(np.float32)
    b = c.rhs(d[:1])
    y = c.apply_A(x)
    lens = np.array([scan.n_t, scan.n_t - 100], dtype=np.int64)
    run = {"set_coarse": lambda: c.set_coarse(Z),
           "build_coarse": lambda: c.build_coarse(None, m_max=12, eps_arn=1e-12, k=4),
           "build_coarse_from_solve": lambda: c.build_coarse_from_solve(k=4),
           "tuner": lambda: c.apply_A(x),
           "solve": lambda: c.solve(d[:1], MM.MM_PRECOND_BD, tol=1e-6, max_iter=500),
           "uneven": lambda: c.solve(d, MM.MM_PRECOND_2L, tol=1e-6, max_iter=500, rhs_len=lens)}[call]
    if call == "build_coarse_from_solve":
        c.set_option("harvest", 20)
        c.solve(d[:1], MM.MM_PRECOND_BD, tol=1e-6, max_iter=500)
        c.set_option("harvest", 0)
    if call == "uneven":
        c.set_coarse(Z)
    if call == "tuner":   # a geometry of its own, so that the plan is timed here
        c.set_option("filter", 0)
        c.set_option("fft_len", 0)
    c.set_option("wait_limit_ns", 0)
    timed_out(run)
    c.set_option("wait_limit_ns", 1e9)
    assert_close(c.apply_A(x)[0], y[0], 1e-5)   # a stale record of the wait would end this call
    assert np.array_equal(c.rhs(d[:1]).shape, b.shape)
    if call in ("set_coarse", "build_coarse", "build_coarse_from_solve"):
        with pytest.raises(MM.MapMakerError) as e:   # no coarse space from such products
            c.apply_precond(MM.MM_PRECOND_2L, x)
        assert e.value.status == MM.MM_ERR_STATE
    run()
    torch.cuda.synchronize()
    c.close()
