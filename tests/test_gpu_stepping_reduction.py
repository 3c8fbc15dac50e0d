"""mm_solve_launch / mm_solve_poll with a reduction staged through the host: the stepping calls grow
their own pinned buffer and leave the reduction's alone."""
import time

import numpy as np
import pytest

import synth
from helpers import assert_close

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker


def test_stepping_with_a_host_reduction_over_growing_batches():
    scan = synth.make_scan(seed=63, nx=8, ny=8, n_det=2, n_t=4096, n_int=2, half_bw=64, f_knee=1.0)
    c = MM.Context(0, None, MM.MM_FP64)
    c.setup_scan(scan)
    c.build_bd()
    calls = []
    for nrhs in (1, 3, 8):
        d = np.random.default_rng(nrhs).standard_normal((nrhs, scan.n_samples))
        c.set_reduction(None)
        want, info = c.solve(d, MM.MM_PRECOND_BD, tol=1e-9, max_iter=300)
        c.set_reduction(lambda arr: calls.append(arr.sum()))   # one rank: the sum over ranks is the array
        c.solve_begin(d, MM.MM_PRECOND_BD, tol=1e-9, max_iter=300)
        done, rounds = False, 0
        while not done:
            c.solve_launch(4)
            ready = False
            t0 = time.monotonic()
            while not ready:
                ready, done = c.solve_poll()
                assert time.monotonic() - t0 < 30
            rounds += 1
        got, _ = c.solve_end(like=d)
        assert rounds > 2 and len(calls) > rounds
        for a, b in zip(got, want):
            assert_close(a, b, 1e-7)
    c.close()
