"""The one-launch PCG step of small maps (a cluster per right-hand side) at the edges of its range.

Maps of 1 to 4096 pixels take it, larger ones the three kernels; each must follow the oracle's iterates:
same product count (one more or less at the tolerance), recurrence residuals and maps at 1e-9.
"""
import numpy as np
import pytest

import oracle as O
import synth
from helpers import assert_close, oracle_problem

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1801_08937_gb300")
MM = P.mapmaker


@pytest.mark.parametrize("nx,ny", [(4, 4), (16, 17), (64, 64), (64, 65)])
@pytest.mark.parametrize("nrhs,products", [(1, 1), (3, 2)])
def test_small_map_solves_follow_the_oracle(nx, ny, nrhs, products):
    scan = synth.make_scan(nx=nx, ny=ny, n_det=4, n_t=max(2048, 10 * nx * ny), n_int=2, half_bw=16, f_knee=1.0, seed=nx)
    prob, mbd, good = oracle_problem(scan)
    rng = np.random.default_rng(ny)
    d = rng.standard_normal((nrhs, scan.n_samples))
    c = MM.Context(0, None, MM.MM_FP64)
    c.set_option("fp64_products", products)
    c.set_option("harvest", 12)
    c.setup_scan(scan)
    c.build_bd()
    m, info = c.solve(d, tol=1e-10, max_iter=300)
    A = lambda v: O.apply_A(prob, v.reshape(-1, 3)).reshape(-1)  # noqa: E731
    M = lambda v: O.bd_apply(mbd, v).reshape(-1)  # noqa: E731
    for r in range(nrhs):
        ref = O.pcg(A, M, O.rhs(prob, d[r]).reshape(-1), tol=1e-10, max_iter=300)
        assert info[r]["status"] == "MM_OK"
        assert abs(info[r]["iters"] - ref[1]["iters"]) <= 1
        if info[r]["iters"] == ref[1]["iters"]:
            assert_close(m[r].reshape(-1), ref[0], 1e-9)
    assert c.get_option("harvested") == min(12, info[0]["iters"])
    # a cap stops every right-hand side after exactly that many products
    m, info = c.solve(d, tol=1e-14, max_iter=5)
    assert [i["iters"] for i in info] == [5] * nrhs and info[0]["status"] == "MM_ERR_NOT_CONVERGED"
    c.close()
