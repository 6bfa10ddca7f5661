"""The selection at the sizes where its routes change: rows that leave warps without scores (fewer
atoms than 4 per thread), the last row that fits shared memory and the first that does not (8192
atoms), chunk maxima that do and do not fit it (262144 atoms), and sets of one atom up to more
than a thread's share; every solution against the FP64 oracle, and the atoms taken (their
number, and the iterations) the same in both precisions where both apply."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import synth
from parity import check_against_oracle
from test_gpu_parity import assert_certified, oracle_solve, solve_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,k,rho", [(16, 20, 1, 1), (32, 127, 2, 1), (32, 128, 2, 3), (32, 129, 3, 2),
                                       (40, 511, 3, 17), (64, 2047, 4, 2), (64, 2049, 4, 40), (64, 8192, 4, 3),
                                       (64, 8193, 4, 3), (64, 65537, 4, 2), (64, 262144, 3, 2), (64, 262145, 3, 2),
                                       (64, 300001, 3, 33)])
def test_selection_route_edges(n, m, k, rho):
    P = synth.small_problem(n, m, 3, 1, k, rho=rho, lam_frac=0.1, seed=n + m + rho)
    _, X64, rp = solve_gpu(P, precision=0)
    assert_certified(rp)
    check_against_oracle(P, X64, oracle_solve(P))
    Xm, X64m, rm = solve_gpu(P, precision=1)
    assert_certified(rm)
    check_against_oracle(P, X64m, oracle_solve(P))
    np.testing.assert_array_equal(rp.stats["outer_iters"], rm.stats["outer_iters"])
    np.testing.assert_array_equal(rp.stats["active_size"], rm.stats["active_size"])
