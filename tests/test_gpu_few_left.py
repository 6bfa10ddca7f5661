"""Iterations with few signals left are launched for their count instead of replayed from the graph of the
whole batch, with other kernels (matrix-vector products, narrow tiles): the solve is, bit for bit, the one that
sizes every iteration by its bound, and the batch that never leaves the graphs (one signal of four)."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import synth
from test_gpu_parity import assert_certified, solve_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,precision,omega,n", [(1, 0, 1, 256), (4, 1, 1, 256), (40, 0, 1, 300), (150, 1, 1, 320),
                                                 (150, 0, 1, 257), (33, 0, 2, 300)])
def test_same_as_launched_one_by_one(p, precision, omega, n):
    # supports of 1 to 50 atoms: most signals end early, a few need many iterations
    P = synth.small_problem(n, 1500, p, 1, 50, rho=4, lam_frac=0.05, seed=1700 + p + n)
    X, X64, r = solve_gpu(P, precision=precision, omega=omega, smax=256, graph=1, reentry=1)
    Xd, X64d, rd = solve_gpu(P, precision=precision, omega=omega, smax=256, graph=0, reentry=1)
    assert_certified(r)
    for f in ("status", "outer_iters", "active_size", "finishes"):
        np.testing.assert_array_equal(r.stats[f], rd.stats[f])
    np.testing.assert_array_equal(X64, X64d)
