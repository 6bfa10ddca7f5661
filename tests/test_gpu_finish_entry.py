"""Atoms that enter the exact finish with a coefficient below what its FP32 Gram block resolves.
The dictionary is orthonormal up to its rounding to FP32, so the solution is the soft-thresholded
correlation: besides k large coefficients, twelve atoms per signal correlate with it by
lambda (1 + d), d from 2e-5 to 1e-4, and their coefficients are lambda d.  A master problem may
leave them at zero or not select them; the exact correlations admit them one by one, each step
refining from the point and the correlations of the step before.  Tolerance: the finish stops at
correlations within 0.1 tol lambda of lambda on the support, so an entry is off by at most
1e-7 lambda times the inverse block's norm (1 + 1e-6), in both solvers; over the at most 300
entries that is 2 sqrt(300) 1e-7 0.05 = 1.8e-7 absolutely, against ||x|| > sqrt(k) >= 3.  The
twelve coefficients, 1e-6 to 5e-6, are checked to be there: within 2e-8 each."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import synth
from test_gpu_parity import assert_certified, oracle_solve, solve_gpu

pytestmark = pytest.mark.gpu

LAM = 0.05


@pytest.mark.parametrize("n,k,p,smax", [(256, 9, 3, 128), (255, 40, 3, 128), (512, 100, 40, 256),
                                        (1024, 240, 3, 512), (1024, 240, 24, 512)])
def test_entries_below_the_gram_block(n, k, p, smax):
    rng = np.random.default_rng(77 * n + k)
    At = np.linalg.qr(rng.standard_normal((n, n)))[0].T.astype(np.float32).copy()
    C = np.zeros((p, n))
    tiny = np.zeros((p, n), dtype=bool)
    for i in range(p):
        at = rng.permutation(n)
        C[i, at[:k]] = rng.choice([-1.0, 1.0], k) * rng.uniform(1.0, 2.0, k)
        C[i, at[k:k + 12]] = rng.choice([-1.0, 1.0], 12) * LAM * (1.0 + np.geomspace(2e-5, 1e-4, 12))
        tiny[i, at[k:k + 12]] = True
    P = synth.Problem("entry", At, (C @ At.astype(np.float64)).astype(np.float32),
                      np.full(p, LAM, dtype=np.float32), 16)
    _, X64, res = solve_gpu(P, precision=0, smax=smax)
    assert_certified(res)
    Xo = oracle_solve(P)
    assert np.linalg.norm(X64 - Xo, axis=1).max() <= 1.8e-7
    assert np.abs(X64 - Xo)[tiny].max() <= 2e-8
    assert np.count_nonzero(X64[tiny]) == np.count_nonzero(Xo[tiny])


@pytest.mark.parametrize("smax", [511, 512])
def test_zero_entries_screened_or_not(smax):
    """Active sets with many zero entries, whose Gram correlations are screened in FP32 when the rows are
    16-byte aligned (512) and summed in FP64 otherwise (511): both end at the oracle's solution.
    Correlations on the support are within 1e-7 lambda, so an entry is off by at most that times the
    inverse block's norm (below 10 for Gaussian blocks of 240 of 1024 rows) in both solvers: relative to
    ||x||, with lambda 0.005 of the largest correlation, below 2e-9 sqrt(240) 10 / sqrt(60) < 1e-7."""
    P = synth.small_problem(1024, 3000, 12, 60, 200, rho=40, lam_frac=0.005, seed=1500)
    _, X64, res = solve_gpu(P, precision=0, smax=smax)
    assert_certified(res)
    Xo = oracle_solve(P)
    assert np.linalg.norm(X64 - Xo) <= 1e-7 * np.linalg.norm(Xo)
