"""Iterations with at most a quarter of the signals left run other kernels (matrix-vector products up to 8
signals of 256 entries or more, narrow tiles, smaller grids) than the graph of the whole batch.
The same hard signals are solved in a batch of easy ones, which end early, and replicated into a batch
that never falls to a quarter: the atoms each iteration takes come from the same FP32 re-scores, so the
iterations and the sets are equal, and the certified solutions differ by no more than both differ
from the exact one (correlations within 1e-7 lambda on the support; the inverse blocks' norms are
below 100 for these Gaussian sets of at most 60 of 256 rows: 2e-5 lambda sqrt(60), against
||x|| > sqrt(25) and lambda below 0.5: 2e-5 relative)."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import synth
from parity import check_against_oracle
from test_gpu_parity import assert_certified, oracle_solve, solve_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("hard,easy,n", [(1, 15, 256), (6, 60, 256), (6, 60, 304), (20, 140, 256), (40, 400, 128)])
def test_same_signals_in_few_and_in_full(hard, easy, n, precision):
    kh = 25 if n >= 256 else 12
    At = synth.gaussian_dictionary(n, 1500, 4242 + n)
    rng = np.random.default_rng(hard + easy + n)
    X = np.zeros((hard + easy, 1500))
    for i in range(hard + easy):
        k = kh if i < hard else 1
        X[i, rng.choice(1500, k, replace=False)] = rng.choice([-1.0, 1.0], k) * rng.uniform(1.0, 1.5, k)
    B = (X @ At.astype(np.float64)).astype(np.float32)
    lam = synth.lambdas_from_fraction(At, B, 0.05)
    P = synth.Problem("few", At, B, lam, 2)
    copies = -(-(hard + easy) // hard)
    Q = P.subset(np.tile(np.arange(hard), copies))
    _, Xf, rf = solve_gpu(P, precision=precision, reentry=1, smax=128)
    _, Xq, rq = solve_gpu(Q, precision=precision, reentry=1, smax=128)
    assert_certified(rf)
    assert_certified(rq)
    # the few did run alone: the easy ones need at most 5 analyses, the hard ones more
    assert rf.stats["outer_iters"][hard:].max() < rf.stats["outer_iters"][:hard].min()
    for f in ("outer_iters", "active_size", "nnz"):
        np.testing.assert_array_equal(rf.stats[f][:hard], rq.stats[f][:hard])
    np.testing.assert_array_equal(Xf[:hard] != 0, Xq[:hard] != 0)
    assert np.linalg.norm(Xf[:hard] - Xq[:hard]) <= 2e-5 * np.linalg.norm(Xq[:hard])
    idx = np.arange(min(hard, 6))
    check_against_oracle(P, Xf[idx], oracle_solve(P, idx), idx)
