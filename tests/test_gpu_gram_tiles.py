"""The computed Gram block at the edges of its tiles (32 and 64 atoms) and of its rule (tiles, signals):
new atoms per iteration around 16, 32 and 64, rows that are not a multiple of 4 or of a slice of 32,
and enough signals for the large tile.  Its entries are one FMA chain over the rows, the order
of the GEMM that builds Q, so a solve with the block computed and one with it gathered from Q agree
in every bit."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import mpl, synth
from test_gpu_parity import solve_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,k,rho", [(256, 5, 9, 7), (255, 5, 40, 16), (260, 5, 60, 17), (130, 6, 33, 32),
                                       (256, 170, 70, 33), (257, 170, 70, 33), (300, 160, 100, 64),
                                       (301, 8, 100, 65)])
def test_computed_block_is_the_gathered_one(n, p, k, rho):
    P = synth.small_problem(n, 900, p, max(1, k // 3), k, rho=rho, lam_frac=0.05, seed=1600 + rho + n)
    _, X64, r0 = solve_gpu(P, precision=0, smax=256, qgram=0, reentry=1)
    _, X64q, r1 = solve_gpu(P, precision=0, smax=256, qgram=1, reentry=1)
    # (a capacity of 256 atoms need not hold every signal's solution: where it does not, both say so)
    assert np.count_nonzero(r0.stats["status"] == mpl.MPL_SIG_CERTIFIED) * 4 >= p
    for f in ("status", "outer_iters", "active_size", "finishes"):
        np.testing.assert_array_equal(r0.stats[f], r1.stats[f])
    np.testing.assert_array_equal(X64, X64q)
