"""The exact finish around the block width (16) of its factorisation: planted supports of 1 to 129
atoms, and a batch whose supports are so mixed that the small ones are factored in global memory
(the launch is sized by the largest) while the large ones take conjugate gradients.  Every
signal is certified and its FP64 solution is the oracle's to 1e-9: the finish refines with
exact residuals, so a wrong factor would not converge to it, and a lost block would not
certify."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import synth
from parity import check_against_oracle
from test_gpu_parity import assert_certified, oracle_solve, solve_gpu

pytestmark = pytest.mark.gpu


def _check(P, smax):
    _, X64, res = solve_gpu(P, precision=0, smax=smax)
    assert_certified(res)
    Xo = oracle_solve(P)
    check_against_oracle(P, X64, Xo)
    assert np.linalg.norm(X64 - Xo) <= 1e-9 * np.linalg.norm(Xo)


@pytest.mark.parametrize("k", [1, 2, 15, 16, 17, 31, 32, 33, 47, 49, 64, 65, 80, 96, 97, 112, 127, 129])
def test_finish_support_sizes(k):
    n = 1021 if k % 2 else 1024  # rows that are and are not a multiple of 4
    _check(synth.small_problem(n, 1500, 4, k, k, rho=max(1, k // 3), lam_frac=0.05, seed=1200 + k), 256)


def test_finish_mixed_supports():
    _check(synth.small_problem(1100, 2200, 12, 5, 240, rho=40, lam_frac=0.02, seed=1400), 512)
