"""Signals of any scale: the rounding terms of the first correlation's bound come from squares in FP32 where
these are in range and in FP64 elsewhere.  Scaling b and lambda by a power of two scales the
problem exactly, so the solution is the unscaled one's times it (to the accuracy of the certificate,
1e-6, whose effect on x is below 1e-6 of its norm for these well-conditioned supports)."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import synth
from test_gpu_parity import assert_certified, solve_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exp2", [-38, -34, -20, 20, 48, 52])
def test_scaled_signals(exp2):
    P = synth.small_problem(320, 1500, 5, 3, 12, rho=4, lam_frac=0.05, seed=1800)
    _, X64, r = solve_gpu(P, precision=1, smax=128)
    assert_certified(r)
    f = np.float32(2.0) ** exp2
    Ps = synth.Problem("scaled", P.At, P.B * f, P.lam * f, P.rho)
    _, X64s, rs = solve_gpu(Ps, precision=1, smax=128)
    assert_certified(rs)
    assert np.linalg.norm(X64s / np.float64(f) - X64) <= 1e-6 * np.linalg.norm(X64)
