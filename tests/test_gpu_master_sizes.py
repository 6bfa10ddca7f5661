"""Master problems at the sizes where their kernel changes: blocks in the registers of a warp (up to
32 atoms) and of 128, 192 and 256 threads (64, 96, 128), in shared memory (up to 200) and
streamed, with capacities that are and are not multiples of 4.  With rho atoms per iteration and
more violators than that, the first master problem has exactly rho atoms.  A signal whose active set
(the FP64 oracle's, which has no capacity) stays within the capacity ends certified; one that
outgrows it may still certify on the atoms that fit, or reports the capacity.  Every certified
signal is at the oracle's solution."""
import numpy as np
import pytest

import oracle
from paper_1302_5010_gb300 import mpl, synth
from parity import check_against_oracle
from test_gpu_parity import solve_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho,smax", [(1, 255), (31, 256), (32, 256), (33, 254), (63, 256), (64, 253), (65, 256),
                                      (96, 255), (97, 256), (127, 256), (128, 254), (129, 256), (199, 255),
                                      (200, 256), (201, 255), (240, 256)])
def test_master_problem_block_sizes(rho, smax):
    P = synth.small_problem(512, 1500, 6, 20, 60, rho=rho, lam_frac=0.02, seed=900 + rho)
    _, X64, res = solve_gpu(P, precision=0, smax=smax)
    Xo, r = oracle.bmpl(P.At, P.B, P.lam, P.rho)
    st = res.stats["status"]
    ok = st == mpl.MPL_SIG_CERTIFIED
    assert np.all(ok | ((st == mpl.MPL_SIG_CAPACITY) & (np.asarray(r["S_size"]) > smax)))
    idx = np.flatnonzero(ok)
    assert len(idx) >= 4
    check_against_oracle(P, X64[idx], Xo[idx], idx)
