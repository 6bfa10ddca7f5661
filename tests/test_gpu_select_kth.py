"""How many atoms one selection may look for (rho omega, or the warm start's W) before the bound of
its short list no longer applies: the list takes at most 32 keys per warp that owns some, of the
score row where it fits shared memory (128 atoms a warp, up to 8192) or of its 32-atom chunk
maxima (8192 < m <= 262144).  One outer iteration at, just above and far above that line takes the
largest correlations, no fewer and no others: the restricted solution is the oracle's on them.
Sizes: (n, m, rho, omega); the comment gives the warps that own keys and the keys looked for."""
import numpy as np
import pytest

import oracle
from paper_1302_5010_gb300 import mpl, synth
from parity import check_against_oracle
from test_gpu_parity import solve_gpu

pytestmark = pytest.mark.gpu

CASES = [(96, 100, 32, 1), (96, 100, 40, 1),       # 1 warp: 32, 40
         (96, 128, 33, 1),                         # 1: 33
         (136, 256, 64, 1), (136, 256, 80, 1),     # 2: 64, 80
         (200, 300, 96, 1), (200, 300, 100, 1),    # 3: 96, 100
         (704, 8192, 512, 1), (704, 8192, 513, 1), (768, 8192, 600, 1),  # 16: 512, 513, 600
         (200, 9000, 96, 1), (200, 9000, 100, 1), (200, 9000, 50, 2),  # 3 (282 maxima): 96, 100, 100
         (216, 10024, 100, 1),                     # 3 (314): 100
         (264, 16384, 128, 1), (264, 16384, 130, 1),  # 4 (512): 128, 130
         (344, 20011, 170, 1),                     # 5 (626): 170
         (704, 20011, 520, 1), (704, 20011, 260, 2)]  # 5 (626): 520


def _problem(n, m, rho, omega, p=5):
    kth = rho * omega
    P = synth.small_problem(n, m, p, 2, 6, rho=rho, lam_frac=0.01, sigma=0.02, seed=n + m + kth)
    c = np.abs(P.B.astype(np.float64) @ P.At.astype(np.float64).T)
    s = np.sort(c, axis=1)[:, ::-1]
    # more violators than atoms looked for, the last one taken told apart from the next in FP32
    P = synth.Problem("kth", P.At, P.B, np.minimum(P.lam, 0.5 * s[:, kth - 1]).astype(np.float32), rho)
    keep = np.nonzero(s[:, kth - 1] - s[:, kth] > 1e-5 * s[:, 0])[0][:3]
    assert keep.size >= 1
    return P.subset(keep), np.argsort(-c[keep], axis=1)[:, :kth]


@pytest.mark.parametrize("n,m,rho,omega", CASES)
@pytest.mark.parametrize("precision", [0, 1])
def test_first_iteration_takes_the_largest(n, m, rho, omega, precision):
    P, top = _problem(n, m, rho, omega)
    smax = min(m, 1024)
    _, X64, res = solve_gpu(P, precision=precision, omega=omega, smax=smax, max_outer=1)
    st = res.stats
    assert np.all(st["active_size"] == rho), st["active_size"]
    assert not np.any(st["status"] == mpl.MPL_SIG_CERTIFIED), st["status"]
    for i in range(P.p):
        assert set(np.nonzero(X64[i])[0]) <= set(top[i])
    if omega == 1:  # (Algorithm 2 keeps the rho largest of an inexact master problem: not compared one by one)
        Xo, r = oracle.bmpl(P.At, P.B, P.lam, rho, max_outer=1)
        assert np.all(r["S_size"] == rho)
        check_against_oracle(P, X64, Xo)


@pytest.mark.parametrize("m,candidates", [(100, 32), (100, 33), (100, 64), (128, 64), (200, 64)])
def test_warm_start_takes_its_candidates(m, candidates):
    """A network that accepts every candidate (all weights 0, output bias 1): the first iteration's set is
    the W largest correlations."""
    import torch
    n, rho = 96, 2
    P, top = _problem(n, m, candidates, 1)
    w = np.zeros(mpl.MPL_PROPOSAL_NPARAM, dtype=np.float32)
    w[3:6] = 1.0
    w[mpl.MPL_PROPOSAL_NPARAM - 1] = 1.0
    s = mpl.Solver(torch.from_numpy(P.At).cuda(), rho=rho, precision=0, warm_candidates=candidates, warm_max=m,
                   warm_threshold=0.0, max_outer=1, smax=m)
    mpl.mpl_proposal_set_weights(s.h, w)
    s.set(mpl.MPL_OPT_WARM_START, 2)
    X = torch.zeros((P.p, m), device="cuda")
    res = s.solve(torch.from_numpy(P.B).cuda(), torch.from_numpy(P.lam).cuda(), X, 1e-6)
    X64 = np.zeros((P.p, m))
    s.solution_f64(X64)
    s.close()
    assert np.all(res.stats["active_size"] == candidates), res.stats["active_size"]
    Xo, r = oracle.bmpl(P.At, P.B, P.lam, candidates, max_outer=1)
    assert np.all(r["S_size"] == candidates)
    for i in range(P.p):
        assert set(np.nonzero(X64[i])[0]) <= set(top[i])
    check_against_oracle(P, X64, Xo)
