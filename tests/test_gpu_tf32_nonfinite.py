"""Infinities in the FP32 correlation on the tensor cores: their scores are FP32 chains, exact like the
chain kernel's, and cost no more than the sizes say.  A tile of 128 atoms x 256 signals takes about
3500 cycles per 32 columns of n; with every row of it infinite its chains are 4 (rows of whole
16-byte units) or 16 reads of 32 cache lines per warp and 16 signals for as many columns, and as many
broadcasts: below 30 and 120 times the tile.  One infinite atom is 2 of 8 warps in one tile of
many, one infinite signal a sixteenth of the tiles' chains: below 8 and 30 times at these sizes, where
the tile that holds the atom is one of at least two per SM."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import mpl

pytestmark = pytest.mark.gpu


def _time(A, R, C, calls):
    import torch
    m, n = A.shape
    p = R.shape[0]
    ms = []
    for k in range(calls + 1):
        a, b = torch.cuda.Event(True), torch.cuda.Event(True)
        a.record()
        assert mpl.mpl_correlate_noalloc(A, n, m, R, p, C) == mpl.MPL_OK
        b.record()
        b.synchronize()
        if k:
            ms.append(a.elapsed_time(b))
    return float(np.median(ms))


@pytest.mark.parametrize("n,m,p,few,all_", [(1024, 40000, 256, 8, 30), (1021, 40000, 256, 30, 120)])
def test_time_with_infinities(n, m, p, few, all_):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(m, n, device="cuda", generator=g)
    R = torch.randn(p, n, device="cuda", generator=g)
    C = torch.empty(p, m, device="cuda")
    clean = _time(A, R, C, 5)
    A[m // 2, 5] = float("inf")
    atom = _time(A, R, C, 3)
    A[m // 2, 5] = 1.0
    R[p // 2, 5] = float("inf")
    signal = _time(A, R, C, 3)
    R[:, 7] = -float("inf")
    every = _time(A, R, C, 1)
    assert atom <= few * clean and signal <= few * clean, (clean, atom, signal)
    assert every <= all_ * clean, (clean, every)


@pytest.mark.parametrize("n,m,p", [(128, 130, 17), (255, 260, 33), (256, 130, 17), (257, 1000, 300), (1021, 700, 129)])
def test_chains_are_those_of_the_fp32_chain(n, m, p):
    """Scores that involve a value without a split, bit for bit as one FP32 FMA chain (FP64 products and
    sums rounded to FP32 at each step: the product of two FP32 values is exact in FP64, and 29 spare
    bits make a second rounding matter once in 2^29 steps)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(n + p)
    A = torch.randn(m, n, device="cuda", generator=g)
    R = torch.randn(p, n, device="cuda", generator=g)
    big = float(np.uint32(0x7f7ff000).view(np.float32))  # the first value without a split
    ra = [0, 31, 32, m - 1]
    rs = [0, 15, 16, p - 1]
    A[ra, 3] = big
    A[ra, 4] = -big
    R[:, 3:5] *= 1e-20
    R[rs, 7] = -big
    A[:, 7] *= 1e-30
    R[rs[1], 9] = float("inf")
    C = torch.full((p, m), float("nan"), device="cuda")
    assert mpl.mpl_correlate_noalloc(A, n, m, R, p, C) == mpl.MPL_OK
    acc = torch.zeros(p, m, dtype=torch.float64, device="cuda")
    A64, R64 = A.double(), R.double()
    for k in range(n):
        acc = (acc + R64[:, k, None] * A64[None, :, k]).float().double()
    acc = acc.float()
    for block, want in ((C[rs], acc[rs]), (C[:, ra], acc[:, ra])):
        np.testing.assert_array_equal(block.cpu().numpy(), want.cpu().numpy())
