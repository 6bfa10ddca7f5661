"""The error of the FP32 correlation, split TF32 from n = 256 on, on data that is hard on that: products of one sign, where the
tensor core's truncation and the dropped low products add up instead of cancelling, at one scale, over
24 binary orders, and as one head with a tail below the accumulator's last bit.  The bound of the
selection's band holds for every score (it assumes 2^-22 of the running magnitude lost per product in
the tensor core, which no document guarantees), and the 2-norm of the error is no larger than that
of one FP32 FMA chain per score, the kernel it took the place of, and still is below n = 256."""
import numpy as np
import pytest

from paper_1302_5010_gb300 import mpl

pytestmark = pytest.mark.gpu


def _data(kind, n, m, p):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n + len(kind))

    def rand(f, *s):
        return f(*s, device="cuda", generator=g)

    A, R = rand(torch.randn, m, n).abs(), rand(torch.randn, p, n).abs()
    if kind == "one_sign_wide_range":
        A *= 2.0 ** torch.randint(-12, 12, (m, n), device="cuda", generator=g)
    elif kind == "one_magnitude":
        A, R = 1 + 1e-3 * rand(torch.rand, m, n), 1 + 1e-3 * rand(torch.rand, p, n)
    elif kind == "head_and_tail":
        A = 1.5 * 2.0 ** -23 * (1 + rand(torch.rand, m, n))
        A[:, 0] = 1.0
        R = torch.ones(p, n, device="cuda")
    elif kind == "head_per_group":  # one large product at the start of every 8 (one MMA's K)
        A = 2.0 ** -13 * (1 + rand(torch.rand, m, n))
        A[:, ::8] = 1.0 + rand(torch.rand, m, (n + 7) // 8)
    return A.contiguous(), R.contiguous()


@pytest.mark.parametrize("kind", ["one_sign", "one_sign_wide_range", "one_magnitude", "head_and_tail", "head_per_group"])
@pytest.mark.parametrize("n,p", [(128, 40), (160, 300), (256, 40), (1024, 300), (4095, 40), (16384, 300)])
def test_one_sign(kind, n, p):
    import torch
    m = 384
    A, R = _data(kind, n, m, p)
    C = torch.full((p, m), float("nan"), device="cuda")
    assert mpl.mpl_correlate_noalloc(A, n, m, R, p, C) == mpl.MPL_OK
    A64, R64 = A.double(), R.double()
    exact = R64 @ A64.T
    absdot = R64.abs() @ A64.abs().T
    err = (C.double() - exact).abs()
    tf = 98.0 * 2.0 ** -22 + (n / 32.0 + 2.0) * 2.0 ** -24
    assert bool((err <= tf * absdot).all())
    acc = torch.zeros(p, m, dtype=torch.float64, device="cuda")
    for k in range(n):  # fused multiply-add: one rounding per term
        acc = (acc + R64[:, k, None] * A64[None, :, k]).float().double()
    chain = (acc - exact).abs()
    assert err.max().item() <= chain.max().item()
    assert err.norm().item() <= chain.norm().item()


@pytest.mark.parametrize("n,m,p", [(255, 300, 20), (256, 1, 9), (256, 20000, 128), (288, 20001, 65), (321, 39000, 16),
                                   (257, 20000, 257), (350, 129, 255)])
def test_first_sizes_of_the_split(n, m, p):
    """Just below and above the first size the tensor cores take, with several tiles per block (slices that are
    2, 0 and 2 modulo 3, so that consecutive tiles of a block start in different stages), on Gaussian data:
    the bound, and a 2-norm that a stale tile or a lost low part (2^-11) would exceed."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(n + m + p)
    A = torch.randn(m, n, device="cuda", generator=g)
    R = torch.randn(p, n, device="cuda", generator=g)
    C = torch.full((p, m), float("nan"), device="cuda")
    assert mpl.mpl_correlate_noalloc(A, n, m, R, p, C) == mpl.MPL_OK
    A64, R64 = A.double(), R.double()
    exact = R64 @ A64.T
    tf = 98.0 * 2.0 ** -22 + (n / 32.0 + 2.0) * 2.0 ** -24
    err = (C.double() - exact).abs()
    assert bool((err <= tf * (R64.abs() @ A64.abs().T)).all())
    assert err.norm().item() <= 2.0 ** -19 * exact.norm().item()


@pytest.mark.parametrize("sa,sr", [(1.0, 1e-34), (1.0, 1e-36), (1.0, 1e-38), (1.0, 1e-40), (1e-35, 1.0), (1e-37, 1e20),
                                   (1e-19, 1e-18)])
def test_small_magnitudes(sa, sr):
    """Entries whose low part is among TF32's subnormals (multiples of 2^-136) are off by up to 2^-137, which the
    band's bound takes beside the relative term (it fails alone at 1e-40); FP32 sums round to multiples of
    2^-149, once per 32 columns and product of parts."""
    import torch
    n, m, p = 512, 300, 40
    g = torch.Generator(device="cuda").manual_seed(17)
    A = torch.randn(m, n, device="cuda", generator=g) * sa
    R = torch.randn(p, n, device="cuda", generator=g) * sr
    C = torch.full((p, m), float("nan"), device="cuda")
    assert mpl.mpl_correlate_noalloc(A, n, m, R, p, C) == mpl.MPL_OK
    A64, R64 = A.double(), R.double()
    err = (C.double() - R64 @ A64.T).abs()
    relative = (98.0 * 2.0 ** -22 + (n / 32.0 + 2.0) * 2.0 ** -24) * (R64.abs() @ A64.abs().T)
    absolute = 2.0 ** -137 * (R64.abs().sum(1)[:, None] + A64.abs().sum(1)[None, :]) + 4 * n * 2.0 ** -149
    assert bool((err <= relative + absolute).all()), ((err - relative) / absolute).max().item()
    if sr == 1e-40:
        assert bool((err > relative).any())
